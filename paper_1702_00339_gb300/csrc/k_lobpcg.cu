// Stage (c): preconditioned block iteration for the lowest k eigenpairs of
// the box pencil (H, S) -- the paper's "structured iteration on subspace"
// (Sec. 2.3), read as LOBPCG (Knyazev 2001) with basis Y = [X | P | W],
// W = K (H X - S X Lambda) and K the inverse of the banded factor (k_band.cu) or, for the
// largest chains, the shifted inverse of the circulant embedding (a Fourier-block
// solve).  All dense work is FP64.
//
//  k_init_x     deterministic pseudo-random start X (splitmix64 counter hash), P = W = 0
//  k_gemm_tn    G = A^T B            (Gram blocks of the Rayleigh-Ritz step; 16- or 20-wide tiles)
//  k_gemm_nn    C = beta C + alpha A B
//  k_resid      R = HX - SX diag(lambda), relative residual norms, soft locking
//  k_colnorm    unit 2-norm columns (non-finite ones zeroed)
//  k_copy_cols  column-block copies
//  k_gather     results of a batch into one staging buffer
//  k_cell_canon / k_cell_transform / k_cell_back
//               canonical cell basis and the exactly symmetric transformed operator
#include <float.h>
#include "common.cuh"
#include "jacobi.cuh"

namespace fock {

// eigenvalue given to the cell directions dropped by the canonical transform
constexpr double kDecoupledEig = 1e6;

__global__ void k_init_x(const InitTask* __restrict__ tasks) {
  const InitTask T = tasks[blockIdx.y];
  const int tot = T.n * 3 * T.k;   // X random in [-1, 1); P and W zero
  for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < tot; it += gridDim.x * blockDim.x) {
    int i = it % T.n, c = it / T.n;
    double v = 0.0;
    if (c < T.k) {
      uint64_t h = splitmix64(T.seed ^ splitmix64(((uint64_t)c << 32) | (uint64_t)i));
      v = 2.0 * ((double)(h >> 11) * (1.0 / 9007199254740992.0)) - 1.0;
    }
    T.X[(size_t)i + (size_t)T.ld * c] = v;
  }
}

// C = alpha A^T B + beta C on TILE x TILE output tiles, one thread per
// output; TILE = 20 when the block sizes are multiples of 20 (less padding
// than 16 for the 3k x 3k Gram and the k x k projections at k = 20).  With
// T.sym the result is symmetric: tiles below the diagonal are skipped and the
// tiles above also write their transposes (diagonal tiles are computed in
// full and not mirrored, so no entry has two writers).
//
// The sum over n is split over T.ksplit CTAs per tile (gemm_tn_ksplit: a property
// of n, so results do not depend on the batch): a tile alone keeps one SM's FP64
// pipe busy for TILE^2 n / 1.7 cycles, 60 us for the Gram matrices of a chain of
// 512 functions, whose dozen tiles left the other SMs idle.  Each CTA leaves its
// partial sums in T.part; the last one of a tile to arrive (a counter in global
// memory that it resets) adds them in the order of the ranges.  Within a range
// partial sums of 8 tiles' rows (128 or 160 terms) are added to the total, so
// rounding grows like (8 TILE + n / (8 TILE)) u instead of n u (n = 16384 on the
// 512-cell chains, where the Gram entries of nearly dependent directions decide
// the pivots of the Rayleigh-Ritz step).  The next rows are loaded into registers
// while the present ones are multiplied.  Measured, mean
// of an iteration's launches: one chain of 512 functions 57 -> 18 us, 32 of them 91 ->
// 65, three of 976 95 -> 26.
template <int TILE>
__global__ void __launch_bounds__(TILE * TILE) k_gemm_tn(const GemmTask* __restrict__ tasks, int max_ks) {
  const GemmTask T = tasks[blockIdx.z];
  const int ks = blockIdx.x % max_ks, bx = blockIdx.x / max_ks;
  if (T.split) return;                       // computed on the tensor cores (mixed form)
  if (T.tile != TILE || ks >= T.ksplit) return;   // the other tile size's launch
  if (T.active && *T.active == 0) return;
  const int i0 = bx * TILE, j0 = blockIdx.y * TILE;
  if (i0 >= T.a || j0 >= T.b) return;
  if (T.sym && j0 < i0) return;
  __shared__ double As[TILE][TILE + 1], Bs[TILE][TILE + 1];
  __shared__ int s_last;
  const int tx = threadIdx.x % TILE, ty = threadIdx.x / TILE;
  // this CTA's range: whole tiles of rows
  const int nt = (T.n + TILE - 1) / TILE;
  const int t0 = (int)((long long)nt * ks / T.ksplit), t1 = (int)((long long)nt * (ks + 1) / T.ksplit);
  const bool ain = i0 + ty < T.a, bin = j0 + ty < T.b;
  const double* Ap = T.A + (size_t)T.lda * (i0 + ty) + tx;
  const double* Bp = T.B + (size_t)T.ldb * (j0 + ty) + tx;
  double an = 0.0, bn = 0.0;
  auto fetch = [&](int t) {
    const int r = t * TILE;
    an = (ain && r + tx < T.n) ? Ap[r] : 0.0;
    bn = (bin && r + tx < T.n) ? Bp[r] : 0.0;
  };
  double acc = 0.0, blk = 0.0;
  int cnt = 0;
  if (t0 < t1) fetch(t0);
  for (int t = t0; t < t1; ++t) {
    As[ty][tx] = an;
    Bs[ty][tx] = bn;
    __syncthreads();
    if (t + 1 < t1) fetch(t + 1);
#pragma unroll
    for (int q = 0; q < TILE; ++q) blk = fma(As[tx][q], Bs[ty][q], blk);
    __syncthreads();
    if (++cnt == 8) { acc += blk; blk = 0.0; cnt = 0; }
  }
  acc += blk;
  // thread (tx, ty) holds G[i0+tx][j0+ty]
  const bool in = i0 + tx < T.a && j0 + ty < T.b;
  if (T.ksplit > 1) {
    const size_t pl = (size_t)T.a * T.b, o = (size_t)(i0 + tx) + (size_t)T.a * (j0 + ty);
    if (in) T.part[pl * ks + o] = acc;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      int* c = T.count + blockIdx.y * ((T.a + TILE - 1) / TILE) + bx;
      s_last = (atomicAdd(c, 1) == T.ksplit - 1);
      if (s_last) *c = 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    acc = 0.0;
    if (in)
      for (int q = 0; q < T.ksplit; ++q) acc += __ldcg(T.part + pl * q + o);
  }
  if (in) {
    double* g = T.C + (size_t)(i0 + tx) + (size_t)T.ldc * (j0 + ty);
    const double v = (T.beta == 0.0) ? T.alpha * acc : T.beta * *g + T.alpha * acc;
    *g = v;
    if (T.sym && j0 > i0) T.C[(size_t)(j0 + ty) + (size_t)T.ldc * (i0 + tx)] = v;
  }
}

// amax, bmax: largest output dimensions; tiles: bit 0 = some task uses 16,
// bit 1 = some task uses 20 (one launch per tile size, each skipping the
// other's tasks, so a problem's products never depend on its batch); ks: the
// largest split of the sum
void launch_gemm_tn(const GemmTask* t, int n, int amax, int bmax, int tiles, int ks, cudaStream_t st) {
  if (!n) return;
  if (tiles & 1) k_gemm_tn<16><<<dim3((amax + 15) / 16 * ks, (bmax + 15) / 16, n), 256, 0, st>>>(t, ks);
  if (tiles & 2) k_gemm_tn<20><<<dim3((amax + 19) / 20 * ks, (bmax + 19) / 20, n), 400, 0, st>>>(t, ks);
}

// C = alpha A B + beta C; a thread owns row i of four consecutive columns,
// so each load of A serves four FP64 FMAs -- or of one column where the product
// is too small to fill the GPU that way (64 CTAs of 256 threads): 512 x 40 outputs
// of a chain of 512 functions, mean of an iteration's launches 19 us -> 10.  The
// same sum either way.
template <int NC>
__device__ __forceinline__ void gemm_nn_cols(const GemmTask& T) {
  const int nbc = (T.b + NC - 1) / NC;
  const int tot = T.n * nbc;
  for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < tot; it += gridDim.x * blockDim.x) {
    const int i = it % T.n, j0 = (it / T.n) * NC;
    const int nj = min(NC, T.b - j0);
    const double* b[NC];
    double acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) { b[c] = T.B + (size_t)T.ldb * (j0 + (c < nj ? c : 0)); acc[c] = 0.0; }
#pragma unroll 4
    for (int q = 0; q < T.a; ++q) {
      const double x = T.A[(size_t)i + (size_t)T.lda * q];
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = fma(x, b[c][q], acc[c]);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c)
      if (c < nj) {
        double* cp = T.C + (size_t)i + (size_t)T.ldc * (j0 + c);
        *cp = (T.beta == 0.0) ? T.alpha * acc[c] : T.beta * *cp + T.alpha * acc[c];
      }
  }
}
__global__ void __launch_bounds__(256) k_gemm_nn(const GemmTask* __restrict__ tasks) {
  const GemmTask T = tasks[blockIdx.y];
  if (T.split) return;                       // computed on the tensor cores (mixed form)
  if (T.active && *T.active == 0) return;
  if ((long long)T.n * T.b <= (long long)gridDim.x * blockDim.x * 2) gemm_nn_cols<1>(T);
  else gemm_nn_cols<4>(T);
}

// Columns at or below lock_tol get R = 0 (soft locking).
__global__ void k_resid(const ResidTask* __restrict__ tasks, double lock_tol) {
  const ResidTask T = tasks[blockIdx.y];
  if (T.active && *T.active == 0) return;
  const int c = blockIdx.x;
  if (c >= T.k) return;
  __shared__ double r1[256], r2[256];
  __shared__ double s_l;
  // Rayleigh quotient of the column from its fresh images: x^T H x / x^T S x
  double xh = 0.0, xs = 0.0;
  for (int i = threadIdx.x; i < T.n; i += blockDim.x) {
    size_t o = (size_t)i + (size_t)T.ld * c;
    xh += T.X[o] * T.HX[o];
    xs += T.X[o] * T.SX[o];
  }
  r1[threadIdx.x] = xh;
  r2[threadIdx.x] = xs;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) { r1[threadIdx.x] += r1[threadIdx.x + s]; r2[threadIdx.x] += r2[threadIdx.x + s]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    s_l = (r2[0] > 0.0) ? r1[0] / r2[0] : T.lam[c];
    T.lam[c] = s_l;
  }
  __syncthreads();
  const double l = s_l;
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < T.n; i += blockDim.x) {
    size_t o = (size_t)i + (size_t)T.ld * c;
    double sx = T.SX[o];
    double r = T.HX[o] - l * sx;
    T.R[o] = r;
    a += r * r;
    b += sx * sx;
  }
  r1[threadIdx.x] = a;
  r2[threadIdx.x] = b;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) { r1[threadIdx.x] += r1[threadIdx.x + s]; r2[threadIdx.x] += r2[threadIdx.x + s]; }
    __syncthreads();
  }
  __shared__ int lock;
  if (threadIdx.x == 0) {
    double den = fmax(fabs(l), 1e-300) * sqrt(r2[0]);
    // a column with no S-image (zero or non-finite) is broken, never converged
    double rv = (den > 0.0) ? sqrt(r1[0]) / den : NAN;
    T.res[c] = rv;
    lock = (rv <= lock_tol);
  }
  __syncthreads();
  if (lock)   // converged column: no search direction (the Rayleigh-Ritz step drops it)
    for (int i = threadIdx.x; i < T.n; i += blockDim.x) T.R[(size_t)i + (size_t)T.ld * c] = 0.0;
}

// One CTA per (column, task): scale dst's column to unit 2-norm (zero
// columns stay zero, non-finite ones become zero).
__global__ void k_colnorm(const CopyTask* __restrict__ tasks) {
  const CopyTask T = tasks[blockIdx.y];
  if (T.active && *T.active == 0) return;
  const int c = blockIdx.x;
  if (c >= T.ncols) return;
  double* col = T.dst + (size_t)T.ldd * c;
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < T.n; i += blockDim.x) s += col[i] * col[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) tot += red[w];
    red[0] = tot;
  }
  __syncthreads();
  const double nrm = sqrt(red[0]);
  if (!isfinite(nrm)) {   // a non-finite search direction: zeroed, so the Rayleigh-Ritz step drops it
    for (int i = threadIdx.x; i < T.n; i += blockDim.x) col[i] = 0.0;
    return;
  }
  if (!(nrm > 0.0)) return;
  const double inv = 1.0 / nrm;
  for (int i = threadIdx.x; i < T.n; i += blockDim.x) col[i] *= inv;
}

// One CTA per segment: dst[seg.dst + w] = seg.src[w].
__global__ void k_gather(const GatherSeg* __restrict__ segs, uint32_t* __restrict__ dst) {
  const GatherSeg g = segs[blockIdx.x];
  for (unsigned int w = threadIdx.x; w < g.words; w += blockDim.x) dst[g.dst + w] = g.src[w];
}

__global__ void k_copy_cols(const CopyTask* __restrict__ tasks) {
  const CopyTask T = tasks[blockIdx.y];
  if (T.active && *T.active == 0) return;
  const int tot = T.n * T.ncols;
  for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < tot; it += gridDim.x * blockDim.x) {
    int i = it % T.n, c = it / T.n;
    T.dst[(size_t)i + (size_t)T.ldd * c] = T.src[(size_t)i + (size_t)T.lds * c];
  }
}

}  // namespace fock

namespace fock {

// One CTA per chain on the structured path: the cell basis.  Jacobi
// eigendecomposition T_S[0] = Q diag(s) Q^T of the cell overlap, kept set
// K = {s > tau} in ascending Jacobi index with tau the dependency cut
// (common.cuh) formed from B = sum over offsets of |T_S[d]|, and
// Xc = Q_K diag(s_K)^-1/2 (m0 x m0, the columns past |K| zero).  A removed
// cell direction v spans vectors e_k (x) v, one per cell, on which the
// chain's overlap form is at most tau: numerically singular directions.
__global__ void k_cell_canon(const CanonTask* __restrict__ tasks) {
  extern __shared__ double cs[];
  const CanonTask T = tasks[blockIdx.x];
  const int m0 = T.m0, ld = m0 + 1;
  double* G = cs;                 // ld x ld
  double* Q = cs + ld * ld;       // ld x ld
  __shared__ double sv[MAXM0 + 1];
  __shared__ int keep[MAXM0 + 1], s_r;
  __shared__ double red[32], s_tau;
  double part = 0.0;
  for (int it = threadIdx.x; it < m0 * m0; it += blockDim.x) {
    int i = it / m0, j = it % m0;
    G[i * ld + j] = 0.5 * (T.TS[i * m0 + j] + T.TS[j * m0 + i]);
    double b = fabs(T.TS[it]);
    for (int d = 1; d <= T.D; ++d)
      b += fabs(T.TS[(size_t)d * m0 * m0 + it]) + (T.ring_full ? 0.0 : fabs(T.TS[(size_t)d * m0 * m0 + j * m0 + i]));
    part += b * b;
  }
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) t += red[w];
    s_tau = null_tau(sqrt(t), (double)T.nb);
  }
  const bool turned = cta_jacobi(G, Q, m0, ld);
  if (threadIdx.x == 0) {
    int r = 0;
    for (int i = 0; i < m0; ++i)
      if (G[i * ld + i] > s_tau && G[i * ld + i] > 0.0) { keep[r] = i; sv[r] = G[i * ld + i]; ++r; }
    s_r = r;
    *T.kept = r;
  }
  __syncthreads();
  for (int it = threadIdx.x; it < m0 * m0; it += blockDim.x) {
    int mu = it / m0, j = it % m0;
    T.Xc[it] = (j < s_r) ? (turned ? Q[mu * ld + keep[j]] : mu == keep[j] ? 1.0 : 0.0) / sqrt(sv[j]) : 0.0;
  }
}

// One CTA per block: B' = Xc^T B Xc.  Blocks: [0, D] generators (H then S),
// then the boundary blocks (H then S).  The dropped directions of the cell
// (zero columns of Xc) get a decoupled diagonal in T_H[0], T_S[0]: H = big,
// S = 1, so their eigenvalue `big` stays above every wanted one.
// Transformed blocks Xc^T B Xc of the generators and boundary blocks, made
// exactly symmetric where the operator is: the zero-offset generators and the
// diagonal boundary blocks are replaced by the mean of the product and its
// transpose, and a boundary pair (k, m) / (m, k) is written by the block with
// k < m as the mean of its product and the transpose of its partner's, the
// partner receiving the bitwise transpose.  (Xc carries factors up to
// tau^{-1/2}; products computed independently differ by rounding amplified by
// that factor squared, which would make the structured operator slightly
// non-symmetric and the one-sided Gram products of the block iteration
// inconsistent.)
__global__ void k_cell_transform(const CanonTask* __restrict__ tasks) {
  extern __shared__ double ts[];
  const CanonTask T = tasks[blockIdx.y];
  const int m0 = T.m0, m2 = m0 * m0;
  const int nblk = 2 * (T.D + 1) + 2 * T.nE;
  const int b = blockIdx.x;
  if (b >= nblk) return;
  const double* src; const double* srcp = nullptr; double* dst; double* dstp = nullptr;
  const int g = T.D + 1;
  bool sym = false;
  if (b < 2 * g) {
    const int d = b < g ? b : b - g;
    src = (b < g ? T.TH : T.TS) + (size_t)d * m2;
    dst = (b < g ? T.THc : T.TSc) + (size_t)d * m2;
    sym = (d == 0);
  } else {
    const bool hs = b < 2 * g + T.nE;
    const int e = hs ? b - 2 * g : b - 2 * g - T.nE;
    const int pe = T.Epart ? T.Epart[e] : -1;
    const double* E = hs ? T.EH : T.ES;
    double* Ec = hs ? T.EHc : T.ESc;
    if (pe >= 0 && pe < e) return;        // written by its partner
    src = E + (size_t)e * m2;
    dst = Ec + (size_t)e * m2;
    if (pe == e) sym = true;
    else if (pe > e) { srcp = E + (size_t)pe * m2; dstp = Ec + (size_t)pe * m2; }
  }
  double* X = ts;
  double* Y = ts + m2;
  double* Yp = ts + 2 * m2;
  for (int it = threadIdx.x; it < m2; it += blockDim.x) X[it] = T.Xc[it];
  __syncthreads();
  for (int it = threadIdx.x; it < m2; it += blockDim.x) {   // Y = B Xc (and the partner's)
    int mu = it / m0, j = it % m0;
    double acc = 0.0, accp = 0.0;
    for (int nu = 0; nu < m0; ++nu) acc += src[mu * m0 + nu] * X[nu * m0 + j];
    Y[it] = acc;
    if (srcp) {
      for (int nu = 0; nu < m0; ++nu) accp += srcp[mu * m0 + nu] * X[nu * m0 + j];
      Yp[it] = accp;
    }
  }
  __syncthreads();
  const int r = *T.kept;
  const double* Yt = srcp ? Yp : Y;         // the product whose transpose is averaged in
  for (int it = threadIdx.x; it < m2; it += blockDim.x) {   // dst = Xc^T Y
    int i = it / m0, j = it % m0;
    double acc = 0.0;
    for (int mu = 0; mu < m0; ++mu) acc += X[mu * m0 + i] * Y[mu * m0 + j];
    if (sym || srcp) {
      double acct = 0.0;                    // (Xc^T Yt)[j][i]
      for (int mu = 0; mu < m0; ++mu) acct += X[mu * m0 + j] * Yt[mu * m0 + i];
      acc = 0.5 * (acc + acct);
    }
    if ((b == 0 || b == g) && i == j && i >= r) acc = (b == 0) ? kDecoupledEig : 1.0;
    dst[it] = acc;
    if (dstp) dstp[j * m0 + i] = acc;
  }
}

// V (original basis) = (I_L (x) Xc) V' for n = L m0 rows, ncol columns.
__global__ void k_cell_back(const double* __restrict__ Xc, int m0, int L, int ncol, const double* Vr,
                            double* V, int ld) {
  const int tot = L * m0 * ncol;
  for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < tot; it += gridDim.x * blockDim.x) {
    int mu = it % m0, rest = it / m0, cell = rest % L, c = rest / L;
    double acc = 0.0;
    for (int j = 0; j < m0; ++j) acc += Xc[mu * m0 + j] * Vr[(size_t)(cell * m0 + j) + (size_t)ld * c];
    V[(size_t)(cell * m0 + mu) + (size_t)ld * c] = acc;
  }
}

void launch_gather(const GatherSeg* segs, int n, uint32_t* dst, cudaStream_t st) {
  if (n) k_gather<<<n, 128, 0, st>>>(segs, dst);
}

void launch_cell_canon(const CanonTask* t, int n, int maxm0, int maxblk, cudaStream_t st) {
  if (!n) return;
  size_t sm = (size_t)2 * (maxm0 + 1) * (maxm0 + 1) * sizeof(double);
  k_cell_canon<<<n, 256, sm, st>>>(t);
  k_cell_transform<<<dim3(maxblk, n), 256, (size_t)3 * maxm0 * maxm0 * sizeof(double), st>>>(t);
}

void launch_cell_back(const double* Xc, int m0, int L, int ncol, const double* Vr, double* V, int ld,
                      cudaStream_t st) {
  k_cell_back<<<64, 256, 0, st>>>(Xc, m0, L, ncol, Vr, V, ld);
}

}  // namespace fock
