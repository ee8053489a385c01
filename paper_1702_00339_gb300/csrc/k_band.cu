// Preconditioner of the box eigensolver: banded block factorisation of H - sigma S.
//
// The box chain matrix is block banded: H = BToepl(T) + E with generators
// T_d = block (k+d, k), |d| <= D (Sec. 2.3, Remark 3.2) and the boundary blocks
// E.  A = H - sigma S, sigma below the spectrum (from the circulant
// embedding's Fourier blocks), is symmetric positive definite with the same
// band, so it factors as M Delta M^T with M unit block lower banded (bandwidth
// D cells) and Delta block diagonal.  W = A^-1 R is the shift-and-invert search
// direction of the block iteration.  In this form (rather than L L^T) one step
// of either substitution is one product of a block column with the row just
// finished, without a triangular solve in between.
//
// A chain of L block rows is long, and a step waits for the one before: where L >= 2 D + 2
// the elimination goes from both ends towards D rows in the middle (twist). Side 0
// eliminates rows 0 .. a - 1 downwards, side 1 rows L - 1 .. a + D upwards, which is the
// same procedure on the chain in reverse order; the sum of what both leave of the middle
// rows is factored by each side for itself, in its own order, so that each goes on into its
// half without waiting for the other: (L + D) / 2 steps instead of L.
//
//  k_band_column  few problems of large blocks: a launch per block column, all SMs
//  k_band_factor  one thread-block cluster per problem: fill the band from T
//                 and E, factor it block column by block column; on a
//                 non-positive pivot lower sigma and start again
//  k_band_solve   forward and back substitution, one CTA per group of columns
//                 of a problem's R
//
// Storage, per problem: win, a ring of D + 1 block rows, row K holding the
// blocks (K, K-d) of what is left of A; fwd[J], the coefficients of one step
// down, [q][d-1][mu] = M_{J+d,J}[mu][q]; bwd[K], those of one step up,
// [q][d][mu] = M_{K,K-d}[q][mu] for d >= 1 and Delta_{K-D-1}^-1[q][mu] for
// d = 0; dinv[K] = Delta_K^-1; side 1's rows, in its own order, after side 0's.  A step's coefficients lie one after another in
// the order its threads (d, mu) read them, padded to a multiple of 16 bytes.
#include <algorithm>

#include "common.cuh"

namespace fock {

namespace {

__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ int cl_rank() { int r; asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ int cl_size() { int r; asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }

// the shared memory of another CTA of the cluster at the address of p in this one
template <typename X> __device__ __forceinline__ uint32_t cl_addr(const X* p, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ int cl_load(const int* p, int rank) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(cl_addr(p, rank)) : "memory");
  return v;
}
__device__ __forceinline__ double cl_load(const double* p, int rank) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(cl_addr(p, rank)) : "memory");
  return v;
}
__device__ __forceinline__ float cl_load(const float* p, int rank) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cl_addr(p, rank)) : "memory");
  return v;
}

constexpr int kFactorThreads = 512;   // 256 where blocks are small

// Row d1 (1-based) of pair number p in the order (1,1) (2,1) (2,2) (3,1) ...
__device__ __forceinline__ int pair_row(int p) {
  int d = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);   // FP32: the loops below correct it
  while ((d + 1) * (d + 2) / 2 <= p) ++d;
  while (d * (d + 1) / 2 > p) --d;
  return d + 1;
}

}  // namespace

namespace {

// One side of a factorisation (the whole chain without twist): L rows in its order, a of
// them before the middle; sg the shift.
struct BandSide {
  const BandTask& T;
  int side, m0, m2, D, D1, LL, a0, a1, a, L, late, steps;
  size_t fst, bst;
  double *fwd, *bwd, *dinv, sg;
  __device__ BandSide(const BandTask& t, int sd) : T(t), side(sd), m0(t.m0), m2(t.m0 * t.m0), D(t.D), D1(t.D + 1), LL(t.L) {
    a0 = (LL - D) / 2;
    a1 = LL - D - a0;                          // a0 <= a1 <= a0 + 1
    a = !T.twist ? LL : side ? a1 : a0;
    L = T.twist ? a + D : LL;
    steps = T.twist ? a1 + D : LL;
    late = T.twist ? a1 - a : 0;               // side 0 may start one step late
    fst = band_step(D, m0);
    bst = band_step(D1, m0);
    const size_t r0 = side ? a0 + D : 0;       // the side's first row of the factor
    fwd = T.fwd + r0 * fst; bwd = T.bwd + r0 * bst; dinv = T.dinv + r0 * m2;
  }
  // block (K, K-d) of the window, a ring of D + 2 rows; written by any CTA: read from L2
  __device__ double* winS(int sd, int K, int d) const { return T.win + ((size_t)(sd * (D1 + 1) + K % (D1 + 1)) * D1 + d) * m2; }
  __device__ double* win(int K, int d) const { return winS(side, K, d); }
  __device__ double at(int J, int d, int nu, int q) const { return __ldcg(win(J + d, d) + nu * m0 + q); }   // column J
  // row K enters the window: Toeplitz part and boundary blocks (a position's
  // entries lie one after another, its first one in efirst); side 1's block (K, K - d)
  // is the transpose of the one at row LL - 1 - K + d, and its middle starts at zero.
  // Shared out over gnth threads.
  __device__ void enter(int K, int gtid, int gnth) const {
    for (int it = gtid; it < D1 * m2; it += gnth) {
      const int d = it / m2, e = it % m2;
      if (d > K) continue;
      const int Kr = side ? LL - 1 - K + d : K, f = side ? (e % m0) * m0 + e / m0 : e;
      double v = 0.0;
      if (!side || K - d < a) {
        v = fma(-sg, T.TS[(size_t)d * m2 + f], T.TH[(size_t)d * m2 + f]);
        const int q0 = T.efirst[(size_t)Kr * D1 + d];
        if (q0 >= 0) {
          double x = 0.0;
          for (int q = q0; q < T.nE && T.Ek[q] == Kr && T.Em[q] == Kr - d; ++q)
            x += fma(-sg, T.ES[(size_t)q * m2 + f], T.EH[(size_t)q * m2 + f]);
          v += x;
        }
      }
      win(K, d)[e] = v;
    }
  }
  // the middle's blocks (a + i, a + j), j <= i: on side 0 the sum of both sides' (its block
  // is the transpose of side 1's (D - 1 - j, D - 1 - i)), on side 1 a copy of that
  __device__ void middle(int gtid, int gnth) const {
    for (long long it = gtid; it < (long long)(D * (D + 1) / 2) * m2; it += gnth) {
      const int p = (int)(it / m2), e = (int)(it % m2), mu = e / m0, nu = e % m0;
      const int i = pair_row(p) - 1, j = p - i * (i + 1) / 2;
      if (i == j && nu > mu) continue;         // diagonal blocks: lower triangle
      const int f = i == j ? e : nu * m0 + mu;
      const double x = __ldcg(winS(1 - side, (side ? a0 : a1) + D - 1 - j, i - j) + f);
      double* out = win(a + i, i - j) + e;
      *out = side ? x : __ldcg(out) + x;
    }
  }
  // column J into shared memory: the diagonal block (lower triangle mirrored: exactly
  // symmetric) into g0, and where it fits [d-1][q][nu] = A_{J+d,J}[nu][q], rows mp apart
  __device__ void load(int J, int dmax, double* g0, double* col, bool fits) const {
    const int mp = m0 + 1;
    for (int e = threadIdx.x; e < m2; e += blockDim.x) {
      const int i = e / m0, j = e % m0;
      g0[e] = at(J, 0, max(i, j), min(i, j));
    }
    if (fits)
      for (int it = threadIdx.x; it < dmax * m2; it += blockDim.x) {
        const int d = 1 + it / m2, e = it % m2, nu = e / m0, q = e % m0;
        col[((d - 1) * m0 + q) * mp + nu] = at(J, d, nu, q);
      }
    __syncthreads();
  }
  // M_{J+d1,J} = A_{J+d1,J} Delta_J^-1 into Ms (rows mp apart)
  __device__ void make_M(int J, int d1, const double* col, const double* Di, double* Ms, bool fits) const {
    const int mp = m0 + 1;
    for (int e = threadIdx.x; e < m2; e += blockDim.x) {
      const int mu = e / m0, q = e % m0;
      double s = 0.0;
      if (fits) {
        const double* c = col + (d1 - 1) * m0 * mp + mu;
        for (int t = 0; t < m0; ++t) s = fma(c[t * mp], Di[t * m0 + q], s);
      } else {
        for (int t = 0; t < m0; ++t) s = fma(at(J, d1, mu, t), Di[t * m0 + q], s);
      }
      Ms[mu * mp + q] = s;
    }
    __syncthreads();
  }
  __device__ void store_M(int J, int d1, const double* Ms) const {
    const int mp = m0 + 1;
    double* f = fwd + (size_t)J * fst + (d1 - 1) * m0;
    double* u = bwd + (size_t)(J + d1) * bst + d1 * m0;
    for (int e = threadIdx.x; e < m2; e += blockDim.x) {
      const int q = e / m0, mu = e % m0;
      f[(size_t)q * D * m0 + mu] = Ms[mu * mp + q];
      u[(size_t)q * D1 * m0 + mu] = Ms[q * mp + mu];
    }
  }
  // A_{J+d1,J+d2} -= M_{d1} A_{d2}^T, d2 = da .. db
  __device__ void update(int J, int d1, int da, int db, const double* col, const double* Ms, bool fits) const {
    const int mp = m0 + 1;
    for (int it = threadIdx.x; it < (db - da + 1) * m2; it += blockDim.x) {
      const int d2 = da + it / m2, e = it % m2, mu = e / m0, nu = e % m0;
      if (d1 == d2 && nu > mu) continue;       // diagonal block: lower triangle suffices
      double* out = win(J + d1, d1 - d2) + e;
      const double old = __ldcg(out);
      double s = 0.0;
      if (fits) {
        const double* c = col + (d2 - 1) * m0 * mp + nu;
        for (int q = 0; q < m0; ++q) s = fma(Ms[mu * mp + q], c[q * mp], s);
      } else {
        for (int q = 0; q < m0; ++q) s = fma(Ms[mu * mp + q], at(J, d2, nu, q), s);
      }
      *out = old - s;
    }
  }
  __device__ void store_inverse(int J, const double* Di) const {
    for (int e = threadIdx.x; e < m2; e += blockDim.x) {
      dinv[(size_t)J * m2 + e] = Di[e];
      if (J + D1 < L) bwd[(size_t)(J + D1) * bst + (size_t)(e / m0) * D1 * m0 + e % m0] = Di[e];
    }
  }
};

// Delta_J^-1 by Gauss-Jordan elimination without pivoting (positive definite exactly
// when every pivot is positive, else *s_bad is set), between g0 and g1; returns the one
// that holds it.
__device__ double* band_invert(double* g0, double* g1, int m0, double* s_r, int* s_bad) {
  const int tid = threadIdx.x, nth = blockDim.x, m2 = m0 * m0;
  if (tid == 0) {
    const double p = g0[0];
    const bool pos = __double_as_longlong(p) > 0;
    if (!pos || !(p == p)) *s_bad = 1;
    s_r[0] = rcp_nr(pos ? p : 1.0);
  }
  __syncthreads();
  double *cur = g0, *nxt = g1;
  const int step = nth - nth % m0, j = tid % m0;   // a thread's entries lie in one column j
  for (int k = 0; k < m0; ++k) {
    const double r = s_r[k & 1];
    if (tid < step) {
      const double g = (j == k) ? r : cur[k * m0 + j] * r;   // row k of the next matrix
      for (int e = tid, i = tid / m0; e < m2; e += step, i += step / m0) {
        const double v = (i == k) ? g : fma(-cur[i * m0 + k], g, (j == k) ? 0.0 : cur[e]);
        nxt[e] = v;
        if (i == k + 1 && j == k + 1) {        // the next pivot
          const bool pos = __double_as_longlong(v) > 0;
          if (!pos || !(v == v)) *s_bad = 1;
          s_r[(k + 1) & 1] = rcp_nr(pos ? v : 1.0);
        }
      }
    }
    __syncthreads();
    double* swp = cur; cur = nxt; nxt = swp;
  }
  return cur;
}

}  // namespace

// Bound by the chain of block columns, not by arithmetic throughput: column J
// needs Delta_J^-1 (m0 dependent pivots), M_d = A_d Delta_J^-1, and the trailing
// update A_{J+d1,J+d2} -= M_{d1} A_{d2}^T, D (D + 1) / 2 block products.  One SM
// takes 180 us per column at m0 = 16, D = 13 (its FP64 pipe: 2 multiply-adds a
// cycle); the cluster divides the block products among its CTAs, each of which
// inverts the m0 x m0 diagonal block for itself (Gauss-Jordan: one
// barrier per pivot, half of a Cholesky factor and its inverse) instead of
// waiting for another CTA to do it; the M_d are made by one CTA each.  Every decision depends on values all CTAs
// compute alike, so all take the same sequence of cluster barriers, and an
// entry's arithmetic does not depend on the cluster's size.  Measured: 64 cells
// of 8 functions 1.96 -> 0.55 ms (0.75 from one end; one problem, one factorisation), 32 of
// those 0.94 -> 0.79 ms.  Few problems of larger blocks go through k_band_column
// first and leave to this kernel only those that need another shift.
__global__ void __launch_bounds__(kFactorThreads) k_band_factor(const BandTask* __restrict__ tasks, int smem_doubles) {
  extern __shared__ double fsm[];
  const int CC = cl_size(), crank = cl_rank();
  const BandTask T = tasks[blockIdx.x / CC];
  if (T.sync[0] == 1) return;                  // factored by k_band_column
  // a side's CTAs
  const int C = T.twist ? CC / 2 : CC, side = crank / C, rank = crank % C;
  BandSide B(T, side);
  const int m0 = T.m0, m2 = m0 * m0, D = T.D, D1 = D + 1, mp = m0 + 1, L = B.L;
  const int tid = threadIdx.x, nth = blockDim.x, gtid = rank * nth + tid, gnth = C * nth;
  double* g0 = fsm;                          // diagonal block, its inverse in the end
  double* g1 = g0 + m2;
  double* Ms = g1 + m2;                      // M_{J+d1,J}, rows mp apart
  double* col = Ms + m0 * mp;                // column J
  const bool fits = 2 * m2 + D1 * m0 * mp <= smem_doubles;   // else the column is read from global memory
  __shared__ double s_r[2];
  __shared__ int s_bad;
  // shift search (every thread of every CTA alike): A = H - sigma S must be
  // positive definite.  The first sigma comes from the defect-free embedding; a
  // bound state below that band (a substituted nucleus) makes A indefinite.
  // Descend geometrically until the factorisation succeeds, then bisect three
  // times between the last failing and the succeeding shift, which brackets
  // lambda_min in (ok, bad); the final shift is ok - (bad - ok), at least one
  // bracket width below lambda_min (close enough for a strong shift-invert
  // preconditioner, far enough for a well-conditioned factor), and the band
  // holds its factor.
  double sg = *T.sigma0, sg_ok = NAN, sg_bad = NAN;
  int nbis = 0;
  bool stop = false;
  for (int attempt = 0; attempt < 24; ++attempt) {
    B.sg = sg;
    for (int K = 0; K < min(D1, L); ++K) B.enter(K, gtid, gnth);
    if (tid == 0) s_bad = 0;
    cl_arrive();
    cl_wait();
    bool bad = false;
    for (int t = 0; t < B.steps; ++t) {
      if (T.twist && t == B.a1) {              // both sides are at their first middle row
        bad = bad || cl_load(&s_bad, (crank + C) % CC) != 0;
        if (!side && !bad) B.middle(gtid, gnth);
        cl_arrive();
        cl_wait();
        if (side && !bad) B.middle(gtid, gnth);
        cl_arrive();
        cl_wait();
        if (bad) break;
      }
      const int J = t - B.late;
      if (J < 0 || (T.twist && bad)) {         // nothing to do: the step's barriers
        cl_arrive();
        cl_wait();
        cl_arrive();
        cl_wait();
        continue;
      }
      const int dmax = min(D, L - 1 - J);
      B.load(J, dmax, g0, col, fits);
      const double* Di = band_invert(g0, g1, m0, s_r, &s_bad);
      bad = s_bad != 0;
      // M_{J+d1,J} into Ms, and its storage for the solves: by one CTA each, read by
      // the others after a barrier (made anew where the column does not fit)
      if (fits) {
        if (!bad)
          for (int d1 = 1 + rank; d1 <= dmax; d1 += C) {
            B.make_M(J, d1, col, Di, Ms, true);
            B.store_M(J, d1, Ms);
            __syncthreads();
          }
        cl_arrive();                          // (and this CTA needs no more of column J)
        cl_wait();
      }
      if (!bad) {
        // this CTA's contiguous share of the pairs (d1, d2), d2 <= d1
        const int np = dmax * (dmax + 1) / 2;
        const int p0 = (int)((long long)np * rank / C), p1 = (int)((long long)np * (rank + 1) / C);
        for (int p = p0; p < p1;) {
          const int d1 = pair_row(p), base = d1 * (d1 - 1) / 2;
          const int da = p - base + 1, db = min(d1, p1 - base);   // d2 in da..db
          if (fits) {
            const double* f = B.fwd + (size_t)J * B.fst + (d1 - 1) * m0;
            for (int e = tid; e < m2; e += nth) Ms[(e % m0) * mp + e / m0] = __ldcg(f + (size_t)(e / m0) * D * m0 + e % m0);
            __syncthreads();
          } else {
            B.make_M(J, d1, col, Di, Ms, false);
            if (da == 1) B.store_M(J, d1, Ms);   // the owner of (d1, 1)
          }
          B.update(J, d1, da, db, col, Ms, fits);
          __syncthreads();
          p = base + db;
        }
        if (rank == 0) B.store_inverse(J, Di);
      }
      if (!fits) {
        cl_arrive();
        cl_wait();                            // every CTA has taken what it needs of row J
      }
      if (!bad && J + D1 < L) B.enter(J + D1, gtid, gnth);
      cl_arrive();
      cl_wait();                              // the trailing update and the new row are visible to all
      if (bad && !T.twist) break;
    }
    if (T.twist) {                             // one decision for both sides
      cl_arrive();
      cl_wait();
      bad = bad || cl_load(&s_bad, (crank + C) % CC) != 0;
      cl_arrive();
      cl_wait();
    }
    if (!bad) {
      sg_ok = sg;
      if (isnan(sg_bad) || nbis >= 3) stop = true;
    } else {
      sg_bad = sg;
    }
    if (stop) break;
    if (isnan(sg_ok)) sg = sg - 0.05 * (1.0 + fabs(sg)) * (double)(1 << min(attempt, 30));
    else if (nbis < 3) { sg = 0.5 * (sg_ok + sg_bad); ++nbis; }
    else { sg = sg_ok - (sg_bad - sg_ok); nbis = 99; }   // refactor one bracket below
  }
  if (crank == 0 && tid == 0) {
    *T.sigma_used = sg;
    if (!stop && T.fail) *T.fail = 1;
  }
}

// The same factorisation at the first shift with a launch per block column, where a
// cluster is too small for the block products (band_columns) of at most four problems.
// A launch is a barrier over the whole GPU of about 4 us.  Every CTA inverts the
// diagonal block and makes the M of its pairs for itself, so a column takes one
// launch; the row that enters goes to a slot of its own (the window has one row more
// than the band).  sync[1 + side]: a pivot was not positive, and what follows is
// skipped; sync[0] = 1: done.  101 cells of 16 functions 1.90 -> 1.36 ms, 512 of 32 40 -> 19
// ms, three rings of 61 cells of 16 with bound states 1.24 -> 0.98 ms.
//   phase 0: the first rows; 1: block column t; 2, 3: the middle, side 0 then 1; 4: the end
__global__ void __launch_bounds__(kFactorThreads) k_band_column(const BandTask* __restrict__ tasks, int phase, int t) {
  extern __shared__ double fsm[];
  const BandTask T = tasks[blockIdx.z];
  if (!band_columns(T.m0, T.D)) return;
  const int side = blockIdx.y, C = gridDim.x, rank = blockIdx.x;
  if (side && !T.twist) return;
  BandSide B(T, side);
  B.sg = *T.sigma0;
  const int tid = threadIdx.x, nth = blockDim.x, gtid = rank * nth + tid, gnth = C * nth;
  if (phase == 0) {
    for (int K = 0; K < min(B.D1, B.L); ++K) B.enter(K, gtid, gnth);
    if (rank == 0 && side == 0 && tid < 3) T.sync[tid] = 0;
    return;
  }
  if (phase >= 2 && phase <= 3) {
    if (!T.twist || t != B.a1 || side != phase - 2 || T.sync[1] || T.sync[2]) return;
    B.middle(gtid, gnth);
    return;
  }
  if (phase == 4) {
    if (rank == 0 && side == 0 && tid == 0 && !T.sync[1] && !T.sync[2]) {
      T.sync[0] = 1;
      *T.sigma_used = B.sg;
    }
    return;
  }
  const int J = t - B.late;
  if (J < 0 || J >= B.L) return;
  const int m0 = T.m0, m2 = m0 * m0;
  double *g0 = fsm, *g1 = g0 + m2, *Ms = g1 + m2, *col = Ms + m0 * (m0 + 1);
  __shared__ double s_r[2];
  __shared__ int s_bad, s_skip;
  // one read for the whole CTA: a CTA of this launch that started earlier may set the
  // flags meanwhile, and the threads of this one have to go on, or leave, together
  if (tid == 0) {
    s_bad = 0;
    s_skip = T.sync[1 + side] || (t >= B.a1 && (T.sync[1] || T.sync[2]));
  }
  __syncthreads();
  if (s_skip) return;
  const int dmax = min(B.D, B.L - 1 - J), np = dmax * (dmax + 1) / 2;
  const int p0 = (int)((long long)np * rank / C), p1 = (int)((long long)np * (rank + 1) / C);
  if (J + B.D1 < B.L) B.enter(J + B.D1, gtid, gnth);
  if (p0 >= p1 && rank != 0) return;
  B.load(J, dmax, g0, col, true);
  const double* Di = band_invert(g0, g1, m0, s_r, &s_bad);
  if (s_bad) {                                 // (every CTA finds the same)
    if (rank == 0 && tid == 0) T.sync[1 + side] = 1;
    return;
  }
  for (int p = p0; p < p1;) {
    const int d1 = pair_row(p), base = d1 * (d1 - 1) / 2;
    const int da = p - base + 1, db = min(d1, p1 - base);   // d2 in da..db
    B.make_M(J, d1, col, Di, Ms, true);
    if (da == 1) B.store_M(J, d1, Ms);         // the owner of (d1, 1)
    B.update(J, d1, da, db, col, Ms, true);
    __syncthreads();
    p = base + db;
  }
  if (rank == 0) B.store_inverse(J, Di);
}

// 16-byte asynchronous global -> shared copies (L2 only)
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// W = (M Delta M^T)^-1 R, one column of R per CTA.  Right-looking: once row J of
// the solution is final, its contribution to rows J+1 .. J+D is subtracted from
// their partial sums, which wait in a ring of rows in shared memory.  Thread
// (d, mu) owns entry mu of row J+d during step J, so a step has m0 dependent
// multiply-adds and no reduction; the threads of d = 0 store the
// finished row and bring in the row that enters the window.  The coefficients
// do not depend on the recursion: they come through two stages of shared memory
// (cp.async), qc rows of a step's coefficients at a time (MULTI; the whole step
// where all tasks' steps fit a stage), so that the L2 latency runs beside the
// multiply-adds.  Per step an SM's FP64 pipe takes (D + 1) m0^2 / 2 cycles, the
// bound; hence one column per CTA (two, which read the coefficients half as often,
// were slower from 20 columns to 2560).  Measured per launch,
// 20 columns a problem: one chain of 64 cells of 8 functions (D = 13) 941 -> 97 us from
// one end, 64 us from two (a cluster of two CTAs per column, which meet once);
// 32 of them 945 -> 185 and 215 us (the middle is done twice, and here the FP64 pipe
// is full; their factor gains as much); with one step of coefficients ahead in
// registers instead of shared memory the first took 205 us.  72 columns of 512 cells
// of 32: 4.9 ms from one end (6.9 without the stages), 2.5 from two.
template <typename R, bool MULTI>
__global__ void __launch_bounds__(1024) k_band_solve(const BandTask* __restrict__ tasks, int sides, int maxstage) {
  extern __shared__ __align__(16) double bsm[];
  const BandTask T = tasks[blockIdx.y];
  if (T.active && *T.active == 0) return;
  if ((T.fp32 != 0) != (sizeof(R) == 4)) return;
  const int col = blockIdx.x / sides, side = blockIdx.x % sides;
  if (col >= T.k || (side && !T.twist)) return;
  const double* Rc = T.R + (size_t)T.ld * col;   // this CTA's column
  double* Wc = T.W + (size_t)T.ld * col;
  const int m0 = T.m0, m2 = m0 * m0, D = T.D, LL = T.L, nslot = D + 2, D1 = D + 1;
  const int a0 = (LL - D) / 2, a = !T.twist ? LL : side ? LL - D - a0 : a0, L = T.twist ? a + D : LL;
  // the side's row r in the column; its part of the factor
  auto at = [&](int r, int mu) { return (size_t)(side ? LL - 1 - r : r) * m0 + mu; };
  const size_t r0 = side ? a0 + D : 0;
  const int tid = threadIdx.x, nth = blockDim.x, items = D1 * m0, fit = D * m0;
  const int fst = (int)band_step(D, m0), bst = (int)band_step(D1, m0);   // doubles per step
  const double *const Tfwd = T.fwd + r0 * fst, *const Tbwd = T.bwd + r0 * bst, *const Tdinv = T.dinv + r0 * m2;
  // rows of coefficients per stage: all m0, or as many as fit
  const int qc = MULTI ? band_rows(D1, m0, maxstage) : m0, nch = MULTI ? (m0 + qc - 1) / qc : 1;
  double* cf = bsm;                           // two stages of maxstage doubles
  R* acc = reinterpret_cast<R*>(bsm + (size_t)2 * maxstage);   // nslot rows, then two of the forward solution
  R* zb = acc + (size_t)nslot * m0;
  R* xm = zb + 2 * m0;                        // twist: what the side leaves of the middle rows, then
  R* zm = xm + (size_t)D * m0;                // their forward solution
  // rows [h qc, ...) of a step of `width` entries a row into stage `slot`
  auto stage = [&](const double* step, int total, int width, int h, int slot) {
    const double* src = step + (size_t)h * qc * width;
    const int n = band_piece(qc, width, total, h);
    double* dst = cf + (size_t)slot * maxstage;
    for (int i = 2 * tid; i < n; i += 2 * nth) cp_async16(dst + i, src + i);
  };
  const int mu0 = tid % m0;
  const bool zero = tid < m0;                 // this thread is (d = 0, mu0)
  // ---- M z = r, downwards ----
  stage(Tfwd, fst, fit, 0, 0);
  cp_async_commit();
  for (int it = tid; it < items; it += nth) {   // rows 0 .. D enter
    const int r = it / m0, mu = it % m0;
    if (r < L) acc[(r % nslot) * m0 + mu] = (side && r >= a) ? (R)0 : (R)Rc[at(r, mu)];
  }
  // the row that enters next (side 1's middle starts at zero)
  auto next = [&](int r) { return (side && r >= a) ? (R)0 : (R)Rc[at(r, mu0)]; };
  R nr = 0;
  if (zero && D1 < L) nr = next(D1);
  cp_async_wait0();
  __syncthreads();
  int st = 0;
  for (int J = 0, js = 0; J < L; ++J) {
    if (J == a) {                              // (twist) the middle rows: both sides' partial sums
      auto mid = [&](int it) { return acc + (js + it / m0 >= nslot ? js + it / m0 - nslot : js + it / m0) * m0 + it % m0; };
      for (int it = tid; it < fit; it += nth) xm[it] = *mid(it);
      __syncthreads();
      cl_arrive();
      cl_wait();
      for (int it = tid; it < fit; it += nth) {
        const R o = cl_load(xm + (D - 1 - it / m0) * m0 + it % m0, side ^ 1);
        *mid(it) = side ? o + xm[it] : xm[it] + o;
      }
      __syncthreads();
      cl_arrive();                             // waited for at the end: xm stays until the other side has read it
    }
    const R* y = acc + js * m0;
    const int live = min(D, L - 1 - J) * m0;
    for (int h = 0; h < nch; ++h, st ^= 1) {
      const double* cs = cf + (size_t)st * maxstage;
      if (h + 1 < nch) stage(Tfwd + (size_t)J * fst, fst, fit, h + 1, st ^ 1);
      else if (J + 1 < L) stage(Tfwd + (size_t)(J + 1) * fst, fst, fit, 0, st ^ 1);
      cp_async_commit();
      if (zero && h == 0) {
        const int r = J + D1, sl = js + D1 >= nslot ? js + D1 - nslot : js + D1;
        if (J < a) Wc[at(J, mu0)] = (double)y[mu0];
        else zm[(J - a) * m0 + mu0] = y[mu0];
        if (r < L) acc[sl * m0 + mu0] = nr;
        if (r + 1 < L) nr = next(r + 1);
      }
      const int qa = h * qc, qn = min(qc, m0 - qa);
      // (from the last thread down: the threads of d = 0 are busy with the rows)
      for (int it = nth - 1 - tid; it < live; it += nth) {
        const int d = 1 + it / m0, mu = it % m0;
        R* a = acc + (js + d >= nslot ? js + d - nslot : js + d) * m0 + mu;
        R s = *a;
#pragma unroll 8
        for (int q = 0; q < qn; ++q) s -= (R)cs[q * fit + it] * y[qa + q];
        *a = s;
      }
      cp_async_wait0();
      __syncthreads();
    }
    js = (js + 1 == nslot) ? 0 : js + 1;
  }
  // ---- M^T x = Delta^-1 z, upwards ----
  stage(Tbwd + (size_t)(L - 1) * bst, bst, items, 0, st);
  cp_async_commit();
  for (int it = tid; it < items; it += nth) {   // rows L-1 .. L-1-D enter
    const int r = L - 1 - it / m0, mu = it % m0;
    if (r >= 0) {
      R s = 0;
      for (int q = 0; q < m0; ++q) s += (R)Tdinv[(size_t)r * m2 + q * m0 + mu] * (r < a ? (R)Wc[at(r, q)] : zm[(r - a) * m0 + q]);
      acc[(r % nslot) * m0 + mu] = s;
    }
  }
  // row that enters at step K: K - D - 1; its z waits in zb, the one after it in nr
  if (zero) {
    const int r = L - 1 - D1;
    if (r >= 0) zb[((L - 1) & 1) * m0 + mu0] = (R)Wc[at(r, mu0)];
    nr = (r - 1 >= 0) ? (R)Wc[at(r - 1, mu0)] : (R)0;
  }
  cp_async_wait0();
  __syncthreads();
  for (int K = L - 1, ks = (L - 1) % nslot; K >= 0; --K) {
    const R* x = acc + ks * m0;
    // d >= 1: row K - d loses M_{K,K-d}^T x_K; d = 0: row K - D - 1 enters as Delta^-1 z
    const int live = (K >= D1) ? items : (K + 1) * m0;
    for (int h = 0; h < nch; ++h, st ^= 1) {
      const double* cs = cf + (size_t)st * maxstage;
      if (h + 1 < nch) stage(Tbwd + (size_t)K * bst, bst, items, h + 1, st ^ 1);
      else if (K > 0) stage(Tbwd + (size_t)(K - 1) * bst, bst, items, 0, st ^ 1);
      cp_async_commit();
      if (zero && h == 0) {
        if (K < a || !side) Wc[at(K, mu0)] = (double)x[mu0];   // (the middle by side 0)
        if (K - D1 - 1 >= 0) zb[((K - 1) & 1) * m0 + mu0] = nr;
        if (K - D1 - 2 >= 0) nr = (R)Wc[at(K - D1 - 2, mu0)];
      }
      const int qa = h * qc, qn = min(qc, m0 - qa);
      for (int it = nth - 1 - tid; it < live; it += nth) {
        const int d = it / m0, mu = it % m0, back = (d == 0) ? D1 : d;
        if (d == 0 && K < D1) continue;
        R* a = acc + (ks - back < 0 ? ks - back + nslot : ks - back) * m0 + mu;
        const R* v = ((d == 0) ? zb + (K & 1) * m0 : x) + qa;
        R s = (d != 0) ? -*a : (h == 0) ? (R)0 : *a;
#pragma unroll 8
        for (int q = 0; q < qn; ++q) s += (R)cs[q * items + it] * v[q];
        *a = (d == 0) ? s : -s;
      }
      cp_async_wait0();
      __syncthreads();
    }
    ks = (ks == 0) ? nslot - 1 : ks - 1;
  }
  if (T.twist) cl_wait();
}

// maxcol: the largest m0 (m0 + 1) (D + 3) among the tasks (shared doubles that
// hold a block column; capped at what the device has, the kernel then reads the
// column from global memory)
void launch_band_factor(const BandTask* t, int n, int maxcol, int maxm0, const BandSteps& cs, cudaStream_t st) {
  if (!n) return;
  FOCK_SMEM_OPTIN(k_band_factor);
  {
    static std::once_flag wide;
    std::call_once(wide, [] { cudaFuncSetAttribute(k_band_factor, cudaFuncAttributeNonPortableClusterSizeAllowed, 1); });
  }
  int dev = 0, mx = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int cap = (mx - 1024) / 8;
  const int doubles = std::min(cap, maxcol);
  // Clusters of 16 (where the device can place them) for few problems, smaller
  // ones as the problems alone fill the GPU.  64 cells of 8 functions, clusters of
  // 16 / 8 / 4: 1 problem 0.77 / 0.94 / 1.19 ms, 16 problems 0.88 / 1.03 / 1.19, 32
  // 0.94 / 1.04 / 1.19, 128 3.7 / 2.3 / 1.65; 64 cells of 16, 32 problems 3.4 / 3.1 /
  // 3.3; 64 cells of 32, 8 problems 16.0 / 11.7 / 18.4.
  int C = (n <= 4) ? 16 : (n <= 64) ? 8 : 4;
  if (n <= kColumnProblems && cs.steps && maxcol <= cap) {
    FOCK_SMEM_OPTIN(k_band_column);
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // CTAs per side: no more than the largest share of the pairs needs
    const int most = std::max(1, sms / (n * cs.sides)), share = (cs.pairs + most - 1) / most;
    const int cta = (cs.pairs + share - 1) / share;
    const dim3 grid((unsigned)cta, (unsigned)cs.sides, (unsigned)n);
    const int th = maxm0 > 16 ? kFactorThreads : 256;
    const size_t sm = (size_t)doubles * 8;
    k_band_column<<<grid, th, sm, st>>>(t, 0, 0);
    for (int i = 0; i < cs.steps; ++i) {
      if (std::binary_search(cs.middles.begin(), cs.middles.end(), i)) {
        k_band_column<<<grid, th, sm, st>>>(t, 2, i);
        k_band_column<<<grid, th, sm, st>>>(t, 3, i);
      }
      k_band_column<<<grid, th, sm, st>>>(t, 1, i);
    }
    k_band_column<<<dim3(1, 1, n), 32, 0, st>>>(t, 4, 0);
  }
  cudaLaunchConfig_t cfg = {};
  // (64 cells of 32 functions 6.5 ms with 256 threads, 5.9 with 512; of 8 0.76 and 0.82)
  cfg.blockDim = dim3(maxm0 > 16 ? kFactorThreads : 256);
  cfg.dynamicSmemBytes = (size_t)doubles * 8;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3((unsigned)(n * C));
  int room = 0;
  if (C == 16 && (cudaOccupancyMaxActiveClusters(&room, k_band_factor, &cfg) != cudaSuccess || room < n)) {
    cudaGetLastError();
    C = 8;
    at[0].val.clusterDim.x = C;
    cfg.gridDim = dim3((unsigned)(n * C));
  }
  cudaLaunchKernelEx(&cfg, k_band_factor, t, doubles);
}

// maxitem: the largest (D + 4) m0 among the tasks, maxrow: the largest band_side_rows,
// maxstep: the largest step (coefficient doubles), max8: the largest band_stage_rows8, sides: 2 if any task is twisted
template <typename R, bool MULTI>
static void solve_go(const BandTask* t, int n, int kmax, int maxitem, int maxrow, int maxstage, int sides, cudaStream_t st) {
  FOCK_SMEM_OPTIN((k_band_solve<R, MULTI>));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(kmax * sides), (unsigned)n);
  cfg.blockDim = dim3(std::min(1024, std::max(64, (maxitem + 31) & ~31)));
  cfg.dynamicSmemBytes = ((size_t)2 * maxstage + (size_t)maxrow) * sizeof(double);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = sides;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_band_solve<R, MULTI>, t, sides, maxstage);
}
void launch_band_solve(const BandTask* t, int n, int kmax, int maxitem, int maxrow, int maxstep, int max8, int sides,
                       cudaStream_t st, bool mixed) {
  if (!n) return;
  // A stage holds a step up to 64 KB, or as many rows of one (8 where there is room).  Two
  // stages are enough and leave room for several CTAs per SM: eight give the same
  // 98 us on one chain of 64 cells of 8 functions, three 929 us against 674 on 32
  // chains of 64 cells of 16.  Pieces of 32 KB instead of 64: 72 columns of 512 cells
  // of 32 functions 5.8 ms against 4.9.
  int dev = 0, mx = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int maxstage = band_stage(maxstep, max8, maxrow, (mx - 1024) / 8);
  if (maxstep <= maxstage) {
    solve_go<double, false>(t, n, kmax, maxitem, maxrow, maxstage, sides, st);
    if (mixed) solve_go<float, false>(t, n, kmax, maxitem, maxrow, maxstage, sides, st);
  } else {
    solve_go<double, true>(t, n, kmax, maxitem, maxrow, maxstage, sides, st);
    if (mixed) solve_go<float, true>(t, n, kmax, maxitem, maxrow, maxstage, sides, st);
  }
}

}  // namespace fock
