// Rayleigh-Ritz step of the block iteration: the k lowest eigenpairs of the
// pencil (Y^T H Y, Y^T S Y) of a basis Y = [X | P | W] whose columns may be
// numerically dependent.  One thread-block cluster of C CTAs per problem.
//
//  1. scale by D = diag(Y^T S Y)^-1/2; L D L^T factorisation of the scaled S-Gram
//     with diagonal pivoting, stopping when the largest remaining pivot falls
//     below the drop threshold (the remaining columns are numerically in the span
//     of the kept ones, as are zero columns), with every elimination step applied
//     to the H-Gram from both sides and to L^-1 as it goes;
//  2. Householder reduction of C = Delta^-1/2 L^-1 (D GH D) L^-T Delta^-1/2 to a
//     tridiagonal T;
//  3. the kk lowest eigenvalues of T by FP32 Sturm multisection, one FP64
//     inverse-iteration vector each (clusters of shifts in turn), Cholesky-QR, a
//     Rayleigh-Ritz step in the vectors' span;
//  4. back-transformation and coefficients D L^-T Delta^-1/2 w in the Y basis.
//
// Bound by FP64 latency and by the FP64 pipe of the SMs it occupies (about
// 1.7 multiply-adds a cycle each, 64 cycles from a multiply-add to the next one
// that needs it), so the design spreads every step over C SMs and keeps the
// dependent chain of a step short.  Rows of the working matrices are dealt
// cyclically to the CTAs and live in their shared memory (two matrices), as
// full rows: a step needs one row of another CTA, which is read or pushed
// through distributed shared memory, and one cluster barrier (450 cycles).
// Small sequential decisions (pivots, reflectors, shifts, the kk x kk factors)
// are repeated in every CTA from equal data, so all CTAs take the same branches
// through the same sequence of barriers, and no sum's order depends on C: the
// result is the same for every cluster size, which the launch picks by how many
// problems share the GPU.
//
// Measured per launch, against a form with the substitutions as phases of their
// own, serial dot products and the matrices of large bases in L2: one problem of 60
// columns 690 -> 450 us, 32 of them 690 -> 480, one of 216 columns 6.3 -> 2.2 ms.
#include <float.h>

#include <algorithm>

#include "common.cuh"
#include "jacobi.cuh"

namespace fock {

namespace {

constexpr int kRRThreads = 256;
constexpr int kRRMax = 256;        // columns of a basis, at most 255
constexpr int kRRBack = 8;         // reflectors per block of the back-transformation
constexpr int kRRCols = 3;         // wanted vectors, at most 85, by 32

// Shifts closer than kShiftCluster ||T|| form a cluster.  The FP32
// multisection places a shift within a few FP32 units of ||T|| of its
// eigenvalue, so two shifts in one such window can both lie much nearer one
// of the two eigenvalues; inverse iteration then turns both vectors into that
// one eigenvector, the Cholesky-QR below meets a singular Gram matrix, and
// the Ritz basis built from it loses rank.  Exactly degenerate pairs (a ring
// with two identical, distant defects) split, as the block iteration
// converges, by about lambda res^2, which crosses that window.  A cluster's
// vectors are therefore computed by one thread in turn, each orthogonalised
// against the cluster's earlier vectors after every solve (the
// reorthogonalisation of LAPACK's inverse iteration, dstein).
constexpr double kShiftCluster = 32.0 * FLT_EPSILON;
// The multisection's own resolution is far finer than that bound wherever
// ||T|| is far above the wanted eigenvalues (the Rayleigh-Ritz matrices of
// box chains), and clusters of the bound's width there chain long runs of
// well separated shifts into one thread.  So clusters are first tight
// (shifts whose final brackets lie within twice their widths: the ones the
// multisection could not tell apart), and the wide clusters are taken only
// when the first Cholesky factor of the vectors' Gram matrix meets a pivot
// below kDepPivot (a unit vector within 1e-5 of the span of the earlier ones).
constexpr double kDepPivot = 1e-10;
// Vectors whose Gram matrix has all pivots above this are orthonormal to a few
// rounding units after one Cholesky-QR pass; below it they take a second one.
constexpr double kGoodPivot = 0.5;

// Whether shift q (> 0) joins the cluster of shift q - 1: tight (brackets lo,
// hi of the multisection) or wide (kShiftCluster ||T||, tnorm = ||T||).
__device__ inline bool shift_clustered(const double* lam, const float* lo, const float* hi, int q,
                                       float tnorm, bool wide) {
  const double gap = lam[q] - lam[q - 1];
  if (wide) return gap <= kShiftCluster * (double)tnorm;
  const double w = (double)(hi[q] - lo[q]) + (double)(hi[q - 1] - lo[q - 1]);
  return gap <= 2.0 * w + 4.0 * FLT_EPSILON * fmax(fabs(lam[q]), fabs(lam[q - 1]));
}

// One inverse-iteration vector of the symmetric tridiagonal (d, e) of order r
// for the shift lm: LU with partial pivoting of T - lm I (pivots below eps
// raised to eps), start vector from a counter hash of (row, c), three sweeps of
// solve and normalisation.  zs: the vectors found so far, entry (i, q) at
// zs[i kk + q]; columns c0..c-1 (the earlier vectors of c's cluster,
// orthonormal) are projected out after every solve; the result goes to column
// c.  ws: 6 r doubles, entry (i, f) at ws[(6 i + f) sw] (threads side by side).
__device__ void inverse_iteration(const double* d, const double* e, int r, double lm, double eps,
                                  double* ws, int sw, double* zs, int kk, int c, int c0) {
  auto W = [&](int i, int f) -> double& { return ws[(size_t)(6 * i + f) * sw]; };   // 0 multiplier, 1 reciprocal
  const long long eps_bits = abs_bits(eps);   // pivot, 2 and 3 the row's other entries, 4 swap flag, 5 the vector
  double a0 = d[0] - lm, a1 = (r > 1) ? e[0] : 0.0;
  for (int i = 0; i + 1 < r; ++i) {
    const double sub = e[i], dn = d[i + 1] - lm, sn = (i + 2 < r) ? e[i + 1] : 0.0;
    const bool sw2 = abs_bits(sub) > abs_bits(a0);
    double p0 = sw2 ? sub : a0;
    const double p1 = sw2 ? dn : a1, p2 = sw2 ? sn : 0.0;
    const double o0 = sw2 ? a0 : sub, o1 = sw2 ? a1 : dn, o2 = sw2 ? 0.0 : sn;
    if (abs_bits(p0) < eps_bits) p0 = (__double_as_longlong(p0) < 0) ? -eps : eps;   // tiny pivot raised to eps
    const double rq = rcp_nr(p0);
    const double m = o0 * rq;
    W(i, 0) = m; W(i, 1) = rq; W(i, 2) = p1; W(i, 3) = p2; W(i, 4) = sw2 ? 1.0 : 0.0;
    a0 = fma(-m, p1, o1);
    a1 = fma(-m, p2, o2);
  }
  if (abs_bits(a0) < eps_bits) a0 = (__double_as_longlong(a0) < 0) ? -eps : eps;
  W(r - 1, 1) = rcp_nr(a0);
  W(r - 1, 2) = 0.0; W(r - 1, 3) = 0.0;
  if (r >= 2) W(r - 2, 3) = 0.0;
  // start vector: counter hash of (row, vector), uniform in [0.5, 1.5)
  for (int i = 0; i < r; ++i) {
    const uint32_t h = (uint32_t)(splitmix64(((uint64_t)(c + 1) << 32) | (uint64_t)(i + 1)) >> 40);
    W(i, 5) = 0.5 + (double)h * (1.0 / 16777216.0);
  }
  for (int sweep = 0; sweep < 3; ++sweep) {
    double zi = W(0, 5);
    for (int i = 0; i + 1 < r; ++i) {                // P and L^-1
      const double zn = W(i + 1, 5);
      const bool sw2 = __double_as_longlong(W(i, 4)) != 0;
      const double bi = sw2 ? zn : zi, bn = sw2 ? zi : zn;
      W(i, 5) = bi;
      zi = fma(-W(i, 0), bi, bn);
    }
    W(r - 1, 5) = zi;
    const bool last = sweep == 2;
    double nxt = 0.0, nxt2 = 0.0, nn = 0.0;          // U^-1, and the squared norm
    for (int i = r - 1; i >= 0; --i) {
      double s = fma(-W(i, 3), nxt2, W(i, 5));
      s = fma(-W(i, 2), nxt, s);
      s *= W(i, 1);
      W(i, 5) = s;
      if (last) nn = fma(s, s, nn);
      nxt2 = nxt; nxt = s;
    }
    // (a sweep grows the vector by at most 1 / eps: three stay far inside the
    // range, so the norm is taken once unless there are vectors to project out)
    if (!last && c0 == c) continue;
    if (c0 < c) {                                    // the cluster's earlier vectors projected out
      for (int p = c0; p < c; ++p) {
        double dp = 0.0;
        for (int i = 0; i < r; ++i) dp = fma(zs[(size_t)i * kk + p], W(i, 5), dp);
        for (int i = 0; i < r; ++i) W(i, 5) = fma(-dp, zs[(size_t)i * kk + p], W(i, 5));
      }
      nn = 0.0;
      for (int i = 0; i < r; ++i) nn = fma(W(i, 5), W(i, 5), nn);
    }
    const double inv = (nn > 0.0 && isfinite(nn)) ? rsqrt_nr(nn) : 0.0;
    for (int i = 0; i < r; ++i) W(i, 5) *= inv;
  }
  for (int i = 0; i < r; ++i) zs[(size_t)i * kk + c] = W(i, 5);
}

// Barrier of the cluster (of the CTA alone for C = 1).  The hardware cluster
// barrier: arrive has release and wait acquire semantics at cluster scope, for
// shared memory of the cluster and global memory alike.
template <int C> __device__ __forceinline__ void group_sync() {
  if (C == 1) __syncthreads();
  else asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the same shared-memory location in CTA q of the cluster
template <int C, typename V> __device__ __forceinline__ V* peer(V* p, int q) {
  if (C == 1) return p;
  V* o;
  asm("mapa.u64 %0, %1, %2;" : "=l"(o) : "l"(p), "r"(q));
  return o;
}

__host__ __device__ inline int rr_pitch(int n) { return ((n + 15) & ~15) + 8; }   // two rows apart in the banks

}  // namespace

// doubles of dynamic shared memory of a CTA: two working matrices of the rows
// it owns; later the vectors (one CTA), the kk x kk matrices of the projected step
size_t rr_doubles(int n, int k, int C) {
  const size_t rows = (n + C - 1) / C, mats = 2 * rows * rr_pitch(n), sq = (size_t)(k + 1) * (k + 1);
  const size_t late = (C == 1) ? (size_t)n * k + std::max((size_t)n * k, sq) + sq : 2 * sq;
  const size_t own = (k + C - 1) / C, back = (own + kRRBack) * (n | 1) + kRRBack * (own + kRRBack);
  return std::max(std::max(mats, late), back + (C == 1 ? (size_t)n * k : 0));
}

template <int C>
__global__ void __launch_bounds__(kRRThreads) k_rr(const RRTask* __restrict__ tasks, int cls, int msize) {
  const RRTask T = tasks[blockIdx.x / C];
  if (T.cls != cls) return;                 // the other launch's problems (the same for the whole cluster)
  if (T.active && *T.active == 0) return;
  extern __shared__ __align__(16) double sm[];
  constexpr int NT = kRRThreads, NW = NT / 32;
  const int rank = (C == 1) ? 0 : (int)(blockIdx.x % C);
  const int n = T.nb, ld = T.ld, k = T.k, P = rr_pitch(n), nl = (n + C - 1) / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // basis directions whose S-independent part is below kDropRel are dropped:
  // 1e-10 with FP64 images, 1e-6 while the images are FP32 (their noise level)
  const double kDropRel = (T.mode && *T.mode) ? 1e-6 : 1e-10;
  double* M1 = sm;                          // local rows of the S-Gram / L^-1, then of the reduced matrix
  double* M2 = sm + (size_t)nl * P;         // local rows of the H-Gram
  const size_t l2 = (size_t)ld * ld;
  double* Kg = T.work;                      // Delta^-1/2 L^-1 D, row per kept pivot, stride ld
  double* Vg = T.work + l2;                 // Householder vectors, row per reflector, stride ld
  double* Zg = T.work + 2 * l2;             // (C > 1) eigenvectors of T, r x kk
  double* Tg = T.work + 3 * l2;             // (C > 1) T Z
  double* Gg = T.work + 4 * l2;             // (C > 1) kk x kk products
  __shared__ double dsc[kRRMax], dg[kRRMax], rl[kRRMax], dpv[kRRMax];
  __shared__ double bufA[2][kRRMax], bufB[2][kRRMax], bufC[2][kRRMax], bufD[2][kRRMax], xr[kRRMax];
  __shared__ double td[kRRMax], te[kRRMax], ttau[kRRMax], tlam[kRRMax];
  __shared__ int perm[kRRMax], pos[kRRMax], act[kRRMax], apos[kRRMax];
  __shared__ int s_p[2];
  __shared__ double s_rd[2], s_K;
  // ---- 1. scaled Gram matrices, pivoted elimination ----
  for (int i = tid; i < n; i += NT) {
    const double g = T.GS[(size_t)i + (size_t)ld * i];
    const double s = (g > 0.0) ? rsqrt_nr(g) : 0.0;
    dsc[i] = s;
    dg[i] = g * (s * s);
    act[i] = apos[i] = i;
    pos[i] = n;                             // not eliminated
  }
  __syncthreads();
  for (int it = tid; it < nl * n; it += NT) {
    const int la = it / n, b = it % n, a = rank + C * la;
    if (a >= n) continue;
    const double gs = 0.5 * (T.GS[(size_t)b + (size_t)ld * a] + T.GS[(size_t)a + (size_t)ld * b]);
    const double gh = 0.5 * (T.GH[(size_t)b + (size_t)ld * a] + T.GH[(size_t)a + (size_t)ld * b]);
    const double sc = dsc[a] * dsc[b];
    M1[la * P + b] = gs * sc;
    M2[la * P + b] = gh * sc;
  }
  // the next pivot (warp 0): the largest remaining diagonal (bit-pattern keys,
  // ties to the lower index); -1 when it is not above the drop threshold
  auto pick = [&](int j) {
    long long bk = -2;
    int bi = n;
    for (int t = lane; t < n - j; t += 32) {
      const int b = act[t];
      const long long kq = pivot_key(dg[b]);
      if (kq > bk || (kq == bk && b < bi)) { bk = kq; bi = b; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const long long ok = __shfl_xor_sync(0xffffffffu, bk, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ok > bk || (ok == bk && oi < bi)) { bk = ok; bi = oi; }
    }
    if (lane == 0) {
      const double dj = (bk >= 0) ? dg[bi] : 0.0;
      const bool ok = bk > __double_as_longlong(kDropRel);   // the diagonal scale is 1
      s_p[j & 1] = ok ? bi : -1;
      s_rd[j & 1] = ok ? rcp_nr(dj) : 0.0;
    }
  };
  if (warp == 0) pick(0);
  group_sync<C>();
  // Step j, pivot p, l = G(:, p) / delta over the remaining indices: G loses l times
  // row p, H loses l u^T + u l^T with u = H(:, p) - l H(p, p) / 2 (the elimination
  // from both sides at once); rows eliminated earlier lose only the column
  // operation.  The row of an eliminated index keeps its part of L^-1 in the
  // columns of M1 that are eliminated too.  Row p of M2 takes its own column
  // operation a step later, since other CTAs read the row during this step.
  int r = 0, pprev = -1;
  for (; r < n; ++r) {
    const int j = r, p = s_p[j & 1];
    if (p < 0) break;                       // the same in every CTA
    const double rd = s_rd[j & 1];
    double *lv = bufA[j & 1], *uv = bufB[j & 1], *kv = bufC[j & 1];
    const double* gk = peer<C>(M1 + (size_t)(p / C) * P, p % C);
    const double* hr = peer<C>(M2 + (size_t)(p / C) * P, p % C);
    for (int b = tid; b < n; b += NT) {
      const double g = gk[b], h = hr[b], hpp = hr[p];
      const bool live = b != p && pos[b] == n;
      const double l = live ? g * rd : 0.0;
      lv[b] = l;
      uv[b] = live ? fma(-0.5 * l, hpp, h) : 0.0;
      kv[b] = g;
      if (live) dg[b] = fma(-l, g, dg[b]);
    }
    __syncthreads();
    if (tid == 0) {                         // p leaves the list of remaining indices
      perm[j] = p;
      dpv[j] = dg[p];
      pos[p] = j;
      const int q = apos[p], last = act[n - 1 - j];
      act[q] = last;
      apos[last] = q;
    }
    __syncthreads();
    const int cnt = n - 1 - j;
    if (warp == 0) pick(j + 1);
    const double* lp = bufA[(j & 1) ^ 1];
    for (int la = (warp + NW - 1) % NW; la < nl; la += NW) {   // (warp 0 last: it has the pivot to find)
      const int a = rank + C * la;
      if (a >= n || a == p) continue;
      double *r1 = M1 + (size_t)la * P, *r2 = M2 + (size_t)la * P;
      if (pos[a] == n) {
        const double l = -lv[a], u = -uv[a];
        for (int b = lane; b < n; b += 32) r1[b] = (b == p) ? l : fma(l, kv[b], r1[b]);
        for (int t = lane; t < cnt; t += 32) {
          const int b = act[t];
          r2[b] = fma(u, lv[b], fma(l, uv[b], r2[b]));
        }
      } else {
        if (a == pprev) {
          const double h = -r2[a];
          for (int b = lane; b < n; b += 32) r2[b] = fma(h, lp[b], r2[b]);   // (zero at eliminated columns)
          __syncwarp();
        }
        const double x = -r2[p];
        for (int t = lane; t < cnt; t += 32) {
          const int b = act[t];
          r2[b] = fma(x, lv[b], r2[b]);
        }
      }
    }
    pprev = p;
    group_sync<C>();
  }
  if (r < k && rank == 0 && tid == 0 && T.fail) *T.fail = 1;
  const int kk = min(k, r);
  for (int a = tid; a < r; a += NT) rl[a] = rsqrt_nr(dpv[a]);
  __syncthreads();
  for (int la = warp; la < nl; la += NW) {   // Delta^-1/2 L^-1 D, by position
    const int i = rank + C * la, q = (i < n) ? pos[i] : n;
    if (q >= r) continue;
    for (int b = lane; b < n; b += 32) {
      const double x = (b == i) ? 1.0 : (pos[b] < q) ? M1[(size_t)la * P + b] : 0.0;
      Kg[(size_t)q * ld + b] = x * (rl[q] * dsc[b]);
    }
  }
  group_sync<C>();
  // reduced matrix by position: entry (a, b) stands in the row eliminated first
  for (int it = tid; it < nl * r; it += NT) {
    const int la = it / r, b = it % r, a = rank + C * la;
    if (a >= r) continue;
    const int i = perm[min(a, b)], c = perm[max(a, b)];
    M1[(size_t)la * P + b] = peer<C>(M2 + (size_t)(i / C) * P, i % C)[c] * (rl[a] * rl[b]);
  }
  group_sync<C>();
  // ---- 2. tridiagonal reduction ----
  // One cluster barrier per column.  At step q every CTA holds row q of the
  // reduced matrix (xr) and makes the same reflector v from it (warp 0) while the
  // other warps apply the previous step's rank-2 update to the local rows; then
  // p = tau A v for the local rows and, by its owner, row q + 1 are pushed to all
  // CTAs.  After the barrier every CTA has w = p - (tau / 2)(v^T p) v and the
  // updated row q + 1.  bufA v, bufB w, bufC p, bufD the pushed row, by parity:
  // a CTA pushes into a buffer again only after a barrier that all reach once
  // they are done with its last contents.
  if (r > 0) {
    for (int i = tid; i < r; i += NT) xr[i] = peer<C>(M1, 0)[i];
    group_sync<C>();
    for (int q = 0; q + 1 < r; ++q) {
      const int par = q & 1;
      double *v = bufA[par], *w = bufB[par], *pp = bufC[par], *xn = bufD[par];
      if (warp == 0) {
        double s = 0.0;
        for (int i = q + 1 + lane; i < r; i += 32) s = fma(xr[i], xr[i], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const double x0 = xr[q + 1];
        double alpha = x0, tk = 0.0;
        if (q + 2 < r) {
          // (signs by bit pattern: an FP64 compare holds the pipe like a multiply-add)
          const double xnorm = (__double_as_longlong(s) > 0) ? s * rsqrt_nr(s) : 0.0;
          alpha = (__double_as_longlong(x0) > 0) ? -xnorm : xnorm;
          const double den = fma(-x0, alpha, s);
          tk = (__double_as_longlong(den) > 0) ? rcp_nr(den) : 0.0;
        }
        for (int i = q + 1 + lane; i < r; i += 32) v[i] = (i == q + 1) ? x0 - alpha : xr[i];
        if (lane == 0) { td[q] = xr[q]; te[q] = alpha; ttau[q] = tk; }
      } else if ((warp & 3) != 0 && q > 0 && __double_as_longlong(ttau[q - 1]) != 0) {
        // (not the warps of warp 0's sub-partition: its FP64 unit is the reflector's)
        const double *vo = bufA[par ^ 1], *wo = bufB[par ^ 1];
        const int l0 = (q >= rank) ? (q - rank) / C + 1 : 0;   // first local row > q
        for (int la = l0 + warp - 1 - (warp >> 2); la < nl; la += NW - NW / 4) {
          const int a = rank + C * la;
          if (a >= r) break;
          const double va = -vo[a], wa = -wo[a];
          double* row = M1 + (size_t)la * P;
          for (int b = ((q + 1) & ~31) + lane; b < r; b += 32)
            if (b > q) row[b] = fma(wa, vo[b], fma(va, wo[b], row[b]));
        }
      }
      __syncthreads();
      const double tk = ttau[q];
      if ((q + 1) % C == rank)
        for (int i = q + 1 + tid; i < r; i += NT) {
          const double x = M1[(size_t)((q + 1) / C) * P + i];
          for (int c = 0; c < C; ++c) peer<C>(xn, c)[i] = x;
        }
      if (__double_as_longlong(tk) != 0) {
        if (rank == 0)
          for (int i = q + 1 + tid; i < r; i += NT) Vg[(size_t)q * ld + i] = v[i];
        // 8 lanes per row, lane o of a group over the columns = o mod 8
        const int grp = tid >> 3, o = tid & 7;
        const int l0 = (q >= rank) ? (q - rank) / C + 1 : 0;
        for (int lb = l0; lb < nl; lb += NT / 8) {
          const int la = lb + grp, a = rank + C * la;
          const bool on = la < nl && a < r;
          double s = 0.0;
          if (on) {
            const double* row = M1 + (size_t)la * P;
            int b = ((q + 1) & ~7) + o;
            if (b <= q) b += 8;
            for (; b < r; b += 8) s = fma(row[b], v[b], s);
          }
          s += __shfl_xor_sync(0xffffffffu, s, 1);
          s += __shfl_xor_sync(0xffffffffu, s, 2);
          s += __shfl_xor_sync(0xffffffffu, s, 4);
          if (on)
            for (int c = o; c < C; c += 8) peer<C>(pp, c)[a] = tk * s;
        }
      }
      group_sync<C>();
      if (warp == 0 && __double_as_longlong(tk) != 0) {
        double s = 0.0;
        for (int i = q + 1 + lane; i < r; i += 32) s = fma(v[i], pp[i], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) s_K = 0.5 * tk * s;
      }
      __syncthreads();
      if (__double_as_longlong(tk) != 0) {
        const double K = s_K, v1 = v[q + 1], w1 = fma(-K, v1, pp[q + 1]);
        for (int i = q + 1 + tid; i < r; i += NT) {
          const double wi = fma(-K, v[i], pp[i]);
          w[i] = wi;
          xr[i] = fma(-w1, v[i], fma(-v1, wi, xn[i]));
        }
      } else {
        for (int i = q + 1 + tid; i < r; i += NT) xr[i] = xn[i];
      }
      __syncthreads();
    }
    if (tid == 0) { td[r - 1] = xr[r - 1]; te[r - 1] = 0.0; ttau[r - 1] = 0.0; }
    __syncthreads();
  }
  // ---- 3. the kk lowest eigenvalues of T: FP32 Sturm multisection, a warp per
  // eigenvalue (each round the lanes count below 32 interior points of its
  // bracket, which becomes 33 times narrower); eigenvalue c on CTA c mod C ----
  __shared__ float s_lo[kRRMax / 2], s_hi[kRRMax / 2], s_g[2], s_e2;
  float* df = reinterpret_cast<float*>(bufC[0]);   // d and e^2 in FP32
  float* e2f = df + kRRMax;
  for (int i = tid; i < r; i += NT) {
    df[i] = (float)td[i];
    e2f[i] = (i + 1 < r) ? (float)(te[i] * te[i]) : 0.0f;
  }
  __syncthreads();
  if (warp == 0) {                                 // Gershgorin bounds
    float glo = FLT_MAX, ghi = -FLT_MAX, emax2 = 0.0f;
    for (int i = lane; i < r; i += 32) {
      const float rad = (i > 0 ? sqrtf(e2f[i - 1]) : 0.0f) + (i + 1 < r ? sqrtf(e2f[i]) : 0.0f);
      glo = fminf(glo, df[i] - rad);
      ghi = fmaxf(ghi, df[i] + rad);
      emax2 = fmaxf(emax2, e2f[i]);
    }
    for (int o = 16; o > 0; o >>= 1) {
      glo = fminf(glo, __shfl_xor_sync(0xffffffffu, glo, o));
      ghi = fmaxf(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
      emax2 = fmaxf(emax2, __shfl_xor_sync(0xffffffffu, emax2, o));
    }
    if (lane == 0) { s_g[0] = glo; s_g[1] = ghi; s_e2 = emax2; }
  }
  __syncthreads();
  const float tnorm = fmaxf(fabsf(s_g[0]), fabsf(s_g[1]));
  {
    const float pivmin = FLT_MIN * fmaxf(1.0f, s_e2);
    const float glo = s_g[0] - (4.0f * FLT_EPSILON * tnorm + pivmin);
    const float ghi = s_g[1] + (4.0f * FLT_EPSILON * tnorm + pivmin);
    for (int c = rank + C * warp; c < kk; c += C * NW) {
      float lo = glo, hi = ghi;
      for (int round = 0; round < 40; ++round) {
        const float x = lo + (hi - lo) * ((float)(lane + 1) * (1.0f / 33.0f));
        const int cnt = sturm_count_f32(df, e2f, r, x, pivmin);
        const unsigned above = __ballot_sync(0xffffffffu, cnt > c);
        const int f = above ? __ffs(above) - 1 : 32;     // the first point above eigenvalue c
        float nlo = __shfl_sync(0xffffffffu, x, max(f - 1, 0)), nhi = __shfl_sync(0xffffffffu, x, min(f, 31));
        nlo = (f > 0) ? fmaxf(lo, nlo) : lo;
        nhi = (f < 32) ? fminf(hi, nhi) : hi;
        if (!(nlo < nhi)) nhi = nlo;                     // bracket collapsed to rounding
        const bool moved = nlo > lo || nhi < hi;
        lo = nlo;
        hi = nhi;
        if (!moved || !(hi - lo > 2.0f * FLT_EPSILON * fmaxf(fabsf(lo), fabsf(hi)) + pivmin)) break;
      }
      if (lane < C) {
        *peer<C>(s_lo + c, lane) = lo;
        *peer<C>(s_hi + c, lane) = hi;
        *peer<C>(tlam + c, lane) = 0.5 * ((double)lo + (double)hi);
      }
    }
  }
  group_sync<C>();
  // ---- inverse iteration: the cluster of shifts led by vector c on CTA c mod C;
  // tight clusters first, wide ones when the Gram factor below finds a dependent
  // vector (every CTA decides alike: the Gram matrices they factor are equal) ----
  double* Z = (C == 1) ? sm : Zg;                  // r x kk
  double* ws = (C == 1) ? sm + (size_t)r * kk : sm;
  const int room = msize - ((C == 1) ? r * kk : 0);
  const int nwk = max(1, min(NT, min((kk + C - 1) / C, room / (6 * max(r, 1)))));
  const double eps_ii = DBL_EPSILON * fmax((double)tnorm, DBL_MIN);
  auto zat = [&](int i, int c) { return (C == 1) ? Z[(size_t)i * kk + c] : __ldcg(Z + (size_t)i * kk + c); };
  auto vectors = [&](bool wide) {
    if (tid < nwk)
      for (int c = rank + C * tid; c < kk; c += C * nwk) {
        if (c > 0 && shift_clustered(tlam, s_lo, s_hi, c, tnorm, wide)) continue;   // its cluster's first thread
        for (int q = c; q < kk && (q == c || shift_clustered(tlam, s_lo, s_hi, q, tnorm, wide)); ++q)
          inverse_iteration(td, te, r, tlam[q], eps_ii, ws + tid, nwk, Z, kk, q, c);
      }
    group_sync<C>();
  };
  // kk x kk products of the columns of Z with those of B (lower triangle), shared
  // out over the cluster, into `out` (stride kj) of every CTA, mirrored
  const int kj = kk + 1;
  const size_t sq = (size_t)kj * kj;
  double* R1 = (C == 1) ? sm + (size_t)r * kk : sm + sq;   // T Z (one CTA), then the Jacobi vectors
  double* R2 = (C == 1) ? R1 + max((size_t)r * kk, sq) : sm;
  auto products = [&](const double* B, double* out) {
    const int np = kk * (kk + 1) / 2;
    const int lo = (int)((long long)np * rank / C), hi = (int)((long long)np * (rank + 1) / C);
    for (int t = lo + tid; t < hi; t += NT) {
      int c1 = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
      while ((c1 + 1) * (c1 + 2) / 2 <= t) ++c1;
      while (c1 * (c1 + 1) / 2 > t) --c1;
      const int c2 = t - c1 * (c1 + 1) / 2;
      double s = 0.0;
#pragma unroll 8
      for (int i = 0; i < r; ++i)
        s = fma(zat(i, c1), (C == 1) ? B[(size_t)i * kk + c2] : __ldcg(B + (size_t)i * kk + c2), s);
      double* o = (C == 1) ? out : Gg;
      o[c1 * kj + c2] = s;
      o[c2 * kj + c1] = s;
    }
    group_sync<C>();
    if (C > 1) {
      for (int it = tid; it < kk * kk; it += NT) {
        const int o = (it / kk) * kj + it % kk;
        out[o] = __ldcg(Gg + o);
      }
      group_sync<C>();                             // Gg is free again
    }
  };
  // Cholesky-QR: the Gram matrix of the vectors eliminated to its pivots delta and
  // inverse unit factor (as in phase 1, without pivoting), Z <- Z L^-T delta^-1/2.
  // Returns the smallest pivot.
  auto orthonormalise = [&](bool check_only, bool* dep) {
    double* G = R2;
    products(Z, G);
    double pmin = INFINITY;
    if (tid == 0) { s_rd[0] = rcp_nr(fmax(G[0], DBL_MIN)); dpv[0] = G[0]; }
    __syncthreads();
    for (int j = 0; j < kk; ++j) {
      const double rdj = s_rd[j & 1];
      double *lc = bufA[j & 1], *lo = bufA[(j & 1) ^ 1];
      for (int a = j + tid; a < kk; a += NT) {
        if (j > 0) G[a * kj + j - 1] = -lo[a];   // column j - 1 becomes L^-1 now that its step is done
        if (a > j) lc[a] = G[a * kj + j] * rdj;
      }
      __syncthreads();
      // rows a > j, columns b <= a: G or L^-1 minus l_a times row j (whose entries
      // right of j are those of column j, by symmetry)
      const int na = kk - j - 1;
      for (int it = tid; it < na * kk; it += NT) {
        const int a = j + 1 + it / kk, b = it % kk;
        if (b > a || b == j) continue;
        const double x = fma(-lc[a], (b < j) ? G[j * kj + b] : G[b * kj + j], G[a * kj + b]);
        G[a * kj + b] = x;
        if (a == j + 1 && b == j + 1) { dpv[j + 1] = x; s_rd[(j + 1) & 1] = rcp_nr(fmax(x, DBL_MIN)); }
      }
      __syncthreads();
    }
    for (int j = 0; j < kk; ++j) pmin = fmin(pmin, (dpv[j] == dpv[j]) ? dpv[j] : 0.0);
    if (dep) *dep = !(pmin >= kDepPivot);
    if (check_only && !(pmin >= kDepPivot)) { __syncthreads(); return pmin; }
    for (int c = tid; c < kk; c += NT) bufB[0][c] = rsqrt_nr(fmax(dpv[c], DBL_MIN));
    __syncthreads();
    // a warp per row of Z, in place (lane over columns: all read before any writes)
    for (int i = rank * NW + warp; i < r; i += C * NW) {
      double t[kRRCols];
#pragma unroll
      for (int u = 0; u < kRRCols; ++u) {
        const int c = lane + 32 * u;
        if (32 * u >= kk) break;
        double s = (c < kk) ? zat(i, c) : 0.0;
        const int qn = min(32 * u + 31, kk - 1);
        for (int q = 0; q < qn; ++q)
          if (q < c && c < kk) s = fma(G[c * kj + q], zat(i, q), s);
        t[u] = s;
      }
      __syncwarp();
#pragma unroll
      for (int u = 0; u < kRRCols; ++u) {
        const int c = lane + 32 * u;
        if (32 * u >= kk) break;
        if (c < kk) Z[(size_t)i * kk + c] = t[u] * bufB[0][c];
      }
    }
    group_sync<C>();
    return pmin;
  };
  int* ord = act;                                  // (the list of remaining indices is done with)
  if (kk > 0) {
    vectors(false);
    bool dep = false;
    double pmin = orthonormalise(true, &dep);
    if (dep) {                                     // uniform over the cluster
      group_sync<C>();
      vectors(true);
      pmin = orthonormalise(false, nullptr);
    }
    if (!(pmin >= kGoodPivot)) orthonormalise(false, nullptr);
    // ---- Rayleigh-Ritz in span(Z): Tz = Z^T (T Z), Jacobi (every CTA on its copy) ----
    double* tz = (C == 1) ? R1 : Tg;
    const int zlo = (int)((long long)r * rank / C), zhi = (int)((long long)r * (rank + 1) / C);
    for (int it = zlo * kk + tid; it < zhi * kk; it += NT) {
      const int i = it / kk, c = it % kk;
      double s = td[i] * zat(i, c);
      if (i > 0) s = fma(te[i - 1], zat(i - 1, c), s);
      if (i + 1 < r) s = fma(te[i], zat(i + 1, c), s);
      tz[it] = s;
    }
    group_sync<C>();
    products(tz, R2);
    const bool turned = cta_jacobi(R2, R1, kk, kj);
    for (int i = tid; i < kk; i += NT) {           // ascending order, ties by index, NaN last:
      double di = R2[i * kj + i];                  // the ranks are always a permutation
      if (isnan(di)) di = DBL_MAX;
      int rk = 0;
      for (int jj = 0; jj < kk; ++jj) {
        double dj = R2[jj * kj + jj];
        if (isnan(dj)) dj = DBL_MAX;
        rk += (dj < di) || (dj == di && jj < i);
      }
      ord[rk] = i;
    }
    __syncthreads();
    for (int i = rank * NW + warp; i < r; i += C * NW) {   // rows of Z Q in ascending order, in place
      double t[kRRCols];
#pragma unroll
      for (int u = 0; u < kRRCols; ++u) {
        const int c = lane + 32 * u;
        if (32 * u >= kk) break;
        const int oc = ord[min(c, kk - 1)];
        double s = 0.0;
        if (turned) {
          for (int q = 0; q < kk; ++q) s = fma(zat(i, q), R1[q * kj + oc], s);
        } else {
          s = zat(i, oc);
        }
        t[u] = s;
      }
      __syncwarp();
#pragma unroll
      for (int u = 0; u < kRRCols; ++u) {
        const int c = lane + 32 * u;
        if (32 * u >= kk) break;
        if (c < kk) Z[(size_t)i * kk + c] = t[u];
      }
    }
    for (int c = tid; c < kk; c += NT) tlam[c] = R2[ord[c] * kj + ord[c]];
    group_sync<C>();
  }
  // ---- 4. back-transformation z = H_0 ... H_{r-3} y of this CTA's vectors
  // (c = rank mod C), eight reflectors at a time: with V their vectors, S = V^T V,
  // w solves (diag(1 / tau) + striu(S)) w = V^T y and y loses V w, which is the
  // product of the eight (the compact WY form without its triangular factor);
  // 4 lanes per dot product ----
  const int nown = (kk > rank) ? (kk - rank + C - 1) / C : 0;
  const int ry = r | 1;                            // odd pitch: vectors side by side in the banks
  double* Y = sm;                                  // own vector m, entry a: Y[m ry + a]
  double* Vs = Y + (size_t)nown * ry;              // the block's vectors, pitch ry
  double* Ws = Vs + (size_t)kRRBack * ry;          // V^T y, then w: [q][m], pitch nown
  double* Ss = Ws + (size_t)kRRBack * nown;        // S[q][p]
  if (C == 1) {
    // Z is in the way: its columns go through the other end of the region first
    double* tmp = sm + msize - (size_t)r * kk;
    for (int it = tid; it < r * kk; it += NT) tmp[it] = Z[it];
    __syncthreads();
    Z = tmp;
  } else {
    __syncthreads();                               // the region held the projected matrices
  }
  for (int it = tid; it < r * nown; it += NT) {
    const int a = it / nown, m = it % nown;
    Y[(size_t)m * ry + a] = zat(a, rank + C * m);
  }
  for (int q0 = ((r - 3) / kRRBack) * kRRBack; r >= 3 && q0 >= 0; q0 -= kRRBack) {
    __syncthreads();
    for (int it = tid; it < kRRBack * r; it += NT) {
      const int q = it / r, i = it % r;
      Vs[(size_t)q * ry + i] = (q0 + q <= r - 3 && i > q0 + q && __double_as_longlong(ttau[q0 + q]) != 0)
                                   ? __ldcg(Vg + (size_t)(q0 + q) * ld + i) : 0.0;
    }
    __syncthreads();
    const int nd = kRRBack * nown + kRRBack * (kRRBack - 1) / 2;   // V^T y and the upper part of S
    const int ndr = (4 * nd + 31) & ~31;
    for (int it = tid; it < ndr; it += NT) {
      const int t = it >> 2, o = it & 3;
      const bool on = t < nd;
      const double *x = Vs, *z = Vs;
      double* out = Ws;
      if (on && t < kRRBack * nown) {
        x = Vs + (size_t)(t / nown) * ry;
        z = Y + (size_t)(t % nown) * ry;
        out = Ws + t;
      } else if (on) {
        int p = 1, e = t - kRRBack * nown;         // (q, p), q < p, in the order (0,1) (0,2) (1,2) ...
        while (e >= p) { e -= p; ++p; }
        x = Vs + (size_t)e * ry;
        z = Vs + (size_t)p * ry;
        out = Ss + e * kRRBack + p;
      }
      double s = 0.0;
      if (on)
        for (int i = ((q0 + 1) & ~3) + o; i < r; i += 4) s = fma(x[i], z[i], s);
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      if (on && o == 0) *out = s;
    }
    __syncthreads();
    for (int m = tid; m < nown; m += NT) {
      double w[kRRBack];
#pragma unroll
      for (int q = kRRBack - 1; q >= 0; --q) {
        double s = Ws[q * nown + m];
#pragma unroll
        for (int p = kRRBack - 1; p > q; --p) s = fma(-Ss[q * kRRBack + p], w[p], s);
        w[q] = (q0 + q <= r - 3) ? s * ttau[q0 + q] : 0.0;
        Ws[q * nown + m] = w[q];
      }
    }
    __syncthreads();
    const int i0 = q0 + 1, ni = r - i0;
    for (int it = tid; it < ni * nown; it += NT) {
      const int i = i0 + it % ni, m = it / ni;
      double s = Y[(size_t)m * ry + i];
#pragma unroll
      for (int q = 0; q < kRRBack; ++q) s = fma(-Vs[(size_t)q * ry + i], Ws[q * nown + m], s);
      Y[(size_t)m * ry + i] = s;
    }
  }
  __syncthreads();
  if (rank == 0)
    for (int c = tid; c < k; c += NT) T.lam[c] = (c < kk) ? tlam[c] : NAN;
  // coefficients z[b] = sum_a Kg[a][b] y[a] of this CTA's vectors, four at a time
  // (Kg is zero for positions a before b's own); the second block is z with the
  // first k rows zeroed
  const int nq = (nown + 3) / 4, nb32 = (n + 31) & ~31;
  for (int it = tid; it < nq * nb32; it += NT) {
    const int b = it % nb32, m0 = (it / nb32) * 4;
    const int a0 = __reduce_min_sync(0xffffffffu, (b < n) ? pos[b] : n);
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    if (b < n) {
#pragma unroll 4
      for (int a = a0; a < r; ++a) {
        const double x = __ldcg(Kg + (size_t)a * ld + b);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (m0 + u < nown) s[u] = fma(x, Y[(size_t)(m0 + u) * ry + a], s[u]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (m0 + u < nown) {
          const int c = rank + C * (m0 + u);
          T.Cc[(size_t)ld * c + b] = s[u];
          T.Cc[(size_t)ld * (k + c) + b] = (b < k) ? 0.0 : s[u];
        }
    }
  }
  for (int c = kk + rank; c < k; c += C)           // fewer directions than wanted pairs: zero columns
    for (int b = tid; b < n; b += NT) T.Cc[(size_t)ld * c + b] = T.Cc[(size_t)ld * (k + c) + b] = 0.0;
  group_sync<C>();                                 // no CTA leaves while another may read its rows
}

template <int C>
static void rr_go(const RRTask* t, int ntask, int cls, int n, int k, cudaStream_t st) {
  FOCK_SMEM_OPTIN(k_rr<C>);
  const int msize = (int)rr_doubles(n, k, C);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ntask * C));
  cfg.blockDim = dim3(kRRThreads);
  cfg.dynamicSmemBytes = (size_t)msize * sizeof(double);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = (C > 1) ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k_rr<C>, t, cls, msize);
}

// Whether the device can place clusters of 16 (not a portable size).
static bool rr_wide() {
  static int room = -1;
  static std::once_flag once;
  std::call_once(once, [] {
    FOCK_SMEM_OPTIN(k_rr<16>);
    cudaFuncSetAttribute(k_rr<16>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(kRRThreads);
    cfg.dynamicSmemBytes = rr_doubles(kRRMax - 1, (kRRMax - 1) / 3, 16) * sizeof(double);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 16;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&room, k_rr<16>, &cfg) != cudaSuccess) { room = 0; cudaGetLastError(); }
  });
  return room > 0;
}

// The tasks of class cls (rr_class); n, k: the largest basis and wanted count
// among them.
void launch_rr(const RRTask* t, int ntask, int cls, int n, int k, cudaStream_t st) {
  if (!ntask || n <= 0) return;
  // CTAs per problem: few problems take more SMs each, many share them (60
  // columns, clusters of 1 / 2 / 4 / 8: 1 problem 606 / 519 / 453 / 442 us, 32
  // problems 630 / 544 / 482 / 495, 64 problems 630 / 541 / 542 / 882, 256 problems
  // 784 / 1119 / 1487 / 2537; clusters of 8 / 16: 108 columns 856 / 832, 216 columns
  // 1 problem 2652 / 2244, 8 problems 2731 / 4440)
  if (cls == 0) {
    if (ntask * 4 <= 152) rr_go<4>(t, ntask, cls, n, k, st);
    else if (ntask * 2 <= 152) rr_go<2>(t, ntask, cls, n, k, st);
    else rr_go<1>(t, ntask, cls, n, k, st);
  } else if (ntask <= 2 && rr_wide()) {
    rr_go<16>(t, ntask, cls, n, k, st);
  } else {
    rr_go<8>(t, ntask, cls, n, k, st);
  }
}

}  // namespace fock
