// Stage (b) and the Fourier side of stage (c).
//
//  k_fblocks   one CTA per Fourier index j: forms the m0 x m0 Hermitian pair
//              (Hbar_j, Sbar_j) and, on request, stores it, finds its lowest
//              eigenvalue or its eigenvectors, Hbar u = l Sbar u, in FP64.
//     source FACTORS (periodic lattice, Thm. 3.3 with the CP rank of the
//       potential, Remark 3.5): Hbar_j = 1/2 sum_p (prod_{l!=p} Shat_l) Ahat_p
//       - sum_t w_t prod_l Mhat_{l,t}, Sbar_j = prod_l Shat_l, elementwise in
//       (mu, nu), each factor picked at the axis component j_l;
//     source TOEPLITZ (box chain, Remark 3.2): the size-M block circulant
//       that embeds the symmetric block Toeplitz matrix with generators
//       T_d = block (k+d, k), |d| <= D: Chat_j = T_0 + sum_d (w^{jd} T_d +
//       w^{-jd} T_d^T), w = exp(-2 pi i / M) (Eq. A.3 convention).
//     eigensolver: Cholesky Sbar = L L^H and C = L^-1 Hbar L^-H when the
//       factor certifies that Sbar has no eigenvalue at or below tau (the
//       dependency cut; lambda_min >= 1 / ||L^-1||_F^2 > tau), else the
//       Jacobi eigendecomposition Sbar = Q diag(s) Q^H,
//       X = Q_K diag(s_K)^-1/2 over the kept directions K = {s > tau} (tau the
//       problem's dependency cut: every direction when none is numerically
//       singular, so C = X^H Hbar X has the pencil's eigenvalues exactly) --
//       then the eigenvectors of C by Jacobi, or Householder reduction to a real
//       tridiagonal and Sturm-sequence bisection for the lowest eigenvalue of an
//       embedding block (preconditioner shift only: 1e-9 relative). One warp
//       per block for m0 <= 8.
//  k_pf_*       the spectra of periodic lattices by the same reductions: a
//               pipeline over chunks of blocks, described there. Eigenvalues
//               ascend within a block, removed directions report +inf.
//  k_sigma      shift of the preconditioner: min_j lambda_min(Chat_j) - delta.
//  k_precond    K_j = (Chat_H,j - sigma Chat_S,j)^-1 per Fourier index.
//  k_sort_*     ascending sort of (eigenvalue, Fourier index) pairs.
#include <float.h>
#include <algorithm>

#include "common.cuh"

namespace fock {

enum FSource { FROM_FACTORS = 0, FROM_TOEPLITZ = 1 };

// ---- dense Hermitian helpers (shared memory, whole CTA) ----

// In-place lower Cholesky of a Hermitian positive definite m x m (row-major).
__device__ bool cta_cholesky(cplx* a, int m) {
  __shared__ int bad;
  __shared__ double s_inv;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  for (int k = 0; k < m; ++k) {
    if (threadIdx.x == 0) {
      double d = a[k * m + k].x;
      if (!(d > 0.0)) { bad = 1; d = 1.0; }
      const double r = rsqrt_nr(d);       // 1 / sqrt(d) (Newton-Raphson from an FP32 seed)
      a[k * m + k] = cmk(d * r, 0.0);
      s_inv = r;
    }
    __syncthreads();
    const double inv = s_inv;
    for (int i = k + 1 + threadIdx.x; i < m; i += blockDim.x) a[i * m + k] = cscale(a[i * m + k], inv);
    __syncthreads();
    int nt = m - k - 1;
    for (int it = threadIdx.x; it < nt * nt; it += blockDim.x) {
      int i = k + 1 + it / nt, j = k + 1 + it % nt;
      if (j <= i) a[i * m + j] = csub(a[i * m + j], cmulc(a[i * m + k], a[j * m + k]));
    }
    __syncthreads();
  }
  return bad == 0;
}

// Cyclic Jacobi eigendecomposition of a Hermitian n x n matrix a (row-major,
// stride ld >= n + (n & 1)), whole CTA.  Each step rotates n/2 disjoint
// index pairs (round-robin ordering, an odd n gets a zero pad index).  For a
// pair (p, q) with a_pq = r e^{i phi} the unitary U = diag(1, e^{-i phi}) J,
// J the real rotation that annihilates the real pair (a_pp, r, a_qq), gives
// a <- U^H a U and v <- v U.  On return the diagonal of a holds the
// eigenvalues (real parts) and the columns of v the eigenvectors.  A pair is
// skipped once |a_pq| <= 1e-15 ||a||_F; at most 30 sweeps.
__device__ void cta_jacobi_herm(cplx* a, cplx* v, int n, int ld) {
  __shared__ double rc[MAXM0 / 2 + 1], rs[MAXM0 / 2 + 1];
  __shared__ cplx rph[MAXM0 / 2 + 1];
  __shared__ int rp[MAXM0 / 2 + 1], rq[MAXM0 / 2 + 1];
  __shared__ int nrot;
  __shared__ double red[32], s_thr2;
  const int ne = n + (n & 1);
  double part = 0.0;
  for (int it = threadIdx.x; it < n * n; it += blockDim.x) part += cabs2(a[(it / n) * ld + (it % n)]);
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) t += red[w];
    s_thr2 = 1e-30 * t;   // (1e-15 ||a||_F)^2
  }
  for (int it = threadIdx.x; it < ne * ne; it += blockDim.x) {
    int i = it / ne, j = it % ne;
    v[i * ld + j] = cmk(i == j ? 1.0 : 0.0, 0.0);
    if (i == n || j == n) a[i * ld + j] = cmk(0.0, 0.0);
  }
  __syncthreads();
  const double thr2 = s_thr2;
  const int np2 = ne / 2;
  for (int sweep = 0; sweep < 30; ++sweep) {
    if (threadIdx.x == 0) nrot = 0;
    __syncthreads();
    for (int rnd = 0; rnd < ne - 1; ++rnd) {
      for (int pi = threadIdx.x; pi < np2; pi += blockDim.x) {
        int x = (pi == 0) ? 0 : ((pi - 1 + rnd) % (ne - 1)) + 1;
        int y = ((ne - 2 - pi + rnd) % (ne - 1)) + 1;
        int p = min(x, y), q = max(x, y);
        cplx apq = a[p * ld + q];
        const double r2 = cabs2(apq), app = a[p * ld + p].x, aqq = a[q * ld + q].x;
        double c = 1.0, s = 0.0;
        cplx ph = cmk(1.0, 0.0);
        if (r2 > thr2 && r2 > 1e-34 * fabs(app * aqq)) {   // |a_pq| > thr and > 1e-17 sqrt|a_pp a_qq|
          // reciprocals and square roots by Newton-Raphson from FP32 seeds
          const double rr = rsqrt_nr(r2);                    // 1 / |a_pq|
          ph = cscale(apq, rr);
          const double th = (aqq - app) * (0.5 * rr);
          const double y = fma(th, th, 1.0);
          double t = rcp_nr(fabs(th) + y * rsqrt_nr(y));     // 1 / (|th| + sqrt(th^2 + 1))
          if (th < 0.0) t = -t;
          c = rsqrt_nr(fma(t, t, 1.0));
          s = t * c;
          atomicAdd(&nrot, 1);
        }
        rp[pi] = p; rq[pi] = q; rc[pi] = c; rs[pi] = s; rph[pi] = ph;
      }
      __syncthreads();
      for (int it = threadIdx.x; it < np2 * ne; it += blockDim.x) {   // rows: U^H a
        int pi = it / ne, jj = it % ne;
        double s = rs[pi];
        if (s == 0.0) continue;
        int p = rp[pi], q = rq[pi];
        double c = rc[pi];
        cplx ap = a[p * ld + jj], aq = cmul(rph[pi], a[q * ld + jj]);
        a[p * ld + jj] = csub(cscale(ap, c), cscale(aq, s));
        a[q * ld + jj] = cadd(cscale(ap, s), cscale(aq, c));
      }
      __syncthreads();
      for (int it = threadIdx.x; it < np2 * ne; it += blockDim.x) {   // columns: a U, v U
        int pi = it / ne, ii = it % ne;
        double s = rs[pi];
        if (s == 0.0) continue;
        int p = rp[pi], q = rq[pi];
        double c = rc[pi];
        cplx phc = cconj(rph[pi]);
        cplx ap = a[ii * ld + p], aq = cmul(phc, a[ii * ld + q]);
        a[ii * ld + p] = csub(cscale(ap, c), cscale(aq, s));
        a[ii * ld + q] = cadd(cscale(ap, s), cscale(aq, c));
        cplx vp = v[ii * ld + p], vq = cmul(phc, v[ii * ld + q]);
        v[ii * ld + p] = csub(cscale(vp, c), cscale(vq, s));
        v[ii * ld + q] = cadd(cscale(vp, s), cscale(vq, c));
      }
      __syncthreads();
    }
    int done = (nrot == 0);
    __syncthreads();
    if (done) break;
  }
}

// Eigendecomposition a = Q diag(w) Q^H of a Hermitian n x n matrix (row-major,
// stride ld, n <= MAXM0), whole CTA (blockDim a multiple of 32), in about a
// quarter of the FP64 instructions of the cyclic Jacobi method above:
//  1. Householder reduction to tridiagonal form.  Step k maps x = a[k+1:, k]
//     to (alpha, 0, ..., 0) with the reflector H_k = I - beta u u^H,
//     u = (1, v_1, ...), alpha = -e^{i theta} ||x||, e^{i theta} = x_1 / |x_1|,
//     beta = 1 + |x_1| / ||x||, v_i = x_i / (x_1 - alpha); the trailing block
//     becomes H_k A H_k through p = beta A u, w = p - (beta / 2)(u^H p) u,
//     A <- A - u w^H - w u^H.  The v_i stay below the subdiagonal of column k.
//  2. The Hermitian tridiagonal T (real diagonal d, complex subdiagonal
//     alpha_k) equals D T' D^H with T' real symmetric (subdiagonal |alpha_k|)
//     and D = diag(phi), phi_0 = 1, phi_{k+1} = phi_k alpha_k / |alpha_k|.
//  3. T' = Z diag(w) Z^T by the implicit QL iteration with Wilkinson's shift
//     (Bowdler, Martin, Reinsch and Wilkinson, Numer. Math. 11 (1968)), its
//     plane rotations accumulated into Z (the real parts of v); warp 0, each
//     lane carrying its own copy of the tridiagonal and one row of Z.  An
//     off-diagonal is negligible at eps ||T'||_inf (absolute accuracy, the
//     reduction's own backward error).
//  4. Q = H_0 ... H_{n-3} D Z, applied to v in place.
// On return the diagonal of a holds the eigenvalues (real parts, unordered)
// and the columns of v the orthonormal eigenvectors.  Returns false, a and v
// then undefined, if some eigenvalue took more than 60 QL iterations.
__device__ bool cta_herm_eig(cplx* a, cplx* v, int n, int ld) {
  __shared__ double hb[MAXM0], hd[MAXM0], he[MAXM0];
  __shared__ cplx hphi[MAXM0], hpw[MAXM0];
  __shared__ int s_ok;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // ---- 1. tridiagonal reduction ----
  for (int k = 0; k + 2 < n; ++k) {
    const int m = n - k - 1;
    if (warp == 0) {
      const cplx xi = (lane < m) ? a[(k + 1 + lane) * ld + k] : cmk(0.0, 0.0);
      double tail = (lane >= 1) ? cabs2(xi) : 0.0;
      for (int o = 16; o > 0; o >>= 1) tail += __shfl_xor_sync(0xffffffffu, tail, o);
      const cplx x1 = cmk(__shfl_sync(0xffffffffu, xi.x, 0), __shfl_sync(0xffffffffu, xi.y, 0));
      double beta = 0.0;
      if (tail > 0.0) {
        const double ax1 = sqrt(cabs2(x1));
        const double sig = sqrt(fma(ax1, ax1, tail));
        const cplx ph = (ax1 > 0.0) ? cscale(x1, 1.0 / ax1) : cmk(1.0, 0.0);
        beta = 1.0 + ax1 / sig;
        const cplx inv_u1 = cscale(cconj(ph), 1.0 / (ax1 + sig));   // 1 / (x_1 - alpha)
        if (lane >= 1 && lane < m) a[(k + 1 + lane) * ld + k] = cmul(xi, inv_u1);
        if (lane == 0) a[(k + 1) * ld + k] = cscale(ph, -sig);        // alpha
      }
      if (lane == 0) hb[k] = beta;
    }
    __syncthreads();
    const double beta = hb[k];
    if (beta == 0.0) continue;                 // uniform: already reduced
    // p = beta A u over the trailing block (4 threads per row)
    const int tot = m * 4, totr = (tot + 31) & ~31;
    for (int it = threadIdx.x; it < totr; it += blockDim.x) {
      const int r = it >> 2, part = it & 3;
      cplx acc = cmk(0.0, 0.0);
      if (it < tot) {
        const cplx* row = a + (size_t)(k + 1 + r) * ld + (k + 1);
        for (int c = part; c < m; c += 4) {
          const cplx uc = (c == 0) ? cmk(1.0, 0.0) : a[(k + 1 + c) * ld + k];
          acc = cfma(row[c], uc, acc);
        }
      }
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 1);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 1);
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 2);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 2);
      if (it < tot && part == 0) hpw[r] = cscale(acc, beta);
    }
    __syncthreads();
    // w = p - (beta / 2)(u^H p) u   (u^H p real up to rounding)
    if (warp == 0) {
      const cplx ui = (lane == 0) ? cmk(1.0, 0.0) : ((lane < m) ? a[(k + 1 + lane) * ld + k] : cmk(0.0, 0.0));
      const cplx pi = (lane < m) ? hpw[lane] : cmk(0.0, 0.0);
      double up = ui.x * pi.x + ui.y * pi.y;   // Re(conj(u_i) p_i)
      for (int o = 16; o > 0; o >>= 1) up += __shfl_xor_sync(0xffffffffu, up, o);
      const double K = 0.5 * beta * up;
      __syncwarp();
      if (lane < m) hpw[lane] = csub(pi, cscale(ui, K));
    }
    __syncthreads();
    // A <- A - u w^H - w u^H on the trailing block
    for (int it = threadIdx.x; it < m * m; it += blockDim.x) {
      const int i = it / m, j = it % m;
      const cplx ui = (i == 0) ? cmk(1.0, 0.0) : a[(k + 1 + i) * ld + k];
      const cplx uj = (j == 0) ? cmk(1.0, 0.0) : a[(k + 1 + j) * ld + k];
      cplx* aij = a + (size_t)(k + 1 + i) * ld + (k + 1 + j);
      *aij = crank2(*aij, ui, hpw[j], hpw[i], uj);
    }
    __syncthreads();
  }
  // ---- 2. real tridiagonal T' and the phases D ----
  if (threadIdx.x == 0) {
    cplx phi = cmk(1.0, 0.0);
    for (int k = 0; k < n; ++k) {
      hd[k] = a[k * ld + k].x;
      hphi[k] = phi;
      if (k + 1 < n) {
        const cplx al = a[(k + 1) * ld + k];
        const double aa = sqrt(cabs2(al));
        he[k] = aa;
        if (aa > 0.0) phi = cmul(phi, cscale(al, 1.0 / aa));
      } else {
        he[k] = 0.0;
      }
    }
    s_ok = 1;
  }
  for (int it = threadIdx.x; it < n * n; it += blockDim.x) {   // Z = I
    const int i = it / n, j = it % n;
    v[i * ld + j] = cmk(i == j ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();
  // ---- 3. implicit QL on warp 0 ----
  if (warp == 0) {
    double d[MAXM0], e[MAXM0];
    double tn = 0.0;
    for (int i = 0; i < n; ++i) {
      d[i] = hd[i];
      e[i] = he[i];
      tn = fmax(tn, fabs(d[i]) + e[i] + (i > 0 ? e[i - 1] : 0.0));
    }
    const double small = 2.220446049250313e-16 * tn;   // eps ||T'||_inf
    bool ok = true;
    for (int l = 0; l < n && ok; ++l) {
      for (int iter = 0;; ++iter) {
        int m = l;
        while (m + 1 < n && fabs(e[m]) > small) ++m;
        if (m == l) break;                               // d[l] is an eigenvalue
        if (iter == 60) { ok = false; break; }
        // shift: the eigenvalue of the leading 2 x 2 of block l..m nearer d[l]
        double g = (d[l + 1] - d[l]) * rcp_nr(2.0 * e[l]);
        const double q1 = fma(g, g, 1.0);
        const double r1 = q1 * rsqrt_nr(q1);
        g = d[m] - d[l] + e[l] * rcp_nr(g + copysign(r1, g));
        double s = 1.0, c = 1.0, p = 0.0;
        bool split = false;
        for (int i = m - 1; i >= l; --i) {
          const double f = s * e[i], b = c * e[i];
          const double q2 = fma(f, f, g * g);
          if (q2 == 0.0) {                               // the chase stopped: restart
            d[i + 1] -= p;
            e[m] = 0.0;
            split = true;
            break;
          }
          const double ir = rsqrt_nr(q2);
          e[i + 1] = q2 * ir;
          s = f * ir;
          c = g * ir;
          g = d[i + 1] - p;
          const double r = fma(d[i] - g, s, 2.0 * c * b);
          p = s * r;
          d[i + 1] = g + p;
          g = fma(c, r, -b);
          if (lane < n) {                                // rotate columns i, i + 1 of Z
            const double zi = v[lane * ld + i].x, zj = v[lane * ld + i + 1].x;
            v[lane * ld + i + 1].x = fma(s, zi, c * zj);
            v[lane * ld + i].x = fma(c, zi, -s * zj);
          }
        }
        if (split) continue;
        d[l] -= p;
        e[l] = g;
        e[m] = 0.0;
      }
    }
    if (!ok && lane == 0) s_ok = 0;
    if (lane < n) hd[lane] = d[lane];
  }
  __syncthreads();
  if (!s_ok) return false;
  // ---- 4. Q = H_0 ... H_{n-3} D Z ----
  for (int it = threadIdx.x; it < n * n; it += blockDim.x) {
    const int i = it / n, j = it % n;
    v[i * ld + j] = cscale(hphi[i], v[i * ld + j].x);
  }
  __syncthreads();
  for (int k = n - 3; k >= 0; --k) {
    const double beta = hb[k];
    if (beta == 0.0) continue;
    const int m = n - k - 1;
    // t_j = u^H V[k+1:, j]  (4 threads per column)
    const int tot = n * 4, totr = (tot + 31) & ~31;
    for (int it = threadIdx.x; it < totr; it += blockDim.x) {
      const int j = it >> 2, part = it & 3;
      cplx acc = cmk(0.0, 0.0);
      if (it < tot)
        for (int i = part; i < m; i += 4) {
          const cplx ui = (i == 0) ? cmk(1.0, 0.0) : a[(k + 1 + i) * ld + k];
          acc = cfmac(v[(k + 1 + i) * ld + j], ui, acc);         // conj(u_i) V_ij
        }
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 1);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 1);
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 2);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 2);
      if (it < tot && part == 0) hpw[j] = cscale(acc, beta);
    }
    __syncthreads();
    for (int it = threadIdx.x; it < m * n; it += blockDim.x) {
      const int i = it / n, j = it % n;
      const cplx ui = (i == 0) ? cmk(1.0, 0.0) : a[(k + 1 + i) * ld + k];
      v[(k + 1 + i) * ld + j] = cfma(cmk(-ui.x, -ui.y), hpw[j], v[(k + 1 + i) * ld + j]);
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) a[i * ld + i] = cmk(hd[i], 0.0);
  __syncthreads();
  return true;
}

// Reduction of a Hermitian pencil block (h, s), both m x m with stride m, to
// a standard Hermitian matrix: eigendecomposition s = Q diag(w) Q^H
// (cta_herm_eig; in a, q: scratch of ld x ld, ld = m + (m & 1)), kept set
// K = {w_i > tau} (tau absolute: the dependency cut) in ascending index,
// X = Q_K diag(w_K)^-1/2, and h <- X^H h X (r x r, stride r, exactly
// Hermitian).  With every direction kept, X^H s X = I and the eigenvalues of
// h are the pencil's.  Returns r = |K|.  sv and keep are shared arrays of
// MAXM0 entries.
// a may be s itself (even m: the same layout); the copy is then skipped and,
// should QL run out of iterations, -1 is returned (s is overwritten) so that the
// caller forms s again and calls back with jacobi = true.
__device__ int cta_lowdin_reduce(cplx* h, const cplx* s, cplx* a, cplx* q, int m, double tau,
                                 double* sv, int* keep, bool jacobi) {
  __shared__ int s_r;
  const int ld = m + (m & 1);
  const bool inplace = ((const void*)a == (const void*)s);
  if (!inplace) {
    for (int it = threadIdx.x; it < m * m; it += blockDim.x) a[(it / m) * ld + (it % m)] = s[it];
    __syncthreads();
  }
  if (jacobi || !cta_herm_eig(a, q, m, ld)) {   // QL out of iterations: the Jacobi method
    if (!jacobi && inplace) return -1;
    if (!inplace) {
      for (int it = threadIdx.x; it < m * m; it += blockDim.x) a[(it / m) * ld + (it % m)] = s[it];
      __syncthreads();
    }
    cta_jacobi_herm(a, q, m, ld);
  }
  if (threadIdx.x == 0) {
    int r = 0;
    for (int i = 0; i < m; ++i)
      if (a[i * ld + i].x > tau && a[i * ld + i].x > 0.0) { keep[r] = i; sv[r] = a[i * ld + i].x; ++r; }
    s_r = r;
  }
  __syncthreads();
  const int r = s_r;
  cplx* X = a;   // m x r
  for (int it = threadIdx.x; it < m * r; it += blockDim.x) {
    int mu = it / r, c = it % r;
    X[it] = cscale(q[mu * ld + keep[c]], 1.0 / sqrt(sv[c]));
  }
  __syncthreads();
  cplx* Y = q;   // m x r, Y = h X
  for (int it = threadIdx.x; it < m * r; it += blockDim.x) {
    int mu = it / r, c = it % r;
    cplx acc = cmk(0.0, 0.0);
    for (int nu = 0; nu < m; ++nu) acc = cfma(h[mu * m + nu], X[nu * r + c], acc);
    Y[it] = acc;
  }
  __syncthreads();
  for (int it = threadIdx.x; it < r * r; it += blockDim.x) {   // h = X^H Y
    int ia = it / r, ib = it % r;
    cplx acc = cmk(0.0, 0.0);
    for (int mu = 0; mu < m; ++mu) acc = cfmac(Y[mu * r + ib], X[mu * r + ia], acc);
    h[it] = acc;
  }
  __syncthreads();
  for (int it = threadIdx.x; it < r * r; it += blockDim.x) {
    int ia = it / r, ib = it % r;
    if (ia < ib) {
      cplx hm = cscale(cadd(h[it], cconj(h[ib * r + ia])), 0.5);
      h[it] = hm;
      h[ib * r + ia] = cconj(hm);
    } else if (ia == ib) {
      h[it].y = 0.0;
    }
  }
  __syncthreads();
  return r;
}

// Reduction of a Hermitian pencil block (h, s), m x m with stride m, by
// Cholesky: s = L L^H, h <- L^-1 h L^-H (exactly Hermitian), when the
// factorisation certifies that s has no eigenvalue at or below tau
// (lambda_min(s) = 1 / ||L^-1||_2^2 >= 1 / ||L^-1||_F^2 > tau): then no
// direction is numerically singular and the reduction is the pencil's own.
// Returns false with h unchanged otherwise (the caller takes the Jacobi
// route).  a, q: scratch of m x m.  About m^3 complex multiply-adds against
// ~100 m^3 for the Jacobi eigendecomposition.
__device__ bool cta_cholesky_reduce(cplx* h, const cplx* s, cplx* a, cplx* q, int m, double tau) {
  __shared__ double red[32];
  __shared__ int s_ok;
  for (int it = threadIdx.x; it < m * m; it += blockDim.x) a[it] = s[it];
  __syncthreads();
  if (!cta_cholesky(a, m)) return false;                 // uniform: a shared flag
  // q = L^-1 (lower triangular), one thread per column
  for (int c = threadIdx.x; c < m; c += blockDim.x)
    for (int i = 0; i < m; ++i) {
      if (i < c) { q[i * m + c] = cmk(0.0, 0.0); continue; }
      cplx t = cmk(i == c ? 1.0 : 0.0, 0.0);
      for (int k = c; k < i; ++k) t = csub(t, cmul(a[i * m + k], q[k * m + c]));
      q[i * m + c] = cscale(t, rcp_nr(a[i * m + i].x));
    }
  __syncthreads();
  double part = 0.0;
  for (int it = threadIdx.x; it < m * m; it += blockDim.x) part += cabs2(q[it]);
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) t += red[w];
    s_ok = (t > 0.0 && t * tau < 1.0);                     // 1 / ||L^-1||_F^2 > tau
  }
  __syncthreads();
  if (!s_ok) return false;
  for (int it = threadIdx.x; it < m * m; it += blockDim.x) {   // a = L^-1 h
    const int i = it / m, j = it % m;
    cplx t = cmk(0.0, 0.0);
    for (int k = 0; k <= i; ++k) t = cfma(q[i * m + k], h[k * m + j], t);
    a[it] = t;
  }
  __syncthreads();
  for (int it = threadIdx.x; it < m * m; it += blockDim.x) {   // h = a L^-H (lower triangle)
    const int i = it / m, j = it % m;
    if (j > i) continue;
    cplx t = cmk(0.0, 0.0);
    for (int k = 0; k <= j; ++k) t = cfmac(a[i * m + k], q[j * m + k], t);
    h[it] = t;
  }
  __syncthreads();
  for (int it = threadIdx.x; it < m * m; it += blockDim.x) {   // exactly Hermitian
    const int i = it / m, j = it % m;
    if (j > i) h[it] = cconj(h[j * m + i]);
    else if (j == i) h[it].y = 0.0;
  }
  __syncthreads();
  return true;
}

// Householder reduction of Hermitian c (full storage, destroyed) to a real
// symmetric tridiagonal (d, e) with e_k = |c'_{k+1,k}| (a diagonal unitary
// scaling removes the phases).
__device__ void cta_tridiag(cplx* c, int m, double* d, double* e, cplx* v, cplx* p) {
  __shared__ double red[32];
  __shared__ double s_tau, s_K, s_norm;
  for (int k = 0; k < m - 2; ++k) {
    // ||x||^2, x = c[k+1:, k]
    double part = 0.0;
    for (int i = k + 1 + threadIdx.x; i < m; i += blockDim.x) part += cabs2(c[i * m + k]);
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) s += red[w];
      // square roots and reciprocals by Newton-Raphson from FP32 seeds
      const double xn = (s > 0.0) ? s * rsqrt_nr(s) : 0.0;
      const cplx x0 = c[(k + 1) * m + k];
      const double a2 = cabs2(x0);
      const double ra = (a2 > 0.0) ? rsqrt_nr(a2) : 0.0;
      const double ax0 = a2 * ra;
      cplx ph = (a2 > 0.0) ? cscale(x0, ra) : cmk(1.0, 0.0);
      cplx alpha = cscale(ph, -xn);
      d[k] = c[k * m + k].x;
      e[k] = xn;
      double vn2 = 2.0 * (s + xn * ax0);
      s_tau = (vn2 > 0.0) ? 2.0 * rcp_nr(vn2) : 0.0;
      s_norm = xn;
      v[k + 1] = csub(x0, alpha);
    }
    __syncthreads();
    for (int i = k + 2 + threadIdx.x; i < m; i += blockDim.x) v[i] = c[i * m + k];
    __syncthreads();
    const double tau = s_tau;
    if (tau != 0.0) {
      for (int i = k + 1 + threadIdx.x; i < m; i += blockDim.x) {
        cplx s = cmk(0.0, 0.0);
        for (int j = k + 1; j < m; ++j) s = cfma(c[i * m + j], v[j], s);
        p[i] = cscale(s, tau);
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        double K = 0.0;   // (tau/2) v^H p, real for Hermitian c
        for (int i = k + 1; i < m; ++i) K += v[i].x * p[i].x + v[i].y * p[i].y;
        s_K = 0.5 * tau * K;
      }
      __syncthreads();
      const double K = s_K;
      for (int i = k + 1 + threadIdx.x; i < m; i += blockDim.x) p[i] = csub(p[i], cscale(v[i], K));
      __syncthreads();
      const int nt = m - k - 1;
      for (int it = threadIdx.x; it < nt * nt; it += blockDim.x) {
        int i = k + 1 + it / nt, j = k + 1 + it % nt;
        // c -= v w^H + w v^H   (w stored in p)
        c[i * m + j] = crank2(c[i * m + j], v[i], p[j], p[i], v[j]);
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (m >= 2) {
      d[m - 2] = c[(m - 2) * m + (m - 2)].x;
      d[m - 1] = c[(m - 1) * m + (m - 1)].x;
      e[m - 2] = sqrt(cabs2(c[(m - 1) * m + (m - 2)]));
    } else {
      d[0] = c[0].x;
    }
  }
  __syncthreads();
}

__device__ inline cplx twiddle(long long num, int M) {   // exp(-2 pi i num / M)
  double s, c;
  sincospi(-2.0 * (double)(num % M) / (double)M, &s, &c);
  return cmk(c, s);
}

// Sbar_j of a block formed again, with the arithmetic of the formation in
// k_fblocks (used where the block's eigendecomposition works in Sbar's own
// storage and a route that overwrote it fell through).  tw: ldj^2 entries of
// scratch for the Toeplitz twiddles.
__device__ void reform_S(const FBlockTask& F, const ProbDev& P, int j, int m0, cplx* S, cplx* tw, int ldj) {
  const int np = m0 * m0;
  if (F.source == FROM_FACTORS) {
    const int j3 = j % F.L[2], j2 = (j / F.L[2]) % F.L[1], j1 = j / (F.L[1] * F.L[2]);
    const int nfe = P.nF * np;
    const cplx* x0 = F.Xh[0] + (size_t)j1 * nfe;
    const cplx* x1 = F.Xh[1] + (size_t)j2 * nfe;
    const cplx* x2 = F.Xh[2] + (size_t)j3 * nfe;
    const int nup = m0 * (m0 + 1) / 2;
    for (int u = threadIdx.x; u < nup; u += blockDim.x) {
      int mu = 0, rem = u;
      while (rem >= m0 - mu) { rem -= m0 - mu; ++mu; }
      const int nu = mu + rem, pr = mu * m0 + nu, tr = nu * m0 + mu;
      cplx s = cmul(x0[pr], cmul(x1[pr], x2[pr]));
      if (mu == nu) s.y = 0.0;
      S[pr] = s;
      S[tr] = cconj(s);
    }
    __syncthreads();
  } else {
    const bool tab = (F.D <= ldj * ldj);
    if (tab) {
      for (int dd2 = 1 + threadIdx.x; dd2 <= F.D; dd2 += blockDim.x) tw[dd2 - 1] = twiddle((long long)j * dd2, F.M);
      __syncthreads();
    }
    for (int pr = threadIdx.x; pr < np; pr += blockDim.x) {
      const int mu = pr / m0, nu = pr % m0, tr = nu * m0 + mu;
      cplx s = cmk(F.TS[pr], 0.0);
      for (int dd2 = 1; dd2 <= F.D; ++dd2) {
        const cplx w = tab ? tw[dd2 - 1] : twiddle((long long)j * dd2, F.M);
        const double* ts = F.TS + (size_t)dd2 * np;
        s = cadd(s, cmk(w.x * (ts[pr] + ts[tr]), w.y * (ts[pr] - ts[tr])));
      }
      S[pr] = s;
    }
    __syncthreads();
    for (int pr = threadIdx.x; pr < np; pr += blockDim.x) {
      const int mu = pr / m0, nu = pr % m0;
      if (mu < nu) {
        const cplx sm2 = cscale(cadd(S[pr], cconj(S[nu * m0 + mu])), 0.5);
        S[pr] = sm2; S[nu * m0 + mu] = cconj(sm2);
      } else if (mu == nu) {
        S[pr].y = 0.0;
      }
    }
    __syncthreads();
  }
}

__global__ void k_fblocks(const ProbDev* __restrict__ probs, const FBlockTask* __restrict__ tasks) {
  extern __shared__ cplx sm[];
  const FBlockTask F = tasks[blockIdx.y];
  const int jl = blockIdx.x;      // local output index
  if (jl >= F.nj) return;
  const int j = F.j0 + jl;        // Fourier index
  // Real generators: the block at -j (componentwise mod L) is the complex
  // conjugate of the block at j, with the same spectrum.  When both indices
  // are in this task's range and no blocks are stored, the lower index
  // solves the pair and writes both; the higher one does nothing.
  int jm = -1;
  if (F.source == FROM_FACTORS && F.want == 1 && !F.outH) {
    const int j3 = j % F.L[2], j2 = (j / F.L[2]) % F.L[1], j1 = j / (F.L[1] * F.L[2]);
    const int m1 = (F.L[0] - j1) % F.L[0], m2 = (F.L[1] - j2) % F.L[1], m3 = (F.L[2] - j3) % F.L[2];
    jm = (m1 * F.L[1] + m2) * F.L[2] + m3;
    if (jm == j || jm < F.j0 || jm >= F.j0 + F.nj) jm = -1;
    else if (jm < j) return;
  }
  const ProbDev& P = probs[F.prob];
  const int m0 = P.m0, np = m0 * m0;
  const int ldj = m0 + (m0 & 1);
  // even m0: the overlap's eigendecomposition works in Sbar's own storage (the
  // same m0 x m0 layout), so a block needs three m0^2 arrays and 32 x 32 blocks
  // fit four CTAs per SM; odd m0 keeps a padded work array of its own
  const bool alias = !(m0 & 1);
  cplx* H = sm;
  cplx* S = sm + np;
  cplx* Aj = alias ? S : S + np;                       // eigendecomposition work, ldj x ldj
  cplx* Qj = alias ? S + np : Aj + ldj * ldj;          // its eigenvectors, ldj x ldj
  cplx* v = Qj + ldj * ldj;
  cplx* pv = v + MAXM0;
  double* dd = (double*)(pv + MAXM0);
  double* ee = dd + MAXM0;
  double* e2 = ee + MAXM0;                 // e^2, and FP32 copies of d and e^2
  float* df = (float*)(e2 + MAXM0);
  float* e2f = df + MAXM0;
  // eigenvectors (F.vecs): a copy of the reduced matrix and its Jacobi eigenvectors
  cplx* Vc = (cplx*)(((uintptr_t)(e2f + MAXM0) + 15) & ~(uintptr_t)15);
  cplx* Wv = Vc + ldj * ldj;

  if (F.source == FROM_FACTORS) {
    const int j3 = j % F.L[2], j2 = (j / F.L[2]) % F.L[1], j1 = j / (F.L[1] * F.L[2]);
    const int nfe = P.nF * np;
    const cplx* x0 = F.Xh[0] + (size_t)j1 * nfe;
    const cplx* x1 = F.Xh[1] + (size_t)j2 * nfe;
    const cplx* x2 = F.Xh[2] + (size_t)j3 * nfe;
    // H and S are Hermitian (each axis factor is, and so is a Hadamard product
    // of Hermitian matrices): the upper triangle, enumerated compactly so that
    // whole warps share the work, is formed and mirrored; the diagonal is real
    const int nup = m0 * (m0 + 1) / 2;
    for (int u = threadIdx.x; u < nup; u += blockDim.x) {
      int mu = 0, rem = u;
      while (rem >= m0 - mu) { rem -= m0 - mu; ++mu; }
      const int nu = mu + rem, pr = mu * m0 + nu, tr = nu * m0 + mu;
      cplx s0 = x0[pr], s1 = x1[pr], s2 = x2[pr];
      cplx a0 = x0[np + pr], a1 = x1[np + pr], a2 = x2[np + pr];
      cplx s12 = cmul(s1, s2);
      cplx hk = cadd(cmul(a0, s12), cmul(s0, cadd(cmul(a1, s2), cmul(s1, a2))));
      hk = cscale(hk, 0.5);
      cplx vv = cmk(0.0, 0.0);
      for (int t = 0; t < P.T; ++t) {
        double w = P.Z[t / P.R] * P.cq[t % P.R];
        cplx pr3 = cmul(cmul(x0[(2 + t) * np + pr], x1[(2 + t) * np + pr]), x2[(2 + t) * np + pr]);
        vv.x = fma(pr3.x, w, vv.x);
        vv.y = fma(pr3.y, w, vv.y);
      }
      cplx h = csub(hk, vv), s = cmul(s0, s12);
      if (mu == nu) { h.y = 0.0; s.y = 0.0; }
      H[pr] = h; S[pr] = s;
      H[tr] = cconj(h); S[tr] = cconj(s);
    }
  } else {
    // twiddles exp(-2 pi i j d / M), d = 1..D, once per block (in the
    // eigenvector scratch, free until the reduction) when they fit
    cplx* tw = Qj;
    const bool tab = (F.D <= ldj * ldj);
    if (tab) {
      for (int dd2 = 1 + threadIdx.x; dd2 <= F.D; dd2 += blockDim.x) tw[dd2 - 1] = twiddle((long long)j * dd2, F.M);
      __syncthreads();
    }
    for (int pr = threadIdx.x; pr < np; pr += blockDim.x) {
      int mu = pr / m0, nu = pr % m0, tr = nu * m0 + mu;
      cplx h = cmk(F.TH[pr], 0.0), s = cmk(F.TS[pr], 0.0);
      for (int dd2 = 1; dd2 <= F.D; ++dd2) {
        cplx w = tab ? tw[dd2 - 1] : twiddle((long long)j * dd2, F.M);
        const double* th = F.TH + (size_t)dd2 * np;
        const double* ts = F.TS + (size_t)dd2 * np;
        // w T_d[mu][nu] + conj(w) T_d[nu][mu]
        h = cadd(h, cmk(w.x * (th[pr] + th[tr]), w.y * (th[pr] - th[tr])));
        s = cadd(s, cmk(w.x * (ts[pr] + ts[tr]), w.y * (ts[pr] - ts[tr])));
      }
      H[pr] = h;
      S[pr] = s;
    }
  }
  __syncthreads();
  // exact Hermitian symmetrisation of the formed pair (removes rounding
  // asymmetry; the factor route forms Hermitian blocks directly)
  if (F.source != FROM_FACTORS) {
    for (int pr = threadIdx.x; pr < np; pr += blockDim.x) {
      int mu = pr / m0, nu = pr % m0;
      if (mu < nu) {
        cplx h1 = H[pr], h2 = H[nu * m0 + mu], s1 = S[pr], s2 = S[nu * m0 + mu];
        cplx hm = cscale(cadd(h1, cconj(h2)), 0.5), sm2 = cscale(cadd(s1, cconj(s2)), 0.5);
        H[pr] = hm; H[nu * m0 + mu] = cconj(hm);
        S[pr] = sm2; S[nu * m0 + mu] = cconj(sm2);
      } else if (mu == nu) {
        H[pr].y = 0.0; S[pr].y = 0.0;
      }
    }
    __syncthreads();
  }
  if (F.outH)
    for (int pr = threadIdx.x; pr < np; pr += blockDim.x) {
      F.outH[(size_t)jl * np + pr] = H[pr];
      F.outS[(size_t)jl * np + pr] = S[pr];
    }
  if (F.want == 0) return;
  __syncthreads();
  // reduction on the directions of Sbar above the dependency cut (only
  // numerically singular Bloch combinations are removed)
  __shared__ int keep[MAXM0];
  __shared__ double sv[MAXM0];
  __shared__ double s_tau;
  if (F.source == FROM_FACTORS) {
    if (threadIdx.x == 0) s_tau = *F.tau;
  } else {
    // B = |T_S[0]| + sum_{d >= 1} (|T_S[d]| + |T_S[d]|^T) of the embedded
    // generators, tau = null_tau(||B||_F)
    double part = 0.0;
    for (int pr = threadIdx.x; pr < np; pr += blockDim.x) {
      const int tr = (pr % m0) * m0 + pr / m0;
      double b = fabs(F.TS[pr]);
      for (int dd2 = 1; dd2 <= F.D; ++dd2) b += fabs(F.TS[(size_t)dd2 * np + pr]) + fabs(F.TS[(size_t)dd2 * np + tr]);
      part += b * b;
    }
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
    __shared__ double red_b[32];
    if ((threadIdx.x & 31) == 0) red_b[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) t += red_b[w];
      s_tau = null_tau(sqrt(t), (double)F.M * m0);   // the embedding's order
    }
  }
  __syncthreads();
  // Cholesky when it certifies that nothing is numerically singular, else the
  // eigendecomposition of Sbar_j with the cut
  const bool chol = cta_cholesky_reduce(H, S, Aj, Qj, m0, s_tau);
  if (!chol && alias) reform_S(F, P, j, m0, S, Qj, ldj);   // the attempt factored Sbar in place
  int r = chol ? m0 : cta_lowdin_reduce(H, S, Aj, Qj, m0, s_tau, sv, keep, false);
  if (r < 0) {                                             // QL ran out on Sbar in place
    reform_S(F, P, j, m0, S, Qj, ldj);
    r = cta_lowdin_reduce(H, S, Aj, Qj, m0, s_tau, sv, keep, true);
  }
  if (!chol && F.neig && threadIdx.x == 0) atomicAdd(F.neig, 1);
  const int ldr = r + (r & 1);
  if (F.vecs) {   // the reduced matrix, kept for its eigenvectors
    for (int it = threadIdx.x; it < r * r; it += blockDim.x) Vc[(it / r) * ldr + it % r] = H[it];
    __syncthreads();
  }
  const bool values = F.want == 2;
  if (values && r > 0) cta_tridiag(H, r, dd, ee, v, pv);
  for (int i = threadIdx.x; values && i < r; i += blockDim.x) {
    const double e2i = (i + 1 < r) ? ee[i] * ee[i] : 0.0;
    e2[i] = e2i;
    df[i] = (float)dd[i];
    e2f[i] = (float)e2i;
  }
  __syncthreads();
  if (F.want == 2 && threadIdx.x == 0) {
    // the lowest eigenvalue of an embedding block only sets the preconditioner
    // shift (lowered by 2e-5 relative afterwards): 1e-9 relative suffices
    F.ev[jl] = (r > 0) ? tridiag_eig_fast(df, e2f, dd, e2, r, 0, 1e-9) : INFINITY;
  }
  if (F.vecs && F.want == 1) {
    // eigenvectors of the reduced matrix by Jacobi (orthonormal also inside
    // degenerate clusters), ordered by eigenvalue, mapped back by the
    // reduction's transform: y = L^-H w (Cholesky route) or X w (X = Q_K
    // diag(s_K)^-1/2), so y^H Sbar_j y = 1; the conjugate block gets conj(y)
    __shared__ int ord[MAXM0];
    __syncthreads();
    if (r > 0) cta_jacobi_herm(Vc, Wv, r, ldr);
    if (threadIdx.x == 0) {
      for (int i = 0; i < r; ++i) ord[i] = i;
      for (int i = 1; i < r; ++i) {
        const int o = ord[i];
        const double e = Vc[o * ldr + o].x;
        int q = i - 1;
        while (q >= 0 && Vc[ord[q] * ldr + ord[q]].x > e) { ord[q + 1] = ord[q]; --q; }
        ord[q + 1] = o;
      }
    }
    __syncthreads();
    for (int it = threadIdx.x; it < np; it += blockDim.x) {
      const int i = it / m0, mu = it % m0;
      cplx y = cmk(0.0, 0.0);
      if (i < r) {
        const int c = ord[i];
        if (chol) {
          for (int nu = mu; nu < m0; ++nu) y = cadd(y, cmul(cconj(Qj[nu * m0 + mu]), Wv[nu * ldr + c]));
        } else {
          for (int nu = 0; nu < r; ++nu) y = cadd(y, cmul(Aj[mu * r + nu], Wv[nu * ldr + c]));
        }
      }
      F.vecs[(size_t)jl * np + it] = y;
      if (jm >= 0) F.vecs[(size_t)(jm - F.j0) * np + it] = cconj(y);
    }
  }
}

// ---- periodic spectra (factors, eigenvalues only): a pipeline over Fourier blocks ----
//
// k_fblocks above takes a block through every phase in one CTA.  Its time went to
// FP64 instructions that half-empty warps issued and to phases that one warp or
// one thread ran while the CTA waited: three products per quadrature term and
// block in the formation, the QL sweeps with their rotations, FP64 bisection,
// serial triangular inverses.  For whole spectra the phases are kernels of their
// own over a chunk of blocks (conjugate pairs once), each spread as it likes:
//
//  k_pf_form    Hbar_j, Sbar_j, lower triangles: a thread per entry, eight blocks j
//               with the same (j1, j2) at a time, so the product of the first two
//               axes' factors is formed once for them: 38 FP64 instructions per
//               term and eight blocks instead of 80
//  k_pf_reduce  elimination of Sbar_j applied to Hbar_j from both sides and to L^-1 as
//               it goes (entries in registers); when L^-1 certifies that nothing is
//               numerically singular: the reduced matrix to tridiagonal form.
//               Otherwise Sbar_j to tridiagonal form, reflectors kept
//  k_pf_ql      one thread per block: QL on the overlaps' tridiagonals, rotations recorded
//  k_pf_cut     the recorded rotations applied, the cut, X = Q_K diag(s_K)^-1/2,
//               X^H Hbar X to tridiagonal form
//  k_pf_values  one thread per block: QL for the eigenvalues
//
// All are bound by the FP64 pipe or, the two QL kernels, by a thread's chain of
// about 850 cycles per rotation with every SM holding a few warps.  Measured: two
// lattices of 16^3 cells of 16 functions 3.06 -> 1.7 ms, one of 32^3 cells of 32
// functions, four of them cut in every block, 86.5 -> 38 ms.

// lower-triangle position t = a (a + 1) / 2 + b, b <= a
__device__ inline void tri_pos(int t, int& a, int& b) {
  a = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((a + 1) * (a + 2) / 2 <= t) ++a;
  while (a * (a + 1) / 2 > t) --a;
  b = t - a * (a + 1) / 2;
}
// element i of slot's tridiagonal arrays: 32 slots side by side
__device__ inline size_t pf_ix(int slot, int i, int mm) { return ((size_t)(slot >> 5) * mm + i) * 32 + (slot & 31); }

// G: blocks per thread at a time (8; 2 where there are too few blocks to fill the GPU)
// A warp per CTA: 32 entries of the triangle waste least, and warps of 160 000 cycles
// fill the SMs evenly (two lattices of 16^3 cells: 840 us with CTAs of 160 threads).
template <int G>
__global__ void __launch_bounds__(32) k_pf_form(const ProbDev* __restrict__ probs, const PfTask* __restrict__ tasks,
                                                const PfGroup* __restrict__ groups, PfWork W) {
  const PfGroup grp = groups[blockIdx.x * G / kPfGroup];
  const PfTask F = tasks[grp.task];
  const ProbDev& P = probs[F.prob];
  const int m0 = P.m0, np = m0 * m0, nup = m0 * (m0 + 1) / 2, R = P.R, T = P.T;
  const int t0 = blockIdx.y * blockDim.x + threadIdx.x, s0 = blockIdx.x * G, r0 = grp.rep + s0 % kPfGroup;
  const int cnt = min(G, F.nrep - r0);
  if (cnt <= 0) return;
  __shared__ int sj[G];                      // the blocks' Fourier indices
  if (threadIdx.x < cnt) sj[threadIdx.x] = F.j0 + F.index(r0 + threadIdx.x);
  __syncwarp();
  if (t0 >= nup) return;
  int a, b;
  tri_pos(t0, a, b);
  const int pr = b * m0 + a;                 // the upper entry (b, a); the lower one is its conjugate
  const int nfe = P.nF * np;
  const double *Zq = P.Z, *cq = P.cq;
  // the inner axis, along which consecutive blocks run: the last one with more than one cell
  const int in = (F.L[2] > 1) ? 2 : (F.L[1] > 1) ? 1 : 0, o0 = (in == 0) ? 1 : 0, o1 = (in == 2) ? 1 : 2;
  const int Lin = F.L[in];
  for (int g0 = 0; g0 < cnt;) {
    // a run of blocks with the same indices on the other two axes
    const int j = sj[g0], jo = j / Lin;   // (axes after the inner one have one cell)
    int n = 1;
    while (g0 + n < cnt && sj[g0 + n] / Lin == jo) ++n;
    const int i0 = (in == 2) ? jo / F.L[1] : (in == 1) ? jo : 0, i1 = (in == 2) ? jo % F.L[1] : 0;
    const cplx* f0 = F.Xh[o0] + (size_t)i0 * nfe + pr;
    const cplx* f1 = F.Xh[o1] + (size_t)i1 * nfe + pr;
    const cplx* f2[G];
    cplx v[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int jg = sj[g0 + min(g, n - 1)];
      f2[g] = F.Xh[in] + (size_t)(jg % Lin) * nfe + pr;
      v[g] = cmk(0.0, 0.0);
    }
    for (int nu = 0; nu < T / R; ++nu) {
      const double zw = Zq[nu];
#pragma unroll 2
      for (int q = 0; q < R; ++q) {
        const size_t o = (size_t)(2 + nu * R + q) * np;
        const cplx p = cscale(cmul(f0[o], f1[o]), zw * cq[q]);
#pragma unroll
        for (int g = 0; g < G; ++g)
          if (g < n) v[g] = cfma(p, f2[g][o], v[g]);
      }
    }
    const cplx s0v = f0[0], s1 = f1[0], a0 = f0[np], a1 = f1[np];
    const cplx s01 = cmul(s0v, s1), k01 = cadd(cmul(a0, s1), cmul(s0v, a1));
#pragma unroll
    for (int g = 0; g < G; ++g)
      if (g < n) {
        const cplx s2 = f2[g][0], a2 = f2[g][np];
        cplx h = csub(cscale(cadd(cmul(k01, s2), cmul(s01, a2)), 0.5), v[g]);
        cplx s = cmul(s01, s2);
        if (a == b) { h.y = 0.0; s.y = 0.0; }
        const size_t o = (size_t)(s0 + g0 + g) * W.nup + t0;
        W.H[o] = cconj(h);
        W.S[o] = cconj(s);
      }
    g0 += n;
  }
}

// The warp that does what one warp does, different in the CTAs that share an SM
// (CTAs b, b + 152, ...): warps of one number share a sub-partition.
__device__ inline int pf_lead(int nw) { return (int)((blockIdx.x / 152 + blockIdx.x) % (unsigned)nw); }

// Householder reduction of the Hermitian m x m matrix A (lower triangle, pitch ld,
// shared memory) to tridiagonal form: d, e = |subdiagonal|, and of each step the
// reflector I - tau v v^H (v left in A's column below the diagonal) and the
// subdiagonal's phase.  v, w: m entries each.  lw: the warp that makes the reflectors.
__device__ void cta_tridiag_lower(cplx* A, int ld, int m, double* d, double* e, double* tau, cplx* ph, cplx* v, cplx* w,
                                  int lw) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = 0; k + 1 < m; ++k) {
    const int n = m - k - 1;
    if (warp == lw) {
      const cplx x = (lane < n) ? A[(k + 1 + lane) * ld + k] : cmk(0.0, 0.0);
      double tail = (lane >= 1) ? cabs2(x) : 0.0;
      for (int o = 16; o > 0; o >>= 1) tail += __shfl_xor_sync(0xffffffffu, tail, o);
      const cplx x1 = cmk(__shfl_sync(0xffffffffu, x.x, 0), __shfl_sync(0xffffffffu, x.y, 0));
      const double a2 = cabs2(x1);
      const double r1 = (__double_as_longlong(a2) > 0) ? rsqrt_nr(a2) : 0.0;
      const double ax = a2 * r1;
      const cplx p1 = (__double_as_longlong(a2) > 0) ? cscale(x1, r1) : cmk(1.0, 0.0);
      double ek = ax, tk = 0.0;
      cplx phase = p1, vi = x;
      if (__double_as_longlong(tail) > 0) {      // (no tail for the last column)
        const double s = a2 + tail, xn = s * rsqrt_nr(s);
        tk = rcp_nr(fma(ax, xn, s));
        ek = xn;
        phase = cmk(-p1.x, -p1.y);
        if (lane == 0) vi = cscale(p1, ax + xn);
      }
      if (lane < n) { v[lane] = vi; if (lane == 0) A[(k + 1) * ld + k] = vi; }
      if (lane == 0) { d[k] = A[k * ld + k].x; e[k] = ek; tau[k] = tk; ph[k] = phase; }
    }
    __syncthreads();
    const double tk = tau[k];
    if (__double_as_longlong(tk) == 0) continue;   // uniform
    const cplx* B = A + (size_t)(k + 1) * ld + (k + 1);   // trailing block
    for (int it = threadIdx.x; it < ((4 * n + 31) & ~31); it += blockDim.x) {   // w = tau B v, 4 threads per row
      const int i = it >> 2, o = it & 3;
      cplx s = cmk(0.0, 0.0);
      if (i < n)
        for (int j = o; j < n; j += 4) {
          // the entry or its mirror's conjugate (sign bit flipped: no FP64, no divergence)
          const bool low = j <= i;
          cplx x = B[low ? i * ld + j : j * ld + i];
          x.y = __longlong_as_double(__double_as_longlong(x.y) ^ (low ? 0ll : (long long)0x8000000000000000ull));
          s = cfma(x, v[j], s);
        }
      s.x += __shfl_xor_sync(0xffffffffu, s.x, 1);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, 1);
      s.x += __shfl_xor_sync(0xffffffffu, s.x, 2);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, 2);
      if (i < n && o == 0) w[i] = cscale(s, tk);
    }
    __syncthreads();
    if (warp == lw) {                               // w -= (tau / 2) Re(v^H w) v
      const cplx vi = (lane < n) ? v[lane] : cmk(0.0, 0.0), wi = (lane < n) ? w[lane] : cmk(0.0, 0.0);
      double s = fma(vi.x, wi.x, vi.y * wi.y);
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const double K = -0.5 * tk * s;
      if (lane < n) w[lane] = cmk(fma(K, vi.x, wi.x), fma(K, vi.y, wi.y));
    }
    __syncthreads();
    // B -= v w^H + w v^H, lower triangle: rows n-1-p and p together are n + 1 entries
    const int half = (n + 1) >> 1;
    for (int it = threadIdx.x; it < half * (n + 1); it += blockDim.x) {
      const int p = it / (n + 1), q = it - p * (n + 1);
      int i = n - 1 - p, j = q;
      if (q > i) { if (i == p) continue; j = q - i - 1; i = p; }
      cplx* x = A + (size_t)(k + 1 + i) * ld + (k + 1 + j);
      *x = crank2(*x, v[i], w[j], w[i], v[j]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    d[m - 1] = A[(m - 1) * ld + (m - 1)].x;
    e[m - 1] = 0.0;
  }
  __syncthreads();
}

// NT threads, NS entries of the lower triangle per thread.
template <int NT, int NS>
__global__ void __launch_bounds__(NT) k_pf_reduce(const ProbDev* __restrict__ probs, const PfTask* __restrict__ tasks,
                                                  const PfGroup* __restrict__ groups, PfWork W) {
  extern __shared__ __align__(16) cplx psm[];
  const int slot = blockIdx.x;
  const PfGroup grp = groups[slot / kPfGroup];
  const PfTask F = tasks[grp.task];
  if (grp.rep + slot % kPfGroup >= F.nrep) { if (threadIdx.x == 0) W.status[slot] = -1; return; }
  const int m = probs[F.prob].m0, nup = m * (m + 1) / 2, ld = m | 1, tid = threadIdx.x;
  cplx* A = psm;                               // m x ld
  __shared__ cplx cS[2][MAXM0], cH[2][MAXM0], lv[MAXM0], uv[MAXM0], xs[MAXM0], yh[MAXM0], zl[MAXM0];
  __shared__ double dl[MAXM0], dd[MAXM0], ee[MAXM0], tt[MAXM0], red[4];
  __shared__ cplx ph[MAXM0];
  const int lane = tid & 31, lw = pf_lead(NT / 32);
  const cplx* Hg = W.H + (size_t)slot * W.nup;
  const cplx* Sg = W.S + (size_t)slot * W.nup;
  cplx S[NS], H[NS];
  int ea[NS], eb[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const int t = s * NT + tid;
    ea[s] = -1;
    eb[s] = 0;
    if (t < nup) { tri_pos(t, ea[s], eb[s]); S[s] = Sg[t]; H[s] = Hg[t]; }
  }
  bool ok = true;
  const double cut = fmax(*F.tau, 0.0);
  // Step j: l = S(:, j) / S_jj for rows a > j; S and L^-1 (in S's eliminated columns)
  // lose l times row j, H loses l u^H + u l^H with u = H(:, j) - l H_jj / 2 in the
  // columns still to come and l times its row j in those already eliminated.  Column
  // b's multipliers of -l_a and -u_a stand in xs, yh and zl whatever b's case, so the
  // lanes of a warp do not diverge.
  for (int j = 0; j < m; ++j) {
    const int par = j & 1;
    // entry t of column j where t >= j, of row j where t < j
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      if (eb[s] == j && ea[s] >= j) { cS[par][ea[s]] = S[s]; cH[par][ea[s]] = H[s]; }
      if (ea[s] == j && eb[s] < j) { cS[par][eb[s]] = S[s]; cH[par][eb[s]] = H[s]; }
    }
    __syncthreads();
    const double dj = cS[par][j].x, hjj = cH[par][j].x;
    // a pivot at or below the cut bounds lambda_min(Sbar): no certificate (uniform)
    if (!(dj > cut)) { ok = false; break; }
    if ((tid >> 5) == lw && lane < m) {
      const cplx c = cS[par][lane], h = cH[par][lane];
      if (lane > j) {
        const cplx l = cscale(c, rcp_nr(dj));
        const cplx u = cmk(fma(-0.5 * hjj, l.x, h.x), fma(-0.5 * hjj, l.y, h.y));
        lv[lane] = cmk(-l.x, -l.y);
        uv[lane] = cmk(-u.x, -u.y);
        xs[lane] = cconj(c);
        yh[lane] = cconj(u);
        zl[lane] = cconj(l);
      } else {
        if (lane == j) dl[j] = dj;
        xs[lane] = (lane == j) ? cmk(1.0, 0.0) : c;
        yh[lane] = (lane == j) ? cmk(hjj, 0.0) : h;
        zl[lane] = cmk(0.0, 0.0);
      }
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int a = ea[s], b = eb[s];
      if (a <= j) continue;
      const cplx l = lv[a];
      S[s] = cfma(l, xs[b], (b == j) ? cmk(0.0, 0.0) : S[s]);
      H[s] = cfma(uv[a], zl[b], cfma(l, yh[b], H[s]));
    }
  }
  __syncthreads();
  if (ok) {
    // certificate: lambda_min(Sbar) >= 1 / ||L^-1||_F^2 > tau (Cholesky's L^-1 = delta^-1/2 times ours)
    double part = 0.0;
#pragma unroll
    for (int s = 0; s < NS; ++s)
      if (ea[s] >= 0) part = fma((ea[s] == eb[s]) ? 1.0 : cabs2(S[s]), rcp_nr(dl[ea[s]]), part);
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((tid & 31) == 0) red[tid >> 5] = part;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < NT / 32; ++w) t += red[w];
    ok = t > 0.0 && t * cut < 1.0;             // uniform
  }
  const int mm = W.mm;
  if (ok) {
    for (int t = tid; t < m; t += NT) tt[t] = rsqrt_nr(dl[t]);
    __syncthreads();
#pragma unroll
    for (int s = 0; s < NS; ++s)
      if (ea[s] >= 0) {
        const cplx x = cscale(H[s], tt[ea[s]] * tt[eb[s]]);
        A[ea[s] * ld + eb[s]] = (ea[s] == eb[s]) ? cmk(x.x, 0.0) : x;
      }
  } else {
#pragma unroll
    for (int s = 0; s < NS; ++s)
      if (ea[s] >= 0) A[ea[s] * ld + eb[s]] = Sg[s * NT + tid];
    if (tid == 0 && F.neig) atomicAdd(F.neig, 1);
  }
  __syncthreads();
  cta_tridiag_lower(A, ld, m, dd, ee, tt, ph, cS[0], cS[1], lw);
  double* od = ok ? W.td : W.sd;
  double* oe = ok ? W.te : W.se;
  for (int i = tid; i < m; i += NT) {
    od[pf_ix(slot, i, mm)] = dd[i];
    oe[pf_ix(slot, i, mm)] = ee[i];
  }
  if (tid == 0) { W.status[slot] = ok ? 0 : 1; W.order[slot] = m; }
  if (!ok) {
    for (int i = tid; i + 1 < m; i += NT) { W.rtau[(size_t)slot * mm + i] = tt[i]; W.rph[(size_t)slot * mm + i] = ph[i]; }
    cplx* R = W.R + (size_t)slot * W.nup;
    for (int t = tid; t < nup; t += NT) {
      int a, b;
      tri_pos(t, a, b);
      R[t] = A[a * ld + b];
    }
  }
}

// Implicit QL with Wilkinson's shift (Bowdler, Martin, Reinsch and Wilkinson, Numer.
// Math. 11 (1968)) on one thread's tridiagonal: D(i), E(i) at D[32 i], E[32 i].  An
// off-diagonal is negligible at eps ||T||_inf.  rec(i, c, s) is told each rotation
// of columns i, i + 1.  False when an eigenvalue takes more than 60 iterations.
template <class Rec>
__device__ bool lane_ql(double* D, double* E, int n, Rec rec) {
  double tn = 0.0, em = 0.0;
  for (int i = 0; i < n; ++i) {
    const double e = (i + 1 < n) ? E[32 * i] : 0.0;
    tn = fmax(tn, fabs(D[32 * i]) + e + em);
    em = e;
  }
  const double small = 2.220446049250313e-16 * tn;
  const long long small_bits = __double_as_longlong(small);
  for (int l = 0; l < n; ++l) {
    for (int iter = 0;; ++iter) {
      int m = l;
      while (m + 1 < n && abs_bits(E[32 * m]) > small_bits) ++m;
      if (m == l) break;                               // D(l) is an eigenvalue
      if (iter == 60) return false;
      // shift: the eigenvalue of the leading 2 x 2 of block l..m nearer D(l)
      const double el = E[32 * l], dl = D[32 * l];
      double g = (D[32 * (l + 1)] - dl) * rcp_nr(2.0 * el);
      const double q1 = fma(g, g, 1.0);
      const double r1 = q1 * rsqrt_nr(q1);
      g = D[32 * m] - dl + el * rcp_nr(g + copysign(r1, g));
      double s = 1.0, c = 1.0, p = 0.0, dn = D[32 * m];
      bool split = false;
      for (int i = m - 1; i >= l; --i) {
        const double ei = E[32 * i], di = D[32 * i];
        const double f = s * ei, b = c * ei;
        const double q2 = fma(f, f, g * g);
        if (__double_as_longlong(q2) == 0) {           // the chase stopped: restart
          D[32 * (i + 1)] = dn - p;
          E[32 * m] = 0.0;
          split = true;
          break;
        }
        const double ir = rsqrt_nr(q2);
        E[32 * (i + 1)] = q2 * ir;
        s = f * ir;
        c = g * ir;
        g = dn - p;
        const double r = fma(di - g, s, 2.0 * c * b);
        p = s * r;
        D[32 * (i + 1)] = g + p;
        g = fma(c, r, -b);
        dn = di;
        rec(i, c, s);
      }
      if (split) continue;
      D[32 * l] = dn - p;
      E[32 * l] = g;
      E[32 * m] = 0.0;
    }
  }
  return true;
}

__global__ void __launch_bounds__(32) k_pf_ql(PfWork W, int nslot) {
  extern __shared__ __align__(16) cplx psm[];
  double* D = reinterpret_cast<double*>(psm) + threadIdx.x;
  double* E = D + 32 * W.mm;
  const int slot = blockIdx.x * 32 + threadIdx.x;
  if (slot >= nslot || W.status[slot] != 1) return;
  const int m = W.order[slot], cap = pf_rot_cap(W.mm);
  for (int i = 0; i < m; ++i) { D[32 * i] = W.sd[pf_ix(slot, i, W.mm)]; E[32 * i] = W.se[pf_ix(slot, i, W.mm)]; }
  int k = 0;
  const size_t base = (size_t)(slot >> 5) * cap * 32 + (slot & 31);
  const bool ok = lane_ql(D, E, m, [&](int i, double c, double s) {
    if (k < cap) { W.rot[base + (size_t)k * 32] = cmk(c, s); W.roti[base + (size_t)k * 32] = (unsigned char)i; }
    ++k;
  });
  W.nrot[slot] = k;
  if (!ok || k > pf_rot_cap(m)) W.status[slot] = 2;    // the Jacobi method (not cap: no choice of the chunk)
  for (int i = 0; i < m; ++i) W.sd[pf_ix(slot, i, W.mm)] = D[32 * i];
}

// Blocks whose overlap has directions at or below the cut (or no certificate
// against them): Sbar = Q diag(s) Q^H with Q = H_0 ... H_{m-3} D Z (reflectors, phases
// and rotations recorded above), K = {s > tau}, C = X^H Hbar X, X = Q_K diag(s_K)^-1/2.
__global__ void __launch_bounds__(128) k_pf_cut(const ProbDev* __restrict__ probs, const PfTask* __restrict__ tasks,
                                                const PfGroup* __restrict__ groups, PfWork W) {
  extern __shared__ __align__(16) cplx psm[];
  const int slot = blockIdx.x;
  const int status = W.status[slot];
  if (status != 1 && status != 2) return;
  const PfTask F = tasks[groups[slot / kPfGroup].task];
  const int m = probs[F.prob].m0, nup = m * (m + 1) / 2, ld = m | 1, mm = W.mm, cap = pf_rot_cap(mm);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nth = blockDim.x, nw = nth >> 5;
  cplx* V = psm;                               // m x ld: eigenvectors, then X
  cplx* H = V + (m + 1) * (m + 1);             // m x ld: Hbar, then C
  cplx* U = H + (m + 1) * (m + 1);             // reflectors (packed) and Z, then Hbar X
  double* Z = reinterpret_cast<double*>(U + nup);   // column i, row r: Z[i ld + r]
  __shared__ double sv[MAXM0], dd[MAXM0], ee[MAXM0], tt[MAXM0];
  __shared__ cplx hw[MAXM0], ph[MAXM0], vv[MAXM0];
  __shared__ cplx rot[128];
  __shared__ unsigned char roti[128];
  __shared__ int keep[MAXM0], s_r;
  __shared__ double rsq[MAXM0];
  // the kept directions, in ascending index, and s^-1/2
  auto choose = [&]() {
    if (tid == 0) {
      int r = 0;
      const double tau = *F.tau;
      for (int i = 0; i < m; ++i)
        if (sv[i] > tau && sv[i] > 0.0) { keep[r] = i; rsq[r] = rsqrt_nr(sv[i]); ++r; }
      s_r = r;
    }
  };
  if (status == 1) {
    for (int it = tid; it < m * m; it += nth) Z[(it / m) * ld + it % m] = (it / m == it % m) ? 1.0 : 0.0;
    for (int t = tid; t < nup; t += nth) U[t] = W.R[(size_t)slot * W.nup + t];
    // rotations on the rows of Z, a lane per row, on a warp that differs from CTA to
    // CTA (the CTAs of an SM then use different sub-partitions' FP64 units)
    const int zw = pf_lead(nw), cnt = W.nrot[slot];
    const size_t base = (size_t)(slot >> 5) * cap * 32 + (slot & 31);
    int last = -1;
    double zc = 0.0;                           // column `last` of this lane's row, in a register
    for (int k0 = 0; k0 < cnt; k0 += 128) {
      const int nk = min(128, cnt - k0);
      for (int k = tid; k < nk; k += nth) { rot[k] = W.rot[base + (size_t)(k0 + k) * 32]; roti[k] = W.roti[base + (size_t)(k0 + k) * 32]; }
      __syncthreads();
      if (warp == zw && lane < m)
        for (int k = 0; k < nk; ++k) {
          const int i = roti[k];
          const double c = rot[k].x, s = rot[k].y;
          double zj = zc;
          if (i + 1 != last) {                 // a new sweep: column `last` goes back first
            if (last >= 0) Z[last * ld + lane] = zc;
            zj = Z[(i + 1) * ld + lane];
          }
          const double zi = Z[i * ld + lane];
          Z[(i + 1) * ld + lane] = fma(s, zi, c * zj);
          zc = fma(c, zi, -s * zj);
          last = i;
        }
      __syncthreads();
    }
    if (warp == zw && lane < m && last >= 0) Z[last * ld + lane] = zc;
    if (tid == 0) {                            // phases: phi_0 = 1, phi_{k+1} = phi_k times the subdiagonal's
      cplx phi = cmk(1.0, 0.0);
      for (int k = 0; k < m; ++k) {
        ph[k] = phi;
        if (k + 1 < m) phi = cmul(phi, W.rph[(size_t)slot * mm + k]);
      }
    }
    for (int i = tid; i + 1 < m; i += nth) tt[i] = W.rtau[(size_t)slot * mm + i];
    for (int i = tid; i < m; i += nth) sv[i] = W.sd[pf_ix(slot, i, mm)];
    __syncthreads();
    choose();
    __syncthreads();
    for (int it = tid; it < m * s_r; it += nth) {   // the kept columns alone, scaled
      const int i = it % m, c = it / m;
      V[i * ld + c] = cscale(ph[i], Z[keep[c] * ld + i] * rsq[c]);
    }
    __syncthreads();
    for (int k = m - 3; k >= 0; --k) {         // V loses tau v (v^H V)
      const double tk = tt[k];
      if (__double_as_longlong(tk) == 0) continue;
      const int n = m - k - 1;
      auto vk = [&](int i) { const int a = k + 1 + i; return U[a * (a + 1) / 2 + k]; };
      const int nk = s_r;
      for (int it = tid; it < ((4 * nk + 31) & ~31); it += nth) {
        const int c = it >> 2, o = it & 3;
        cplx s = cmk(0.0, 0.0);
        if (c < nk)
          for (int i = o; i < n; i += 4) s = cfmac(V[(k + 1 + i) * ld + c], vk(i), s);
        s.x += __shfl_xor_sync(0xffffffffu, s.x, 1);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, 1);
        s.x += __shfl_xor_sync(0xffffffffu, s.x, 2);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, 2);
        if (c < nk && o == 0) hw[c] = cscale(s, -tk);
      }
      __syncthreads();
      for (int it = tid; it < n * nk; it += nth) {
        const int i = it / nk, c = it - i * nk;
        V[(k + 1 + i) * ld + c] = cfma(vk(i), hw[c], V[(k + 1 + i) * ld + c]);
      }
      __syncthreads();
    }
  } else {
    // QL ran out of iterations or rotations: cyclic Jacobi on Sbar
    const int lj = m + (m & 1);
    cplx* a = U;                               // lj x lj
    for (int t = tid; t < nup; t += nth) {
      int i, j;
      tri_pos(t, i, j);
      const cplx x = W.S[(size_t)slot * W.nup + t];
      a[i * lj + j] = x;
      a[j * lj + i] = cconj(x);
    }
    __syncthreads();
    cta_jacobi_herm(a, H, m, lj);              // (H is loaded below)
    for (int i = tid; i < m; i += nth) sv[i] = a[i * lj + i].x;
    __syncthreads();
    choose();
    __syncthreads();
    for (int it = tid; it < m * s_r; it += nth) {
      const int i = it / s_r, c = it - i * s_r;
      V[i * ld + c] = cscale(H[i * lj + keep[c]], rsq[c]);
    }
    __syncthreads();
  }
  for (int t = tid; t < nup; t += nth) {
    int a, b;
    tri_pos(t, a, b);
    const cplx x = W.H[(size_t)slot * W.nup + t];
    H[a * ld + b] = x;
    H[b * ld + a] = cconj(x);
  }
  __syncthreads();
  const int r = s_r;
  cplx* Y = U;                                 // m x r, pitch ld: Hbar X
  for (int it = tid; it < m * r; it += nth) {
    const int i = it / r, c = it - i * r;
    cplx s = cmk(0.0, 0.0);
    for (int q = 0; q < m; ++q) s = cfma(H[i * ld + q], V[q * ld + c], s);
    Y[i * ld + c] = s;
  }
  __syncthreads();
  for (int t = tid; t < r * (r + 1) / 2; t += nth) {   // C = X^H Y, lower triangle
    int a, b;
    tri_pos(t, a, b);
    cplx s = cmk(0.0, 0.0);
    for (int q = 0; q < m; ++q) s = cfmac(Y[q * ld + b], V[q * ld + a], s);
    if (a == b) s.y = 0.0;
    H[a * ld + b] = s;
  }
  __syncthreads();
  if (r > 0) cta_tridiag_lower(H, ld, r, dd, ee, tt, ph, vv, hw, pf_lead(nw));
  for (int i = tid; i < r; i += nth) {
    W.td[pf_ix(slot, i, mm)] = dd[i];
    W.te[pf_ix(slot, i, mm)] = ee[i];
  }
  if (tid == 0) { W.order[slot] = r; W.status[slot] = 0; }
}

__global__ void __launch_bounds__(32) k_pf_values(const ProbDev* __restrict__ probs, const PfTask* __restrict__ tasks,
                                                  const PfGroup* __restrict__ groups, PfWork W, int nslot) {
  extern __shared__ __align__(16) cplx psm[];
  double* D = reinterpret_cast<double*>(psm) + threadIdx.x;
  double* E = D + 32 * W.mm;
  const int slot = blockIdx.x * 32 + threadIdx.x;
  if (slot >= nslot) return;
  const PfGroup grp = groups[slot / kPfGroup];
  const PfTask F = tasks[grp.task];
  const int rep = grp.rep + slot % kPfGroup;
  if (rep >= F.nrep) return;
  const int m0 = probs[F.prob].m0, r = W.order[slot];
  for (int i = 0; i < r; ++i) { D[32 * i] = W.td[pf_ix(slot, i, W.mm)]; E[32 * i] = W.te[pf_ix(slot, i, W.mm)]; }
  if (!lane_ql(D, E, r, [](int, double, double) {})) {
    // out of iterations: bisection on the tridiagonal itself
    double d[MAXM0], e2[MAXM0];
    float df[MAXM0], e2f[MAXM0];
    for (int i = 0; i < r; ++i) {
      d[i] = W.td[pf_ix(slot, i, W.mm)];
      const double e = W.te[pf_ix(slot, i, W.mm)];
      e2[i] = (i + 1 < r) ? e * e : 0.0;
      df[i] = (float)d[i];
      e2f[i] = (float)e2[i];
    }
    for (int i = 0; i < r; ++i) D[32 * i] = tridiag_eig_fast(df, e2f, d, e2, r, i, 0.0);
  }
  // the conjugate block's spectrum too, where the task's range holds it
  const int jl = F.index(rep), j = F.j0 + jl;
  const int j3 = j % F.L[2], j2 = (j / F.L[2]) % F.L[1], j1 = j / (F.L[1] * F.L[2]);
  const int c1 = (F.L[0] - j1) % F.L[0], c2 = (F.L[1] - j2) % F.L[1], c3 = (F.L[2] - j3) % F.L[2];
  const int jm = (c1 * F.L[1] + c2) * F.L[2] + c3;
  const bool pair = jm != j && jm >= F.j0 && jm < F.j0 + F.nj;
  for (int i = 0; i < m0; ++i) {
    const double lam = (i < r) ? D[32 * i] : INFINITY;
    F.ev[(size_t)jl * m0 + i] = lam;
    if (F.blk) F.blk[(size_t)jl * m0 + i] = j;
    if (pair) {
      F.ev[(size_t)(jm - F.j0) * m0 + i] = lam;
      if (F.blk) F.blk[(size_t)(jm - F.j0) * m0 + i] = jm;
    }
  }
}

// Lattice eigenvectors from Fourier-block eigenvectors (Prop. A.1, the
// columns of the inverse DFT over the lattice index, U = (F^* (x) I) Ubar):
// U[c][(k, mu)] = f_j[k] y[mu] with f_j[k] = exp(+2 pi i j.k / L) / sqrt(|L|),
// for each requested pair c (Fourier index jbar[c], block-local vector
// vec[c] in ys).  One thread per entry; twiddles by sincospi of the exact
// integer phase j.k mod L.
__global__ void k_bloch_vectors(int L1, int L2, int L3, int m0, int nsel, const int* __restrict__ jbar,
                                const cplx* __restrict__ ys, const int* __restrict__ slot, cplx* __restrict__ U) {
  const long long nb = (long long)L1 * L2 * L3 * m0, tot = nb * nsel;
  const double inv = rsqrt((double)L1 * L2 * L3);
  for (long long it = blockIdx.x * (long long)blockDim.x + threadIdx.x; it < tot; it += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(it / nb);
    const long long a = it % nb;
    const int mu = (int)(a % m0);
    const long long kb = a / m0;
    const int k3 = (int)(kb % L3), k2 = (int)((kb / L3) % L2), k1 = (int)(kb / ((long long)L2 * L3));
    const int j = jbar[c];
    const int j3 = j % L3, j2 = (j / L3) % L2, j1 = j / (L2 * L3);
    // phase 2 pi (j1 k1 / L1 + j2 k2 / L2 + j3 k3 / L3), each term reduced exactly
    const double ph = 2.0 * ((double)((long long)j1 * k1 % L1) / L1 + (double)((long long)j2 * k2 % L2) / L2 +
                             (double)((long long)j3 * k3 % L3) / L3);
    double sn, cs;
    sincospi(ph, &sn, &cs);
    const cplx y = ys[(size_t)slot[c] * m0 + mu];
    U[it] = cscale(cmul(cmk(cs, sn), y), inv);
  }
}

void launch_bloch_vectors(int L1, int L2, int L3, int m0, int nsel, const int* jbar, const cplx* ys, const int* slot,
                          cplx* U, cudaStream_t st) {
  if (nsel > 0) k_bloch_vectors<<<1024, 256, 0, st>>>(L1, L2, L3, m0, nsel, jbar, ys, slot, U);
}

// One CTA per periodic problem: its dependency cut (NullTask).
__global__ void k_null_tau(const NullTask* __restrict__ tasks) {
  const NullTask T = tasks[blockIdx.x];
  const int np = T.m0 * T.m0;
  const size_t os = (size_t)T.nF * np;   // offset stride of a factor tensor
  double part = 0.0;
  for (int pr = threadIdx.x; pr < np; pr += blockDim.x) {
    double b = 1.0;
    for (int a = 0; a < 3; ++a) {
      double acc = 0.0;
      for (int o = 0; o < T.noff[a]; ++o) acc += fabs(T.X[a][(size_t)o * os + pr]);
      b *= acc;
    }
    part += b * b;
  }
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) t += red[w];
    *T.tau = null_tau(sqrt(t), (double)T.nb);
  }
}

void launch_null_tau(const NullTask* tasks, int ntask, cudaStream_t st) {
  if (ntask) k_null_tau<<<ntask, 256, 0, st>>>(tasks);
}

// ---- preconditioner ----


__global__ void k_sigma(const PrecTask* __restrict__ tasks) {
  const PrecTask T = tasks[blockIdx.x];
  __shared__ double red[256];
  double mn = DBL_MAX;
  for (int j = threadIdx.x; j < T.M; j += blockDim.x) mn = fmin(mn, T.emin[j]);
  red[threadIdx.x] = mn;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] = fmin(red[threadIdx.x], red[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *T.sigma = red[0] - T.rel_shift * (1.0 + fabs(red[0]));
}

__global__ void k_precond(const ProbDev* __restrict__ probs, const PrecTask* __restrict__ tasks) {
  extern __shared__ cplx sm[];
  const PrecTask T = tasks[blockIdx.y];
  const int j = blockIdx.x;
  if (j >= T.M) return;
  const int m0 = probs[T.prob].m0, np = m0 * m0;
  const double sg = *T.sigma;
  cplx* A = sm;
  cplx* Li = sm + np;
  for (int pr = threadIdx.x; pr < np; pr += blockDim.x) {
    cplx h = T.CH[(size_t)j * np + pr], s = T.CS[(size_t)j * np + pr];
    A[pr] = csub(h, cscale(s, sg));
  }
  __syncthreads();
  cta_cholesky(A, m0);
  // Li = L^-1 (lower), thread per column
  for (int c = threadIdx.x; c < m0; c += blockDim.x) {
    for (int i = 0; i < m0; ++i) {
      cplx s = cmk(i == c ? 1.0 : 0.0, 0.0);
      for (int q = c; q < i; ++q) s = csub(s, cmul(A[i * m0 + q], Li[q * m0 + c]));
      Li[i * m0 + c] = (i < c) ? cmk(0.0, 0.0) : cscale(s, 1.0 / A[i * m0 + i].x);
    }
  }
  __syncthreads();
  // K = L^-H L^-1 : K[a][b] = sum_i conj(Li[i][a]) Li[i][b]
  for (int pr = threadIdx.x; pr < np; pr += blockDim.x) {
    int a = pr / m0, b = pr % m0;
    cplx s = cmk(0.0, 0.0);
    for (int i = max(a, b); i < m0; ++i) s = cadd(s, cmulc(Li[i * m0 + b], Li[i * m0 + a]));
    T.K[(size_t)j * np + pr] = s;
  }
}

// ---- sorting of (value, index) pairs ----
// Order: ascending value, ties by ascending index.  Pads carry the largest key
// and an index above every real one, so they sort after the removed directions'
// +inf entries and the result is deterministic.  The values are compared as
// unsigned integers of the same order (an FP64 compare holds the FP64 pipe for
// 64 cycles a warp, twice per exchange: most of a pass's time).
__device__ inline unsigned long long sort_key(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x + 0.0);   // -0 sorts as +0
  return (b >> 63) ? ~b : b | 0x8000000000000000ull;
}
__device__ inline double sort_value(unsigned long long k) {
  return __longlong_as_double((long long)((k >> 63) ? k & 0x7FFFFFFFFFFFFFFFull : ~k));
}
__device__ inline bool pair_gt(unsigned long long va, int ia, unsigned long long vb, int ib) {
  return va > vb || (va == vb && ia > ib);
}
__device__ inline void sort_exchange(unsigned long long* v, int* idx, int i, int ij, bool up) {
  const unsigned long long a = v[i], b = v[ij];
  const int ia = idx[i], ib = idx[ij];
  if (pair_gt(a, ia, b, ib) == up) { v[i] = b; v[ij] = a; idx[i] = ib; idx[ij] = ia; }
}

__global__ void k_sort_small(const SortTask* __restrict__ tasks) {
  extern __shared__ unsigned long long ssv[];
  const SortTask T = tasks[blockIdx.x];
  int n2 = 1;
  while (n2 < T.n) n2 <<= 1;
  unsigned long long* sv = ssv;
  int* si = (int*)(ssv + n2);
  for (int i = threadIdx.x; i < n2; i += blockDim.x) {
    sv[i] = (i < T.n) ? sort_key(T.v[i]) : ~0ull;
    si[i] = (i < T.n) ? (T.idx ? T.idx[i] : i) : 0x7fffffff;
  }
  __syncthreads();
  for (int k = 2; k <= n2; k <<= 1)
    for (int jj = k >> 1; jj > 0; jj >>= 1) {
      for (int t = threadIdx.x; t < n2 / 2; t += blockDim.x) {
        const int i = ((t & ~(jj - 1)) << 1) | (t & (jj - 1));
        sort_exchange(sv, si, i, i + jj, (i & k) == 0);
      }
      __syncthreads();
    }
  for (int i = threadIdx.x; i < T.n; i += blockDim.x) {
    T.v[i] = sort_value(sv[i]);
    if (T.idx) T.idx[i] = si[i];
  }
}

// The global bitonic network: compare-exchange passes over pairs kSortTile or more
// apart go over global memory, one launch each; the runs of closer passes that
// follow each of them, and the first levels up to kSortTile, are done on tiles in
// shared memory.  15 of 136 passes are global for 65536 pairs, 45 of 210 for 2^20:
// 568 -> 142 us and 1.49 -> 0.51 ms (one launch and two FP64 compares per pass before).
constexpr int kSortTile = 2048;
__global__ void __launch_bounds__(1024) k_bitonic_tile(unsigned long long* v, int* idx, int n2, int k0, int k1) {
  __shared__ unsigned long long sv[kSortTile];
  __shared__ int si[kSortTile];
  const int tile = min(kSortTile, n2), base = blockIdx.x * tile;
  for (int i = threadIdx.x; i < tile; i += blockDim.x) { sv[i] = v[base + i]; si[i] = idx[base + i]; }
  __syncthreads();
  for (int k = k0; k <= k1; k <<= 1)
    for (int jj = min(k, tile) >> 1; jj > 0; jj >>= 1) {
      for (int t = threadIdx.x; t < tile / 2; t += blockDim.x) {
        const int i = ((t & ~(jj - 1)) << 1) | (t & (jj - 1));
        sort_exchange(sv, si, i, i + jj, ((base + i) & k) == 0);
      }
      __syncthreads();
    }
  for (int i = threadIdx.x; i < tile; i += blockDim.x) { v[base + i] = sv[i]; idx[base + i] = si[i]; }
}

// one compare-exchange pass over pairs jj apart (n2 a power of 2; padded)
__global__ void k_bitonic_pass(unsigned long long* v, int* idx, int n2, int k, int jj) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n2 / 2; t += gridDim.x * blockDim.x) {
    const int i = ((t & ~(jj - 1)) << 1) | (t & (jj - 1));
    sort_exchange(v, idx, i, i + jj, (i & k) == 0);
  }
}

__global__ void k_pad_copy(const double* v, const int* idx, int n, unsigned long long* pv, int* pidx, int n2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += gridDim.x * blockDim.x) {
    pv[i] = (i < n) ? sort_key(v[i]) : ~0ull;
    pidx[i] = (i < n) ? (idx ? idx[i] : i) : 0x7fffffff;
  }
}

__global__ void k_unpad_copy(const unsigned long long* pv, const int* pidx, int n, double* v, int* idx) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    v[i] = sort_value(pv[i]);
    if (idx) idx[i] = pidx[i];
  }
}

// ---- launchers ----
// m0: the launch's largest block order; any_odd: some block of the launch has
// odd m0 (its layout keeps a padded work array of its own)
size_t fblocks_smem(int m0, bool vectors, bool any_odd) {
  const int ldj = m0 + (m0 & 1);
  const size_t mats = (!any_odd && !(m0 & 1)) ? (size_t)2 * m0 * m0 + (size_t)ldj * ldj
                                              : (size_t)2 * m0 * m0 + (size_t)2 * ldj * ldj;
  return (mats + 2 * MAXM0) * sizeof(cplx) + 3 * MAXM0 * sizeof(double) + 2 * MAXM0 * sizeof(float) +
         (vectors ? 16 + 2 * ldj * ldj * sizeof(cplx) : 0);
}

void launch_fblocks(const ProbDev* probs, const FBlockTask* tasks, int ntask, int maxnj, int maxm0,
                    cudaStream_t st, bool vectors, bool any_odd) {
  if (!ntask || maxnj <= 0) return;
  size_t sm = fblocks_smem(maxm0, vectors, any_odd);
  FOCK_SMEM_OPTIN(k_fblocks);
  {   // the largest shared-memory carveout: four 32 x 32 blocks (~54 KB each) per SM
    static std::once_flag carve;
    std::call_once(carve, [] { cudaFuncSetAttribute(k_fblocks, cudaFuncAttributePreferredSharedMemoryCarveout, 100); });
  }
  // the rotation and update phases of an m0 x m0 block have about m0^2 / 2
  // parallel items: one warp for m0 <= 8 (more independent blocks resident
  // per SM keep the FP64 pipe busy), up to four warps for m0 = 32
  const int threads = (maxm0 <= 8) ? 32 : (maxm0 <= 16) ? 64 : 128;
  k_fblocks<<<dim3(maxnj, ntask), threads, sm, st>>>(probs, tasks);
}

// Bytes of workspace for nslot blocks of order at most m, and its layout. The arrays
// hold multiples of 32 slots.
size_t pf_layout(char* base, int m, size_t nslot, PfWork* W) {
  const size_t ns = (nslot + 31) & ~(size_t)31, nup = (size_t)m * (m + 1) / 2, cap = pf_rot_cap(m);
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = base + off;
    off += (bytes + 255) & ~(size_t)255;
    return p;
  };
  PfWork w;
  w.mm = m; w.nup = (int)nup;
  w.H = (cplx*)take(ns * nup * sizeof(cplx)); w.S = (cplx*)take(ns * nup * sizeof(cplx));
  w.R = (cplx*)take(ns * nup * sizeof(cplx));
  w.sd = (double*)take(ns * m * sizeof(double)); w.se = (double*)take(ns * m * sizeof(double));
  w.td = (double*)take(ns * m * sizeof(double)); w.te = (double*)take(ns * m * sizeof(double));
  w.rtau = (double*)take(ns * m * sizeof(double)); w.rph = (cplx*)take(ns * m * sizeof(cplx));
  w.rot = (cplx*)take(ns * cap * sizeof(cplx)); w.roti = (unsigned char*)take(ns * cap);
  w.nrot = (int*)take(ns * sizeof(int)); w.order = (int*)take(ns * sizeof(int)); w.status = (int*)take(ns * sizeof(int));
  if (W) *W = w;
  return off;
}

// The blocks of ng groups; none of an order above W.mm.
void launch_pf(const ProbDev* probs, const PfTask* tasks, const PfGroup* groups, int ng, const PfWork& W,
               cudaStream_t st) {
  if (ng <= 0) return;
  const int m = W.mm, nslot = ng * kPfGroup;
  const size_t qs = (size_t)2 * 32 * m * sizeof(double), rs = (size_t)m * (m | 1) * sizeof(cplx);
  const size_t cs = (size_t)3 * (m + 1) * (m + 1) * sizeof(cplx);
  const int tiles = (W.nup + 31) / 32;
  if ((long long)ng * tiles >= 4 * 152)
    k_pf_form<kPfGroup><<<dim3(ng, tiles), 32, 0, st>>>(probs, tasks, groups, W);
  else
    k_pf_form<2><<<dim3(nslot / 2, tiles), 32, 0, st>>>(probs, tasks, groups, W);
  if (m <= 8) k_pf_reduce<32, 2><<<nslot, 32, rs, st>>>(probs, tasks, groups, W);
  else if (m <= 16) k_pf_reduce<64, 3><<<nslot, 64, rs, st>>>(probs, tasks, groups, W);
  else {
    FOCK_SMEM_OPTIN((k_pf_reduce<128, 5>));
    k_pf_reduce<128, 5><<<nslot, 128, rs, st>>>(probs, tasks, groups, W);
  }
  k_pf_ql<<<(nslot + 31) / 32, 32, qs, st>>>(W, nslot);
  FOCK_SMEM_OPTIN(k_pf_cut);
  {   // the largest shared-memory carveout: four 32 x 32 blocks per SM
    static std::once_flag carve;
    std::call_once(carve, [] { cudaFuncSetAttribute(k_pf_cut, cudaFuncAttributePreferredSharedMemoryCarveout, 100); });
  }
  k_pf_cut<<<nslot, m <= 8 ? 32 : m <= 16 ? 64 : 128, cs, st>>>(probs, tasks, groups, W);
  k_pf_values<<<(nslot + 31) / 32, 32, qs, st>>>(probs, tasks, groups, W, nslot);
}

void launch_precond(const ProbDev* probs, const PrecTask* tasks, int ntask, int maxM, int maxm0,
                    cudaStream_t st) {
  if (!ntask) return;
  k_sigma<<<ntask, 256, 0, st>>>(tasks);
  size_t sm = (size_t)2 * maxm0 * maxm0 * sizeof(cplx);
  FOCK_SMEM_OPTIN(k_precond);
  k_precond<<<dim3(maxM, ntask), 128, sm, st>>>(probs, tasks);
}

void launch_sort_small(const SortTask* tasks, int ntask, int maxn, cudaStream_t st) {
  if (!ntask) return;
  int n2 = 1;
  while (n2 < maxn) n2 <<= 1;
  size_t sm = (size_t)n2 * (sizeof(double) + sizeof(int));
  FOCK_SMEM_OPTIN(k_sort_small);
  k_sort_small<<<ntask, 512, sm, st>>>(tasks);
}

// sort n pairs in place with scratch (pv, pidx of length n2 = next pow2)
void launch_sort_global(double* v, int* idx, int n, double* pv, int* pidx, cudaStream_t st) {
  int n2 = 1;
  while (n2 < n) n2 <<= 1;
  unsigned long long* key = reinterpret_cast<unsigned long long*>(pv);
  const int grid = std::min(4096, (n2 + 255) / 256), half = std::min(4096, (n2 / 2 + 255) / 256);
  const int tile = std::min(kSortTile, n2), nt = n2 / tile;
  k_pad_copy<<<grid, 256, 0, st>>>(v, idx, n, key, pidx, n2);
  k_bitonic_tile<<<nt, 1024, 0, st>>>(key, pidx, n2, 2, tile);
  for (int k = 2 * tile; k <= n2; k <<= 1) {
    for (int jj = k >> 1; jj >= tile; jj >>= 1) k_bitonic_pass<<<half, 256, 0, st>>>(key, pidx, n2, k, jj);
    k_bitonic_tile<<<nt, 1024, 0, st>>>(key, pidx, n2, k, k);
  }
  k_unpad_copy<<<grid, 256, 0, st>>>(key, pidx, n, v, idx);
}

}  // namespace fock
