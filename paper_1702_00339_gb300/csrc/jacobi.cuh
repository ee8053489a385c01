// Parallel cyclic Jacobi of one CTA, for the Rayleigh-Ritz step's projected matrices
// (k_rr.cu) and the cell overlaps (k_lobpcg.cu).
#pragma once
#include "common.cuh"

namespace fock {

constexpr int kJacobiMax = 256;   // order, at most 255

// Parallel cyclic Jacobi on the symmetric n x n matrix a (row-major, stride
// ld >= n + 1), round-robin pairing, A' = J^T A J; eigenvectors accumulated in
// v.  Odd n is padded with a decoupled huge diagonal entry.  At exit the
// eigenvalues are on the diagonal of a (unsorted).  The matrices met here are
// nearly diagonal: rounds without a rotation cost one barrier, and a matrix that
// needs none returns false at once, v untouched (the identity).
static __device__ bool cta_jacobi(double* a, double* v, int n, int ld) {
  __shared__ double rc[kJacobiMax / 2], rs[kJacobiMax / 2];
  __shared__ int rp[kJacobiMax / 2], rq[kJacobiMax / 2];
  __shared__ double red[32], s_thr;
  const int ne = n + (n & 1);
  // rotation threshold: |a_pq| <= 1e-14 ||A||_F leaves the pair alone (rounding level)
  double part = 0.0;
  for (int it = threadIdx.x; it < n * n; it += blockDim.x) {
    const double x = a[(it / n) * ld + (it % n)];
    part = fma(x, x, part);
  }
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) t += red[w];
    s_thr = 1e-14 * sqrt(t);
  }
  __syncthreads();
  const double thr = s_thr;
  auto rotates = [&](int p, int q) {   // |a_pq| above the threshold and > 1e-17 sqrt|a_pp a_qq|
    const double apq = a[p * ld + q];
    return fabs(apq) > thr && apq * apq > 1e-34 * fabs(a[p * ld + p] * a[q * ld + q]);
  };
  int need = 0;
  for (int it = threadIdx.x; it < n * n; it += blockDim.x)
    if (it / n < it % n) need |= rotates(it / n, it % n);
  if (!__syncthreads_or(need)) return false;
  for (int it = threadIdx.x; it < ne * ne; it += blockDim.x) {
    int i = it / ne, j = it % ne;
    v[i * ld + j] = (i == j) ? 1.0 : 0.0;
    if (i == n || j == n) a[i * ld + j] = (i == j) ? 1e300 : 0.0;
  }
  __syncthreads();
  for (int sweep = 0; sweep < 40; ++sweep) {
    bool any = false;
    for (int rnd = 0; rnd < ne - 1; ++rnd) {
      int rot = 0;
      for (int pi = threadIdx.x; pi < ne / 2; pi += blockDim.x) {
        int x = (pi == 0) ? 0 : ((pi - 1 + rnd) % (ne - 1)) + 1;
        int y = ((ne - 2 - pi + rnd) % (ne - 1)) + 1;
        int p = min(x, y), q = max(x, y);
        double c = 1.0, s = 0.0;
        if (rotates(p, q)) {
          // reciprocals and square roots by Newton-Raphson from FP32 seeds
          const double th = (a[q * ld + q] - a[p * ld + p]) * (0.5 * rcp_nr(a[p * ld + q]));
          const double yy = fma(th, th, 1.0);
          double t = rcp_nr(fabs(th) + yy * rsqrt_nr(yy));
          if (th < 0.0) t = -t;
          c = rsqrt_nr(fma(t, t, 1.0));
          s = t * c;
          rot = 1;
        }
        rp[pi] = p; rq[pi] = q; rc[pi] = c; rs[pi] = s;
      }
      if (!__syncthreads_or(rot)) continue;
      any = true;
      const int np2 = ne / 2;
      for (int it = threadIdx.x; it < np2 * ne; it += blockDim.x) {   // rows p, q
        int pi = it / ne, jj = it % ne;
        double s = rs[pi];
        if (s == 0.0) continue;
        int p = rp[pi], q = rq[pi];
        double c = rc[pi];
        double ap = a[p * ld + jj], aq = a[q * ld + jj];
        a[p * ld + jj] = c * ap - s * aq;
        a[q * ld + jj] = s * ap + c * aq;
      }
      __syncthreads();
      for (int it = threadIdx.x; it < np2 * ne; it += blockDim.x) {   // columns p, q and v
        int pi = it / ne, ii = it % ne;
        double s = rs[pi];
        if (s == 0.0) continue;
        int p = rp[pi], q = rq[pi];
        double c = rc[pi];
        double ap = a[ii * ld + p], aq = a[ii * ld + q];
        a[ii * ld + p] = c * ap - s * aq;
        a[ii * ld + q] = s * ap + c * aq;
        double vp = v[ii * ld + p], vq = v[ii * ld + q];
        v[ii * ld + p] = c * vp - s * vq;
        v[ii * ld + q] = s * vp + c * vq;
      }
      __syncthreads();
    }
    if (!any) break;      // uniform
  }
  return true;
}

}  // namespace fock
