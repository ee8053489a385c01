// Representatives of the Fourier indices of an L1 x L2 x L3 lattice: with real generators the
// block at -j (componentwise mod L) is the conjugate of the block at j, with the same
// spectrum; the lower index stands for the pair.  Host and device, and on the CPU alone for the
// tests.
#ifndef FOCK_PF_INDEX_H
#define FOCK_PF_INDEX_H

#ifdef __CUDACC__
#define FOCK_PF_HD __host__ __device__
#else
#define FOCK_PF_HD
#endif

namespace fock {

// For j1 = 0 (and L1 / 2) the representatives are those of the L2 x L3 lattice, for 0 < j1 < L1 / 2 every
// (j2, j3), for larger j1 none; likewise for the second axis.
FOCK_PF_HD inline int pf_count(const int* L) {
  const int c3 = L[2] / 2 + 1, c2 = c3 * (2 - L[1] % 2) + (L[1] - 1) / 2 * L[2];
  return c2 * (2 - L[0] % 2) + (L[0] - 1) / 2 * (L[1] * L[2]);
}

// The r-th representative in ascending order: a few additions, so that a spectrum needs no list.
FOCK_PF_HD inline int pf_index(const int* L, int r) {
  const int n3 = L[2], n23 = L[1] * L[2], h1 = (L[0] - 1) / 2 * n23, h2 = (L[1] - 1) / 2 * n3;
  const int c3 = n3 / 2 + 1, c2 = c3 * (2 - L[1] % 2) + h2;
  int base = 0;
  if (r >= c2) {
    r -= c2;
    if (r < h1) return n23 + r;
    r -= h1;
    base = L[0] / 2 * n23;
  }
  if (r < c3) return base + r;
  r -= c3;
  if (r < h2) return base + n3 + r;
  return base + L[1] / 2 * n3 + (r - h2);
}

}  // namespace fock

#endif
