// FP64 matrix products on the fifth-generation tensor cores by exact
// split products (the error-free splitting of Ozaki, Ogita, Oishi and Rump,
// "Error-free transformations of matrix multiplication by using fast routines
// of matrix multiplication", Numer. Algorithms 59 (2012)), used by the mixed
// form for the quadrature contractions of stage (a) (Lemma 2.1 display,
// Eqs. 2.16-2.17: X_t[mu nu] = sum_r P_t[r] Z[r][mu nu]) and for the dense
// products of the block iteration.
//
// Over a range of up to RANGE = 512 of the summation index, every row of A and
// every column of B is aligned to its largest binary exponent (k_split_exps) and
// cut to 55 bits below it, which are written as NDIG = 8 balanced base-128
// digits (-64 .. 64, exact in FP16).  For each level g = j + l (2 <= g <= NDIG + 1)
// the products of digit planes j of A and l of B are summed by tcgen05.mma
// (kind::f16, FP16 x FP16 -> FP32) into one TMEM accumulator per level: at most
// 8 x 512 x 64^2 = 2^24, so FP32 accumulation is exact over a whole range.
// Then each thread combines its row's levels in 64-bit integers, makes a double
// of the sum with integer instructions (an FP64 instruction costs 64 of them
// here) and adds ranges in FP64.  With 2^a, 2^b the powers of two at or below the largest
// of the row and of the column, a summand's error is below 2^(a + b) times 2^-52 (the cut
// operands) and 2^-51.2 (the levels above NDIG + 1): 2^-50.5.  On random operands 6e-16
// to 3e-15 of the largest entries' product (with 7 truncated digits, 49 bits, aligned over
// 64 summands, as this was: 2^-44 and 1e-13).
//
// Where a row falls while a column rises, the largest over a range say little about the
// products: with both over 2^40 the sum would keep 20 bits.  So, where the task asks for it
// (SplitTask::graded), a tile's range is aligned as a
// whole only if every row and column of it has a block of 64 summands in which the
// two, together, are within 2^3 of their largest over the range: 512 summands' errors of
// 2^(a + b - 50.5) are then below what that one block's 64 of 2^(a' + b' - 44) may be. Else the
// range is taken in its blocks of 64, each aligned for itself.  The look is taken before the
// loop over the ranges: inside it, where all registers are in use, it made long sums 5 % slower.
// 216 x 216 x 16384, not symmetric: 146 us a call, 257 where every range is graded.
//
// One CTA of 384 threads per 128 x 64 output tile and K range.  Stages of KC = 32
// summands in two buffers: the threads load and split the next stage while the
// tensor core works on this one.  A thread splits eight summands of a row into the
// 16 bytes of a core matrix row per plane (no-swizzle K-major layout: 8 rows x 16
// bytes per core matrix); summands oct + 4 i, i = 0..7, go to octet oct, the same
// permutation in A and B, so that four lanes read whole sectors.  The B planes
// lie one after another, so one MMA of up to 256 columns covers four levels of an
// A plane: 12 reads of A instead of 36.  One thread issues; every wait is bounded
// (clock64), after which the kernel flags an error, frees its TMEM and returns.
//
// 216 x 216 x 16384 (a symmetric Gram product, at most 32 ranges): 384 -> 119 us with the
// reduction; bound by the splitting, about 55 instructions per summand and row that every
// tile does for its own rows and columns (ALU pipe 59 %, issue slots 46 %, tensor pipe 30 %
// of active cycles, and a barrier per stage).
#include <cuda_fp16.h>
#include <stdint.h>

#include "common.cuh"

namespace fock {

namespace {

constexpr int TM = 128, TN = 64, KC = 32, NDIG = 8;                // digit levels g = 2 .. NDIG + 1
constexpr int kSplitThreads = 384;   // three warps a sub-partition split the operands, eight of the twelve read TMEM
constexpr int TMEM_COLS = 512;                                     // NDIG * TN
constexpr uint32_t A_PLANE = TM * KC * 2, B_PLANE = TN * KC * 2;   // bytes per digit plane
constexpr uint32_t STAGE = NDIG * (A_PLANE + B_PLANE);
constexpr int kFineRanges = 2048;    // ranges of a CTA looked at; any more (past 2^20 summands) are taken in blocks
constexpr size_t SPLIT_SMEM = 2 * (size_t)STAGE + 1024;
constexpr long long kWaitCycles = 4000000000ll;                    // ~2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// byte offset of octet o of row r of an R x KC operand: core matrix (r/8, o), K-adjacent
// core matrices 128 B apart (LBO), 8-row groups KC/8 * 128 B apart (SBO)
__device__ __forceinline__ uint32_t core_off(int r, int o) {
  return (uint32_t)(((r >> 3) * (KC >> 3) + o) * 128 + (r & 7) * 16);
}

__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  const uint64_t lbo = 128, sbo = (KC / 8) * 128;
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((lbo >> 4) & 0x3FFF) << 16 | ((sbo >> 4) & 0x3FFF) << 32 |
         (uint64_t)1 << 46;   // version 1, base offset 0, no swizzle
}

// instruction descriptor: D FP32, A and B FP16, both K-major, M = TM, N = n
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(TM >> 4) << 24);

// biased exponent field of |x| from its high word (0 for zero and subnormals: they align as exponent 1)
__device__ __forceinline__ int exp_field(int hi) { return max((hi >> 20) & 0x7FF, 1); }

// x = w 2^(E - 1077), cut to an integer |w| <= 2^55, plus 64 in every base-128 digit: the low
// and the high word
__device__ __forceinline__ uint2 offset_digits(double x, int E) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const int ex = (int)((h >> 20) & 0x7FF), s = min(E - max(ex, 1), 63);
  const uint32_t mh = (h & 0xFFFFFu) + (uint32_t)min(ex, 1) * 0x100000u;
  uint32_t a = l << 2, b = __funnelshift_l(l, mh, 2);
  if (s >= 32) { a = b; b = 0; }
  a = __funnelshift_r(a, b, s & 31);
  b >>= s & 31;
  const uint32_t sg = (uint32_t)((int)h >> 31);
  constexpr unsigned long long off = 64ull * ((1ull << 56) - 1) / 127;   // 64 (1 + 128 + ... + 128^7)
  const unsigned long long t = ((unsigned long long)(b ^ sg) << 32 | (a ^ sg)) +
                               ((unsigned long long)(uint32_t)(off >> 32) << 32 | ((uint32_t)off - sg));
  return make_uint2((uint32_t)t, (uint32_t)(t >> 32));
}

// A digit of two offset numbers as a pair of FP16, from the words a and b that hold it at byte P,
// bit O (at most 3): a byte permutation and a mask put u 2^O into the mantissas of 1024, one
// packed FMA takes the offsets off and the scale away (exact).
template <int P, int O, uint32_t MASK>
__device__ __forceinline__ uint32_t digit_pair(uint32_t a, uint32_t b) {
  constexpr uint32_t q = P < 3 ? P + 1 : 3, sel = P | q << 4 | (P + 4) << 8 | (q + 4) << 12;
  constexpr uint32_t m = MASK << O;
  const uint32_t w = (__byte_perm(a, b, sel) & (m | m << 16)) | 0x64006400u;
  __half2 v;
  *reinterpret_cast<uint32_t*>(&v) = w;
  v = __hfma2(v, __float2half2_rn(1.0f / (1 << O)), __float2half2_rn(-1024.0f / (1 << O) - 64.0f));
  return *reinterpret_cast<uint32_t*>(&v);
}
template <int P, int O, uint32_t MASK>
__device__ __forceinline__ void put_plane(const uint32_t* w, unsigned char* p) {
  *reinterpret_cast<uint4*>(p) = make_uint4(digit_pair<P, O, MASK>(w[0], w[1]), digit_pair<P, O, MASK>(w[2], w[3]),
                                            digit_pair<P, O, MASK>(w[4], w[5]), digit_pair<P, O, MASK>(w[6], w[7]));
}

__device__ __forceinline__ bool wait_phase(uint32_t mbar, uint32_t phase) {
  const long long t0 = clock64();
  uint32_t done = 0;
  while (!done) {
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(mbar), "r"(phase) : "memory");
    if (!done && clock64() - t0 > kWaitCycles) return false;
  }
  return true;
}

// One warp's share of an operand: eight rows, four lanes each (summands contiguous), or
// 32 rows of one octet.  Rows that do not exist and summands from kend on are zero.
struct Share {
  const double* p;     // the row's element 0, null: no such row
  long long sk;
  int row, oct, E;
  __device__ void place(const double* P, long long sr, long long k1, int rows, int it, int lane) {
    sk = k1;
    if (k1 == 1) { row = it * 8 + (lane & 7); oct = lane >> 3; }
    else { row = (it >> 2) * 32 + lane; oct = it & 3; }
    p = row < rows ? P + row * sr : nullptr;
  }
  __device__ void load(double* x, int k0, int kend) const {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = k0 + oct + 4 * i;
      x[i] = (p && k < kend) ? p[k * sk] : 0.0;
    }
  }
  __device__ void store(const double* x, unsigned char* planes, uint32_t plane) const {
    uint32_t lo[8], hi[8], l4[8];   // l4: the number four bits down, low word
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint2 t = offset_digits(x[i], E);
      lo[i] = t.x;
      hi[i] = t.y;
      l4[i] = __funnelshift_r(t.x, t.y, 4);
    }
    unsigned char* p = planes + core_off(row, oct);
    put_plane<2, 1, 0xFF>(hi, p);              // bit 49; up to 128
    put_plane<1, 2, 0x7F>(hi, p + plane);      // 42
    put_plane<0, 3, 0x7F>(hi, p + 2 * plane);  // 35
    put_plane<3, 0, 0x7F>(l4, p + 3 * plane);  // 28
    put_plane<2, 1, 0x7F>(l4, p + 4 * plane);  // 21
    put_plane<1, 2, 0x7F>(l4, p + 5 * plane);  // 14
    put_plane<0, 3, 0x7F>(l4, p + 6 * plane);  // 7
    put_plane<0, 0, 0x7F>(lo, p + 7 * plane);  // 0
  }
};

// S 2^e, rounded to nearest, by integer instructions where the result is a normal number
__device__ __forceinline__ double scaled_int(long long S, int e) {
  const unsigned long long a = S < 0 ? 0ull - (unsigned long long)S : (unsigned long long)S;
  if (a == 0) return 0.0;
  const int lz = __clzll((long long)a), be = 1086 - lz + e;
  if (be < 1 || be > 2045) return scalbn((double)S, e);
  const unsigned long long m = a << lz, r = (m >> 11) + ((m >> 10) & 1);   // 2^52 <= r <= 2^53
  return __longlong_as_double((long long)((((unsigned long long)(be - 1)) << 52) + r) | (S & (1ll << 63)));
}

}  // namespace

// Exponents of the rows of A (and columns of B) over each range, and where ranges have more
// than one block over those (SplitExps): a warp per row, or where summands are apart a lane.
__global__ void __launch_bounds__(256) k_split_exps(const SplitTask* __restrict__ tasks) {
  const SplitTask T = tasks[blockIdx.y];
  if (T.active && *T.active == 0) return;
  const SplitRanges R(T.K, T.ksplit);
  const SplitExps X(T, R);
  constexpr int NB = SplitRanges::BLOCKS, KB = SplitRanges::BLOCK;
  const int lane = threadIdx.x & 31, nb = R.blocks();
  const bool looked = T.blocks() > 1;
  const long long w0 = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), nw = (long long)gridDim.x * (blockDim.x >> 5);
  for (int o = 0; o < (T.same() ? 1 : 2); ++o) {
    const double* P = o ? T.B : T.A;
    const long long sr = o ? T.b_n : T.a_m, sk = o ? T.b_k : T.a_k;
    const int rows = o ? T.N : T.M;
    int *const wide = X.wide(o), *const near = X.near(o), *const block = X.block(o, nb);
    if (sk == 1) {
      for (long long w = w0; w < (long long)R.count() * rows; w += nw) {
        const int e = (int)(w / rows), r = (int)(w % rows), k0 = R.begin(e) + lane, k1 = R.end(e);
        const int* p = reinterpret_cast<const int*>(P + r * sr) + 1;   // (high words; all loads before the first use)
        int h[NB][2], Eb = 1;
#pragma unroll
        for (int c = 0; c < NB; ++c)
          if (c < nb) {                        // uniform
            h[c][0] = k0 + c * KB < k1 ? p[2 * (k0 + c * KB)] : 0;
            h[c][1] = k0 + c * KB + 32 < k1 ? p[2 * (k0 + c * KB + 32)] : 0;
          }
#pragma unroll
        for (int c = 0; c < NB; ++c)
          if (c < nb) {
            const int E = __reduce_max_sync(0xffffffffu, max(exp_field(h[c][0]), exp_field(h[c][1])));
            if (lane >> 2 == c) Eb = E;        // four lanes a block
          }
        const int E = nb > 1 ? __reduce_max_sync(0xffffffffu, Eb) : __shfl_sync(0xffffffffu, Eb, 0);
        uint32_t q = 0;
        if (looked) {
          for (int i = 0; i < 4; ++i) q |= __ballot_sync(0xffffffffu, E - Eb <= i) & (0x11111111u << i);
          if ((lane & 3) == 0 && lane >> 2 < nb) block[((long long)e * nb + (lane >> 2)) * rows + r] = Eb;
        }
        if (lane == 0) {
          wide[w] = E;
          if (looked) near[w] = (int)q;
        }
      }
    } else {
      const int rg = (rows + 31) >> 5;
      for (long long w = w0; w < (long long)R.count() * rg; w += nw) {
        const int e = (int)(w / rg), r = (int)(w % rg) * 32 + lane;
        if (r >= rows) continue;
        int Eb[NB], E = 1;
#pragma unroll 1
        for (int c = 0; c < nb; ++c) {
          const int k0 = R.begin(e) + c * KB, k1 = min(k0 + KB, R.end(e));
          int x = 1;
#pragma unroll 8
          for (int k = k0; k < k1; ++k) x = max(x, exp_field(__double2hiint(P[r * sr + k * sk])));
          if (looked) block[((long long)e * nb + c) * rows + r] = x;
          Eb[c] = x;
          E = max(E, x);
        }
        wide[(long long)e * rows + r] = E;
        if (!looked) continue;
        uint32_t q = 0;
#pragma unroll 1
        for (int c = 0; c < nb; ++c) q |= (0xfu << min(E - Eb[c], 4) & 0xfu) << (4 * c);   // bits E - Eb[c] .. 3
        near[(long long)e * rows + r] = (int)q;
      }
    }
  }
}

// the four bits of each block in reverse
__device__ __forceinline__ uint32_t near_rev(uint32_t x) {
  x = (x & 0x55555555u) << 1 | (x >> 1 & 0x55555555u);
  return (x & 0x33333333u) << 2 | (x >> 2 & 0x33333333u);
}

__global__ void __launch_bounds__(kSplitThreads, 1) k_split_gemm(const SplitTask* __restrict__ tasks, int max_ks, int* err) {
  const SplitTask T = tasks[blockIdx.z / max_ks];
  const int ks = blockIdx.z % max_ks;
  const SplitRanges R(T.K, T.ksplit);
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  if (ks >= R.nks || m0 >= T.M || n0 >= T.N) return;
  if (T.active && *T.active == 0) return;
  if (T.work && T.sym && n0 + TN <= m0) return;   // wholly below the diagonal: mirrored by the reduction
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* buf = (unsigned char*)(((uintptr_t)smem + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail, exB[TN];
  __shared__ uint32_t s_fine[kFineRanges / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rowsA = min(TM, T.M - m0), colsB = min(TN, T.N - n0);
  if (tid == 0) {
    s_fail = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&mbar[0])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&mbar[1])));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(smem_u32(&tmem_base)), "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  // The ranges to be taken in blocks, a warp each, before the loop (whose registers are all in
  // use).  A row and a column agree in block c for some i if c is among the row's within i
  // and the column's within 3 - i: one AND with the column's bits in reverse.  Mostly all
  // rows and columns of the tile agree in one block and i; else each pair is looked at.
  const SplitExps X(T, R);
  const int nb = T.blocks();
  if (nb > 1) {
    if (tid < kFineRanges / 32) s_fine[tid] = 0;
    __syncthreads();
    for (int d = warp; d < min(R.per, kFineRanges); d += kSplitThreads / 32) {
      const int e = ks * R.per + d;
      const int* nA = X.near(false) + (long long)e * T.M + m0;
      const int* nB = X.near(!T.same()) + (long long)e * T.N + n0;
      uint32_t a[TM / 32], b[TN / 32], common = ~0u;
#pragma unroll
      for (int j = 0; j < TM / 32; ++j) common &= a[j] = lane + 32 * j < rowsA ? (uint32_t)nA[lane + 32 * j] : ~0u;
#pragma unroll
      for (int j = 0; j < TN / 32; ++j) common &= b[j] = lane + 32 * j < colsB ? near_rev((uint32_t)nB[lane + 32 * j]) : ~0u;
      if (__reduce_and_sync(0xffffffffu, common)) continue;
      bool apart = false;
#pragma unroll 1
      for (int c = 0; c < 32; ++c)
#pragma unroll
        for (int i = 0; i < TN / 32; ++i) {
          const uint32_t x = __shfl_sync(0xffffffffu, b[i], c);
#pragma unroll
          for (int j = 0; j < TM / 32; ++j) apart |= (a[j] & x) == 0;
        }
      if (__any_sync(0xffffffffu, apart) && lane == 0) atomicOr(&s_fine[d >> 5], 1u << (d & 31));
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tbase = tmem_base;
  const int row = 32 * (warp & 3) + lane, cb = 32 * (warp >> 2);   // this thread's TMEM lane and first column
  Share sh[2];   // of A's sixteen, then B's eight
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int it = warp + 12 * i;
    if (it < 16) sh[i].place(T.A + (long long)m0 * T.a_m, T.a_m, T.a_k, rowsA, it, lane);
    else sh[i].place(T.B + (long long)n0 * T.b_n, T.b_n, T.b_k, colsB, it - 16, lane);
  }
  const bool b1 = warp + 12 >= 16;   // the second share is B's (the first is A's)
  double acc[32], x[2][8];
#pragma unroll
  for (int c = 0; c < 32; ++c) acc[c] = 0.0;
  int st = 0;   // stages so far
  bool ok = true, first = true;
  for (int d = 0; d < R.per && ok; ++d) {
    const int e = ks * R.per + d, r0 = R.begin(e), r1 = R.end(e);
    if (r0 >= r1) break;
    const bool fine = nb > 1 && (d >= kFineRanges || (s_fine[d >> 5] >> (d & 31) & 1));
    for (int k0 = r0, k1; k0 < r1 && ok; k0 = k1) {
      k1 = fine ? min(k0 + SplitRanges::BLOCK, r1) : r1;
      const int *eA = X.wide(false) + (long long)e * T.M, *eB = X.wide(!T.same()) + (long long)e * T.N;
      if (fine) {
        const long long x = (long long)e * nb + (k0 - r0) / SplitRanges::BLOCK;
        eA = X.block(false, nb) + x * T.M;
        eB = X.block(!T.same(), nb) + x * T.N;
      }
      sh[0].E = sh[0].p ? eA[m0 + sh[0].row] : 1;
      sh[1].E = sh[1].p ? (b1 ? eB[n0 + sh[1].row] : eA[m0 + sh[1].row]) : 1;
      const int EA = row < rowsA ? eA[m0 + row] : 1;
      if (tid < TN) exB[tid] = tid < colsB ? eB[n0 + tid] : 1;   // read after a barrier below
#pragma unroll
      for (int i = 0; i < 2; ++i) sh[i].load(x[i], k0, k1);
      for (int k = k0; k < k1; k += KC, ++st) {
        unsigned char* Ap = buf + (st & 1) * STAGE;
        unsigned char* Bp = Ap + NDIG * A_PLANE;
        // the MMAs that read this buffer two stages ago are done
        if (st >= 2 && !wait_phase(smem_u32(&mbar[st & 1]), (uint32_t)((st >> 1) - 1) & 1)) atomicExch(&s_fail, 1);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          sh[i].store(x[i], i && b1 ? Bp : Ap, i && b1 ? B_PLANE : A_PLANE);
          sh[i].load(x[i], k + KC, k1);                        // the next stage's
        }
        asm volatile("fence.proxy.async.shared::cta;");        // generic-proxy writes -> tensor-core reads
        __syncthreads();
        if (s_fail) { ok = false; break; }
        if (tid == 0) {
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t a0 = smem_u32(Ap), b0 = smem_u32(Bp);
          for (int kk = 0; kk < KC / 16; ++kk)
            for (int j = 0; j < NDIG; ++j)                     // planes j of A, q .. q + nl - 1 of B: levels j + q on
              for (int q = 0; q < NDIG - j; q += 4) {
                const int nl = min(4, NDIG - j - q);
                const uint64_t da = smem_desc(a0 + j * A_PLANE + kk * 256);
                const uint64_t db = smem_desc(b0 + q * B_PLANE + kk * 256);
                const uint32_t accum = (k > k0 || kk > 0 || j > 0) ? 1u : 0u;
                const uint32_t idesc = kIdesc | (uint32_t)((nl * TN) >> 3) << 17;
                asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                             "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                             :: "r"(tbase + (uint32_t)((j + q) * TN)), "l"(da), "l"(db), "r"(idesc), "r"(accum));
              }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                       :: "r"(smem_u32(&mbar[st & 1])) : "memory");
        }
      }
      if (!ok) break;
      if (!wait_phase(smem_u32(&mbar[(st - 1) & 1]), (uint32_t)((st - 1) >> 1) & 1)) atomicExch(&s_fail, 1);
      __syncthreads();
      if (s_fail) { ok = false; break; }
      asm volatile("tcgen05.fence::after_thread_sync;");
      // sum = (hi 2^28 + lo) 2^(49 + EA + EB - 2154), the last 8 bits of lo dropped
      const uint32_t lane_addr = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)cb;
      if (warp < 8)
#pragma unroll
      for (int c0 = 0; c0 < 32; c0 += 8) {
        uint32_t v[NDIG][8];
#pragma unroll
        for (int g = 0; g < NDIG; ++g)
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                       : "=r"(v[g][0]), "=r"(v[g][1]), "=r"(v[g][2]), "=r"(v[g][3]), "=r"(v[g][4]), "=r"(v[g][5]),
                         "=r"(v[g][6]), "=r"(v[g][7])
                       : "r"(lane_addr + (uint32_t)(g * TN + c0)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          long long hi = 0, lo = 0;
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            hi = hi * 128 + __float2int_rn(__uint_as_float(v[g][c]));
            lo = lo * 128 + __float2int_rn(__uint_as_float(v[4 + g][c]));
          }
          const double val = scaled_int(hi * (1ll << 20) + (lo >> 8), EA + exB[cb + c0 + c] - 2097);
          acc[c0 + c] = first ? val : acc[c0 + c] + val;
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncthreads();   // TMEM and exB are reused by the next range
      asm volatile("tcgen05.fence::after_thread_sync;");
      first = false;
    }
  }
  if (!ok) {
    // an MMA group did not complete in time: wait (bounded) once more so no
    // write to TMEM is in flight when it is freed, flag the error
    if (tid == 0) {
      if (st > 0) wait_phase(smem_u32(&mbar[(st - 1) & 1]), (uint32_t)((st - 1) >> 1) & 1);
      atomicExch(err, 1);
    }
    __syncthreads();
  } else if (warp < 8 && row < rowsA && T.work) {
    // a partial sum over this CTA's range, reduced by k_split_reduce
    double* Wr = T.work + ((long long)ks * T.M + m0 + row) * T.N + n0;
#pragma unroll
    for (int c = 0; c < 32; ++c)
      if (cb + c < colsB) Wr[cb + c] = acc[c];
  } else if (warp < 8 && row < rowsA) {
    double* Cr = T.C + (long long)(m0 + row) * T.c_m + (long long)(n0 + cb) * T.c_n;
#pragma unroll
    for (int c = 0; c < 32; ++c)
      if (cb + c < colsB) {
        double v = T.alpha * acc[c];
        if (T.beta != 0.0) v = fma(T.beta, Cr[(long long)c * T.c_n], v);
        Cr[(long long)c * T.c_n] = v;
      }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tbase), "r"(TMEM_COLS));
}

// C = alpha sum_ks work[ks] + beta C for the tasks with partial sums, the
// K ranges added in a fixed order (results independent of scheduling); a
// symmetric C takes its upper triangle and mirrors it bitwise.
__global__ void k_split_reduce(const SplitTask* __restrict__ tasks) {
  const SplitTask T = tasks[blockIdx.y];
  if (!T.work) return;
  if (T.active && *T.active == 0) return;
  const long long mn = (long long)T.M * T.N;
  const int nks = max(T.ksplit, 1);
  for (long long it = blockIdx.x * (long long)blockDim.x + threadIdx.x; it < mn; it += (long long)gridDim.x * blockDim.x) {
    const int m = (int)(it / T.N), n = (int)(it % T.N);
    if (T.sym && m > n) continue;
    double s = 0.0;
#pragma unroll 8
    for (int ks = 0; ks < nks; ++ks) s += T.work[ks * mn + it];
    double* c = T.C + (long long)m * T.c_m + (long long)n * T.c_n;
    const double v = (T.beta != 0.0) ? fma(T.beta, *c, T.alpha * s) : T.alpha * s;
    *c = v;
    if (T.sym && m < n) T.C[(long long)n * T.c_m + (long long)m * T.c_n] = v;
  }
}

// The number of K ranges, at most `most`, that a product alone on sms SMs (a CTA each) should
// take: the fewest rounds of stages, a range's reading of TMEM counted as one. 216 x 216 x
// 16384, symmetric, at most 32 ranges: six tiles by 25 ranges fill one round, 32 take two
// with the second a quarter full, 119 against 137 us.
int split_ranges(const SplitTask& T, int most, int sms) {
  const int tm = (T.M + TM - 1) / TM, tn = (T.N + TN - 1) / TN;
  int tiles = 0, best = most;
  for (int i = 0; i < tm; ++i)
    for (int j = 0; j < tn; ++j) tiles += !(T.sym && (j + 1) * TN <= i * TM);
  double least = 0.0;
  for (int n = most; n >= 1; --n) {
    const SplitRanges R(T.K, n);
    const double rounds = (double)(((long long)tiles * n + sms - 1) / sms), cost = rounds * (2.0 * R.cps + R.per);
    if (n == most || cost < least) { least = cost; best = n; }
  }
  return best;
}

void launch_split_gemm(const SplitTask* tasks, int ntask, int max_m, int max_n, int* err, cudaStream_t st,
                       int max_ks, bool reduce) {
  if (!ntask || max_m <= 0 || max_n <= 0) return;
  FOCK_SMEM_OPTIN(k_split_gemm);
  max_ks = max_ks < 1 ? 1 : max_ks;
  k_split_exps<<<dim3(ntask < 4 ? 304 : 76, ntask), 256, 0, st>>>(tasks);
  dim3 grid((max_n + TN - 1) / TN, (max_m + TM - 1) / TM, ntask * max_ks);
  k_split_gemm<<<grid, kSplitThreads, SPLIT_SMEM, st>>>(tasks, max_ks, err);
  if (reduce) k_split_reduce<<<dim3(152, ntask), 256, 0, st>>>(tasks);
}

}  // namespace fock
