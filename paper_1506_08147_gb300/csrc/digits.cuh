// FP64 products on the tensor cores by exact digit splitting (the error-free
// splitting of Ozaki et al., Numer. Algorithms 59, 2012, in the
// integer-digit form used for tensor cores).
//
// Every operand row (the vector that runs along the contraction index K) gets
// one exponent e, that of its largest entry (at least 64), and every entry x becomes the
// integer X = trunc(x 2^(1076 - e)), |X| < 2^54 (e the biased exponent), cut into
// seven balanced base-256 digits d_0 .. d_6 in [-128, 127], which FP16 holds
// exactly.  X Y = sum over i, j of d_i d_j 256^(12 - i - j); the 28 digit products
// with i + j <= 6 are formed by tcgen05.mma kind::f16.  All products of one
// order s = i + j accumulate in the same tensor-memory block: seven blocks,
// and since the digits of the B operand are stacked along N, one instruction
// (two where N > 256) takes digit i of A against digits 0 .. 6 - i of B and
// lands on blocks i .. 6.  |d_i d_j| <= 2^14 and at most 7 products of an order
// over 128 values of K stay below 2^24, so every FP32 sum is an exact integer.
// The seven sums are joined in integer arithmetic.  The result is exact but
// for the digits beyond 2^-54 of a row's largest entry and the dropped orders
// i + j >= 7 (below 2^-55 of the product of the largest entries).
//
// Why: this part's FP64 pipe does 1.2 TFLOP/s; the tensor cores do the 28
// products of a multiply-add at 1850 / 28 = 66 TFLOP/s.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "common.cuh"
#include "tcgen05.cuh"

namespace dgdft {

namespace {

constexpr int DIG = 7;                        // digits of an operand
constexpr int DIG_M = 128;                    // rows of A
constexpr int DIG_K = 64;                     // K values per stage: one 128-byte swizzle row of FP16
constexpr int DIG_WINDOW = 2;                 // stages per exact accumulation (128 values)
constexpr int DIG_A_BYTES = DIG_M * DIG_K * 2;  // one digit of A
constexpr int DIG_THREADS = 512;
constexpr int DIG_ISSUER = DIG_THREADS - 32;  // the thread that issues the products
constexpr uint32_t DIG_POLLS = 1u << 22;

__device__ __forceinline__ int dig_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// x 2^s (zero where that is subnormal; infinities and NaN stay)
__device__ __forceinline__ double dig_scale(double x, int s) {
  const int h = __double2hiint(x), ex = (h >> 20) & 0x7ff, ne = ex + s;
  if (ex == 0x7ff) return x;
  if (ex == 0 || ne <= 0) return 0.0;
  if (ne >= 0x7ff) return __hiloint2double((h & 0x80000000) | 0x7ff00000, 0);
  return __hiloint2double(h + s * (1 << 20), __double2loint(x));
}

constexpr uint32_t DIG_BIAS_HI = 0x64808080u, DIG_BIAS_LO = 0x80808080u;

// The digits of eight entries from their magnitudes m < 2^54 (as lo, hi with
// DIG_BIAS added: the digits are then bytes less 128) and words whose top bits
// are the signs, as seven 16-byte groups of FP16.  The free eighth byte of the
// biased integer is 0x64, so that one byte permutation makes the FP16 values
// 1024 + byte of two entries, and one multiply-add the signed digits: integer
// instructions (64 lanes a cycle and SM) are what a split costs.
__device__ __forceinline__ void dig_bytes8(const uint32_t (&lo)[8], const uint32_t (&hi)[8], const uint32_t (&sg)[8],
                                           uint4 (&q)[DIG]) {
  uint32_t r[DIG][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const uint32_t ha = hi[2 * p], hb = hi[2 * p + 1], la = lo[2 * p], lb = lo[2 * p + 1];
    const uint32_t ma = __byte_perm(la, 0x64u, 0x4321), mb = __byte_perm(lb, 0x64u, 0x4321);
    const uint32_t o = (__byte_perm(sg[2 * p], sg[2 * p + 1], 0x7632) & 0x80008000u) | 0x3c003c00u;  // +-1
    const __half2 one = *reinterpret_cast<const __half2*>(&o);
    const __half2 off = __hmul2(one, __floats2half2_rn(-1152.0f, -1152.0f));  // -+(1024 + 128)
    auto put = [&](int i, uint32_t w) {
      const __half2 d = __hfma2(*reinterpret_cast<const __half2*>(&w), one, off);
      r[i][p] = *reinterpret_cast<const uint32_t*>(&d);
    };
    put(0, __byte_perm(ha, hb, 0x7632));
    put(1, __byte_perm(ha, hb, 0x7531));
    put(2, __byte_perm(ha, hb, 0x7430));
    put(3, __byte_perm(ma, mb, 0x7632));
    put(4, __byte_perm(ma, mb, 0x7531));
    put(5, __byte_perm(ma, mb, 0x7430));
    put(6, (__byte_perm(la, lb, 0x4400) & 0x00ff00ffu) | 0x64006400u);
  }
#pragma unroll
  for (int i = 0; i < DIG; ++i) q[i] = make_uint4(r[i][0], r[i][1], r[i][2], r[i][3]);
}

__device__ __forceinline__ void dig_biased(unsigned long long m, uint32_t& lo, uint32_t& hi) {
  m += ((unsigned long long)DIG_BIAS_HI << 32) | DIG_BIAS_LO;
  lo = (uint32_t)m;
  hi = (uint32_t)(m >> 32);
}

// The digits of eight entries of a row with exponent e >= 64 (a zero's or a
// subnormal's shift is then 63 and leaves nothing).
__device__ __forceinline__ void dig_split8(const double (&x)[8], int e, uint4 (&q)[DIG]) {
  uint32_t lo[8], hi[8], sg[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const uint32_t h = (uint32_t)__double2hiint(x[u]), l = (uint32_t)__double2loint(x[u]);
    const int sh = min(e - (int)((h >> 20) & 0x7ff), 63);
    sg[u] = h;
    dig_biased((((unsigned long long)((h & 0xfffffu) | 0x100000u) << 33) | ((unsigned long long)l << 1)) >> sh, lo[u], hi[u]);
  }
  dig_bytes8(lo, hi, sg, q);
}

// Eight digits where a sum has few terms, so that seven's dropped orders (rms
// 2^-53 of the largest product a term) would show: X = x 2^(1084 - e), |X| < 2^62,
// the 36 products with i + j <= 7; the result is exact to 2^-60 of the product of
// the largest entries, and entries above 2^-9 of them keep all their bits.
constexpr int DIG8 = 8;

// Eight digits of eight entries, entry u standing for x[u] 2^s[u] (e at least
// their exponents).
__device__ __forceinline__ void dig8_split8s(const double (&x)[8], const int (&s)[8], int e, uint4 (&q)[DIG8]) {
  uint32_t r[DIG8][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    uint32_t lo[2], hi[2], sg[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int u = 2 * p + c;
      const uint32_t h = (uint32_t)__double2hiint(x[u]), l = (uint32_t)__double2loint(x[u]);
      const int ex = (h >> 20) & 0x7ff;
      const int sh = ex == 0 ? 63 : max(min(e - ex - s[u], 63), 0);
      unsigned long long m = ((unsigned long long)((h & 0xfffffu) | 0x100000u) << 41) | ((unsigned long long)l << 9);
      m = (m >> sh) + 0x8080808080808080ull;
      sg[c] = h;
      lo[c] = (uint32_t)m;
      hi[c] = (uint32_t)(m >> 32);
    }
    const uint32_t o = (__byte_perm(sg[0], sg[1], 0x7632) & 0x80008000u) | 0x3c003c00u;  // +-1
    const __half2 one = *reinterpret_cast<const __half2*>(&o);
    const __half2 off = __hmul2(one, __floats2half2_rn(-1152.0f, -1152.0f));
    auto put = [&](int i, uint32_t w) {
      const __half2 d = __hfma2(*reinterpret_cast<const __half2*>(&w), one, off);
      r[i][p] = *reinterpret_cast<const uint32_t*>(&d);
    };
    auto word = [&](int i, uint32_t a, uint32_t b) {  // four digits of a 32-bit half
      const uint32_t ma = __byte_perm(a, 0x64u, 0x4321), mb = __byte_perm(b, 0x64u, 0x4321);
      put(i, __byte_perm(ma, mb, 0x7632));
      put(i + 1, __byte_perm(ma, mb, 0x7531));
      put(i + 2, __byte_perm(ma, mb, 0x7430));
      put(i + 3, (__byte_perm(a, b, 0x4400) & 0x00ff00ffu) | 0x64006400u);
    };
    word(0, hi[0], hi[1]);
    word(4, lo[0], lo[1]);
  }
#pragma unroll
  for (int i = 0; i < DIG8; ++i) q[i] = make_uint4(r[i][0], r[i][1], r[i][2], r[i][3]);
}

// A weight: its mantissa left-aligned, the leading bit (always 1) replaced by
// the sign, and its exponent; a zero's (or a subnormal's) is far below any entry's
struct DigWeight {
  uint32_t hi, lo;
  int ex;
};
__device__ __forceinline__ DigWeight dig_weight(double w) {
  const uint32_t h = (uint32_t)__double2hiint(w), l = (uint32_t)__double2loint(w);
  DigWeight r;
  const int ex = (h >> 20) & 0x7ff;
  r.hi = (h & 0x80000000u) | ((h & 0xfffffu) << 11) | (l >> 21);
  r.lo = l << 11;
  r.ex = ex ? ex : -8192;
  return r;
}

// The digits of x w for eight entries and their weights; e at least the sum of
// the exponents less 1022 and 64.  The product is formed from the integer
// mantissas (61 leading bits): an FP64 multiply would hold its sub-partition
// 64 cycles.
__device__ __forceinline__ void dig_split8w(const double (&x)[8], const DigWeight* w, int wstep, int e, uint4 (&q)[DIG]) {
  uint32_t lo[8], hi[8], sg[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const uint32_t h = (uint32_t)__double2hiint(x[u]), l = (uint32_t)__double2loint(x[u]);
    const uint32_t xh = 0x80000000u | (((h << 11) | (l >> 21)) & 0x7fffffffu), xl = l << 11;
    const DigWeight b = w[u * wstep];
    const int ex = (h >> 20) & 0x7ff;
    const uint32_t wh = b.hi | 0x80000000u;
    unsigned long long m = (unsigned long long)xh * wh + __umulhi(xh, b.lo) + __umulhi(xl, wh);
    const int sh = max(min(e + 1032 - ex - b.ex, 63), 0);
    sg[u] = h ^ b.hi;
    dig_biased(ex ? m >> sh : 0ull, lo[u], hi[u]);
  }
  dig_bytes8(lo, hi, sg, q);
}

// byte offset of 16-byte group c (eight K values) of a row in a K-major
// 128-byte-swizzled operand tile
__device__ __forceinline__ uint32_t dig_off(int row, int c) { return (uint32_t)(row * 128 + ((c ^ (row & 7)) << 4)); }

// kind::f16 instruction descriptor: D = F32, A = B = F16, both K-major
__device__ __forceinline__ uint32_t dig_idesc(int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(DIG_M >> 4) << 24);
}
__device__ __forceinline__ void dig_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n"
      " .reg .pred p;\n"
      " setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
      "}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// The products of one stage: nk16 groups of 16 K values; A: D digit tiles,
// `astep` bytes apart, of 128 rows (those beyond the rows in use may hold
// anything: their accumulators are not read), B: D of NB rows one after
// another.  first: the accumulators start at zero.  One thread.
template <int NB, int D>
__device__ __forceinline__ void dig_issue(uint32_t tmem, uint32_t a, uint32_t astep, uint32_t b, int nk16, bool first) {
  constexpr int PER = 256 / NB;  // digit blocks an instruction can take
  // the address field (16-byte units) is the only one that changes
  const uint64_t da0 = sw128_desc(a), db0 = sw128_desc(b);
  const uint32_t dhi_a = (uint32_t)(da0 >> 32), dhi_b = (uint32_t)(db0 >> 32);
  uint32_t la = (uint32_t)da0, lb = (uint32_t)db0;
  const uint32_t as = astep >> 4;
  uint32_t acc = first ? 0u : 1u;
  for (int ks = 0; ks < nk16; ++ks) {
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const uint64_t da = ((uint64_t)dhi_a << 32) | (la + i * as);
#pragma unroll
      for (int j = 0; j < D - i; j += PER) {
        const int nb = (D - i - j) < PER ? D - i - j : PER;
        const uint64_t db = ((uint64_t)dhi_b << 32) | (lb + j * (NB * 8));
        dig_mma(tmem + (i + j) * NB, da, db, dig_idesc(nb * NB), i == 0 ? acc : 1u);
      }
    }
    la += 2;
    lb += 2;
    acc = 1u;
  }
}

// The order sums of four neighbouring columns for this thread's lane
// (tensor-memory row).
template <int NB, int D>
__device__ __forceinline__ void dig_sums4(uint32_t taddr, int (&a)[4][D]) {
  uint32_t r[D][4];
#pragma unroll
  for (int s = 0; s < D; ++s)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[s][0]), "=r"(r[s][1]), "=r"(r[s][2]), "=r"(r[s][3])
                 : "r"(taddr + s * NB));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int s = 0; s < D; ++s) a[c][s] = __float2int_rn(__uint_as_float(r[s][c]));
}

// Joined exactly: value = hi 2^32 + lo in units of 256^6 of the integer product.
template <int NB>
__device__ __forceinline__ void dig_drain4(uint32_t taddr, long long (&hi)[4], long long (&lo)[4]) {
  int a[4][DIG];
  dig_sums4<NB, DIG>(taddr, a);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    hi[c] = (long long)a[c][0] * 65536 + (a[c][1] * 256 + a[c][2]);
    lo[c] = (long long)a[c][3] * 16777216 + ((long long)a[c][4] * 65536 + ((long long)a[c][5] * 256 + a[c][6]));
  }
}

// The same of eight digits, in units of 256^7.
template <int NB>
__device__ __forceinline__ void dig8_drain4(uint32_t taddr, long long (&hi)[4], long long (&lo)[4]) {
  int a[4][DIG8];
  dig_sums4<NB, DIG8>(taddr, a);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    hi[c] = (long long)a[c][0] * 16777216 + ((long long)a[c][1] * 65536 + ((long long)a[c][2] * 256 + a[c][3]));
    lo[c] = (long long)a[c][4] * 16777216 + ((long long)a[c][5] * 65536 + ((long long)a[c][6] * 256 + a[c][7]));
  }
}

// Joined to 63 bits (units of 2^5 256^6; what is cut off lies 2^-55 below the
// product of the rows' largest entries): the leading sum, of products of two
// leading digits in [-64, 64], is at most 2^19, the others 2^24.
template <int NB>
__device__ __forceinline__ void dig_join4(uint32_t taddr, long long (&t)[4]) {
  int a[4][DIG];
  dig_sums4<NB, DIG>(taddr, a);
#pragma unroll
  for (int c = 0; c < 4; ++c)
    t[c] = ((long long)(a[c][0] * 256 + a[c][1]) << 35) + (long long)a[c][2] * (1 << 27) + (long long)a[c][3] * (1 << 19) +
           (long long)a[c][4] * (1 << 11) + (a[c][5] * 8 + (a[c][6] >> 5));
}

// a row's exponent for dig_value: far above all others where the row held an
// infinity or a NaN
__device__ __forceinline__ int dig_row_exp(int e) { return e >= 0x7ff ? 1 << 20 : e; }

// t 2^(e + f - 2099) rounded to FP64, by integer operations (FP64 ones would
// cost more than the products); |t| < 2^63.  NaN where a row held an infinity
// or a NaN.
__device__ __forceinline__ double dig_value(long long t, int e, int f) {
  const uint32_t s = (uint32_t)(t >> 63);
  unsigned long long m = (unsigned long long)(t < 0 ? -t : t);
  const int lz = __clzll((long long)m);
  m = ((m << (lz & 63)) >> 1) + 512ull;
  const int ex = e + f - lz - (m == 512ull ? 10000 : 1013);
  uint32_t hi = (uint32_t)(m >> 42), lo = (uint32_t)(m >> 10);
  hi += (uint32_t)(ex - 1) << 20;
  if ((uint32_t)(ex - 1) >= 0x7feu) {  // zero, underflow, overflow, not a number
    lo = 0u;
    hi = ex <= 0 ? 0u : ex > (1 << 18) ? 0x7ff80000u : 0x7ff00000u;
  }
  return __hiloint2double((int)(hi | (s & 0x80000000u)), (int)lo);
}

// The same for D digits' sums over several windows (|hi| < 2^62, |lo| < 2^63), in
// FP64.
template <int D>
__device__ __forceinline__ double dig_value_sum(long long hi, long long lo, int e, int f) {
  if (e >= 0x7ff || f >= 0x7ff) return __longlong_as_double(0x7ff8000000000000LL);
  return scalbn((double)hi * 4294967296.0 + (double)lo, e + f - (D == DIG8 ? 2112 : 2104));
}

// Eight digits' sums over at most 1,024 values (below 2^78 units), by integer
// operations; e and f as dig_value takes them.  The 63 leading bits are kept
// wherever they lie (the 63 at fixed places would cut results well below the
// largest product short).
__device__ __forceinline__ double dig8_value_sum(long long hi, long long lo, int e, int f) {
  hi += lo >> 32;
  const int sh = min(__clzll(hi ^ (hi >> 63)) - 1, 32);  // at least 16
  const unsigned long long t = ((unsigned long long)hi << sh) | ((unsigned long long)(uint32_t)lo >> (32 - sh));
  return dig_value((long long)t, e + 19 - sh, f);
}

// Tensor memory and the completion barrier of a CTA.  All threads call; every
// wait is bounded.
struct DigCta {
  uint32_t tmem;
  uint64_t* bar;
  uint32_t phase;
};
__device__ __forceinline__ void dig_open(DigCta& c, uint64_t* bar, uint32_t* slot) {  // bar[2]
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    mbar_init(bar + 1, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  c.tmem = *slot;
  c.bar = bar;
  c.phase = 0;
}
// aborted: a wait ran out; the products still in flight are waited for (again
// with a limit, through a barrier of its own) before tensor memory is freed
__device__ __forceinline__ void dig_close(const DigCta& c, uint64_t* last, bool aborted) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (aborted && threadIdx.x == DIG_ISSUER) {
    mma_commit(last);
    mbar_wait(last, 0, DIG_POLLS);
  }
  __syncthreads();
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(c.tmem), "r"(512) : "memory");
}
// operands written with ordinary stores become visible to the tensor core
__device__ __forceinline__ void dig_publish() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
}
template <int NB, int D = DIG>
__device__ __forceinline__ void dig_launch(const DigCta& c, uint32_t a, uint32_t astep, uint32_t b, int nk16, bool first) {
  if (threadIdx.x == DIG_ISSUER) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    dig_issue<NB, D>(c.tmem, a, astep, b, nk16, first);
    mma_commit(c.bar);
  }
}
// the launched products are done, or the bounded wait ran out: then *abort is
// set and every later wait of the block is a single poll
__device__ __forceinline__ void dig_wait(DigCta& c, int* abort) {
  if (!mbar_wait(c.bar, c.phase, *reinterpret_cast<volatile int*>(abort) ? 1u : DIG_POLLS)) atomicOr(abort, 1);
  c.phase ^= 1;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// columns of B per chunk: a multiple of 16, at most 64 (seven blocks of
// accumulators in tensor memory), the chunks as even as can be
inline int chunk_cols(int n) {
  const int c = (n + 63) / 64;
  return ((n + c - 1) / c + 15) / 16 * 16;
}

// dynamic shared memory a CTA can have beside 3 KB of static
constexpr size_t DIG_SMEM_MAX = 232448 - 3200;

inline int sm_count() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n;
}

template <class K> void dig_opt_in(K k, size_t smem) {
  cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

}  // namespace

}  // namespace dgdft
