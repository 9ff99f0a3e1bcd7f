// Sliced FP64 products on tcgen05 (see oz_gemm.h).
//
// One CTA owns a 128 x NT (real columns) tile of C over spc K segments.
// Sixteen worker warps read the segment twice: once for the row exponents,
// once to convert it, 16 complex k at a time, into digit tiles in shared
// memory (64-byte-swizzled rows, one tile per digit, two stages).  The
// second read comes from L2.  One warp issues the MMAs: digit i of A against
// the stacked digits 0..7-i of B, whose result columns are the accumulators
// i..7 (columns [g NT, (g+1) NT) of tensor memory hold the sum of the
// products i + j = g).  The workers then read the eight accumulators back,
// join them in integer arithmetic and round once to a double.
//
// No FP64 instruction is used on the way to a first result: conversion and
// joining are integer work, because an SM has 64 times fewer FP64 lanes than
// integer ones.  FP64 sums again what fixed point cannot hold as accurately
// (settle).  The code is kept small (rolled loops): fetched once per tile,
// 85 KB of straight-line code took longer than the work.  Bound by the
// integer work and load latencies (3800 x 14440 x 48: 52000 warp instructions
// and 31000 clocks per tile, of which the MMAs take 7000; 17.6 ms on the FP64
// cores, 1.49 ms here, 0.13 of them for the test that settle() needs).
#include "oz_gemm.h"

#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "tc_ptx.h"

namespace rtcc3 {

namespace {

constexpr int kSl = 8;              // digits
constexpr int kRows = 128;          // A rows per tile
constexpr int kKC = 16;             // complex k per stage (64-byte FP16 rows)
constexpr int kWorkers = 16;        // worker warps
constexpr int kSegMax = 128;        // complex k per segment (256 real: see oz_gemm.h; a power of two)

constexpr int kWPitch = 48;         // bytes between the weights of two rows (32 each, no bank conflicts)

template <int NT>
struct OzSmem {
  static constexpr int kASlice = kRows * 64, kBSlice = NT * 64;
  static constexpr int kStage = kSl * (kASlice + kBSlice);
  static constexpr int kPitch = NT / 2 + 1;  // complex per staged output row
  static constexpr int kBarOff = 2 * kStage;
  static constexpr int kExpOff = kBarOff + 64;  // row exponents, two segments
  static constexpr int kTabOff = kExpOff + 2 * (kRows + 32) * 4;  // k offsets (two segments), output offsets
  static constexpr int kWOff = kTabOff + (4 * kSegMax + kRows + NT / 2) * 8;  // weights of the rows' elements
  static constexpr int kRowOff = kWOff + (kRows + 32) * kWPitch;  // offsets of the rows
  static constexpr int kTotal = kRowOff + (kRows + 32) * 8 + 1024;
  static constexpr int kCols = NT <= 16 ? 128 : (NT <= 32 ? 256 : 512);  // TMEM columns (a power of two)
  static_assert(kRows * kPitch * 16 <= 2 * kStage, "output staging");
  static_assert(kTotal <= 232448, "shared memory per CTA");
};

// Shared-memory descriptor: K-major, 64-byte swizzle, 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t desc64(uint32_t addr) {
  return uint64_t((addr >> 4) & 0x3FFF) | (uint64_t(1) << 16) | (uint64_t(512 >> 4) << 32) |
         (uint64_t(1) << 46) | (uint64_t(4) << 61);
}

// FP16 x FP16 -> FP32, both K-major.
__host__ __device__ constexpr uint32_t idesc_f16(int N) {
  return (1u << 4) | (uint32_t(N >> 3) << 17) | (uint32_t(kRows >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tmem_ld(uint32_t t, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(t));
}

// |x| as a sortable word whose top 11 bits are its exponent field.
__device__ __forceinline__ uint32_t hiabs(uint32_t hi) { return hi & 0x7fffffffu; }

// |a| (below 2^(F - 1022), F >= 64) as the biased digits of its 62-bit
// fixed-point form, rounded to nearest: byte 7 - s is digit s of |a| plus 128.
// Elements below 2^-63 of the bound (zeros and subnormals among them) have zero
// digits.  The bias of the lower digits and the rounding are added one bit
// further left; the shift back brings in the first digit's bias.
__device__ __forceinline__ void digits(double a, int F, uint32_t& yh, uint32_t& yl) {
  const uint32_t hi = uint32_t(__double2hiint(a)), lo = uint32_t(__double2loint(a));
  const int n = min(F - int(hiabs(hi) >> 20), 63);
  const unsigned long long m =
      (static_cast<unsigned long long>((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  const unsigned long long t = ((m << 10) >> n) + 0x0101010101010101ULL;
  yh = __funnelshift_r(uint32_t(t >> 32), 1u, 1);
  yl = __funnelshift_r(uint32_t(t), uint32_t(t >> 32), 1);
}

// The eight digits of a complex number as pairs of halves (re, im), signs
// applied: u has the bits 0x6400 | byte = 1024 + byte, so one FMA by (+-1, +-1)
// with the addend -+1152 gives the digit.
struct DigitPairs {
  uint32_t q[4];  // interleaved bytes (re_s, im_s, re_s+1, im_s+1), s = 0, 2, 4, 6
  __half2 sg, c;
  __device__ __forceinline__ DigitPairs(double2 z, int F) {
    uint32_t rh, rl, ih, il;
    digits(z.x, F, rh, rl);
    digits(z.y, F, ih, il);
    q[0] = __byte_perm(rh, ih, 0x6273);  // bytes 3, 7, 2, 6 from low to high
    q[1] = __byte_perm(rh, ih, 0x4051);
    q[2] = __byte_perm(rl, il, 0x6273);
    q[3] = __byte_perm(rl, il, 0x4051);
    const uint32_t sr = uint32_t(__double2hiint(z.x)), si = uint32_t(__double2hiint(z.y));
    const uint32_t w = (__byte_perm(sr, si, 0x7030) & 0x80008000u) | 0x3c003c00u;
    sg = *reinterpret_cast<const __half2*>(&w);
    c = __hmul2(sg, __half2(__ushort_as_half(0xe480), __ushort_as_half(0xe480)));  // -1152
  }
  template <int S>
  __device__ __forceinline__ uint32_t get() const {
    const uint32_t u = __byte_perm(q[S >> 1], 0x64u, (S & 1) ? 0x4342 : 0x4140);
    const __half2 h = __hfma2(*reinterpret_cast<const __half2*>(&u), sg, c);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
};

__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

template <int S, int STRIDE>
__device__ __forceinline__ void store_a(uint32_t addr, const DigitPairs& d) {
  if constexpr (S < kSl) {
    sts32(addr + S * STRIDE, d.template get<S>());
    store_a<S + 1, STRIDE>(addr, d);
  }
}

// One row of B's embedding: (re, -im) at row 2n (odd = false), (im, re) at row
// 2n + 1.
struct RowPairs {
  uint32_t sel0, sel1;  // byte selectors of the even and odd digits
  __half2 sg, c;
  __device__ __forceinline__ RowPairs(const DigitPairs& d, bool odd) {
    sel0 = odd ? 0x4041 : 0x4140;
    sel1 = odd ? 0x4243 : 0x4342;
    const uint32_t w = *reinterpret_cast<const uint32_t*>(&d.sg);
    const uint32_t x = odd ? __byte_perm(w, w, 0x1032) : w ^ 0x80000000u;
    sg = *reinterpret_cast<const __half2*>(&x);
    c = __hmul2(sg, __half2(__ushort_as_half(0xe480), __ushort_as_half(0xe480)));
  }
};

template <int S, int STRIDE>
__device__ __forceinline__ void store_b(uint32_t addr, const DigitPairs& d, const RowPairs& r) {
  if constexpr (S < kSl) {
    const uint32_t u = __byte_perm(d.q[S >> 1], 0x64u, (S & 1) ? r.sel1 : r.sel0);
    const __half2 h = __hfma2(*reinterpret_cast<const __half2*>(&u), r.sg, r.c);
    sts32(addr + S * STRIDE, *reinterpret_cast<const uint32_t*>(&h));
    store_b<S + 1, STRIDE>(addr, d, r);
  }
}

constexpr int kZeroExp = 1 << 16;  // row exponent that makes every digit zero
constexpr int kNanExp = 1 << 18;  // exponent of a row with a non-finite element
constexpr int kNullRow = -(1 << 16);  // exponent of a row of zeros (E below half of it: the sum is 0)

__device__ __forceinline__ double join_rare(uint32_t w2, uint32_t w1, uint32_t w0, int e, uint32_t sign) {
  if (e >= kNanExp / 2) return __longlong_as_double(0x7ff8000000000000LL);
  if (w2 == 0) { w2 = w1; w1 = w0; w0 = 0; e -= 32; }
  if (w2 == 0) { w2 = w1; w1 = w0; w0 = 0; e -= 32; }
  if (w2 == 0) return 0.0;
  const int lz = __clz(w2);
  const unsigned long long top =
      (static_cast<unsigned long long>(__funnelshift_l(w1, w2, lz)) << 32) | __funnelshift_l(w0, w1, lz);
  const unsigned long long t = (top >> 11) + ((top >> 10) & 1ULL);
  const int field = e - lz + 63 + 1023;
  unsigned long long bits = 0ULL;  // below the normal range: zero
  if (field > 0) bits = (static_cast<unsigned long long>(field - 1) << 52) + t;
  if (field >= 2047 || bits > 0x7ff0000000000000ULL) bits = 0x7ff0000000000000ULL;
  return __longlong_as_double((long long)(bits | (static_cast<unsigned long long>(sign & 0x80000000u) << 32)));
}

// (hi 2^32 + lo) 2^16 as sign (all ones or 0) and 96-bit magnitude w2:w1:w0
// (|hi| < 2^47).
__device__ __forceinline__ uint32_t magnitude(long long hi, long long lo, uint32_t& w2, uint32_t& w1,
                                              uint32_t& w0) {
  hi += int(lo >> 32);
  const uint32_t s = uint32_t(hi >> 63);
  const uint32_t h1 = uint32_t(static_cast<unsigned long long>(hi) >> 32), h0 = uint32_t(hi), l = uint32_t(lo);
  w2 = __byte_perm(h0, h1, 0x5432) ^ s;
  w1 = __byte_perm(l, h0, 0x5432) ^ s;
  w0 = (l << 16) ^ s;
  asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %3;\n\tsubc.u32 %2, %2, %3;"
      : "+r"(w0), "+r"(w1), "+r"(w2)
      : "r"(s));
  return s;
}

// join() of any accumulators: above 2^22, zero sums, results outside the
// normal range, rows with a non-finite element (NaN).  The sums i + j >= 5 are
// not exact beyond 2^24; that needs digits of nearly the largest size and one
// sign in four fifths of all terms, which leave more than 0.6 2^24 at the end:
// NaN too.
__device__ __noinline__ double join_any(float v0, float v1, float v2, float v3, float v4, float v5,
                                        float v6, float v7, int E, uint32_t sgn) {
  if (fmaxf(fmaxf(fabsf(v5), fabsf(v6)), fabsf(v7)) >= 10066329.0f)
    return __longlong_as_double(0x7ff8000000000000LL);
  auto iv = [](float v) { return (long long)__float2int_rn(v); };
  uint32_t w2, w1, w0;
  const uint32_t s = magnitude((iv(v0) << 24) + (iv(v1) << 16) + (iv(v2) << 8) + iv(v3),
                               (iv(v4) << 24) + (iv(v5) << 16) + (iv(v6) << 8) + iv(v7), w2, w1, w0);
  return join_rare(w2, w1, w0, E + 16, s ^ sgn);
}

// sum_g v_g 2^(56 - 8 g) 2^E, the v_g integers held in FP32, rounded to
// nearest; sgn: all ones for the negative.  Integers up to 2^22 (nearly all; v0
// and v1 always) leave FP32 by an addition that puts them into the mantissa:
// the conversion instruction has an eighth of that rate.
__device__ __forceinline__ double join(const float (&v)[kSl], int E, uint32_t sgn) {
  const float big = fmaxf(fmaxf(fmaxf(fabsf(v[2]), fabsf(v[3])), fabsf(v[4])),
                          fmaxf(fmaxf(fabsf(v[5]), fabsf(v[6])), fabsf(v[7])));
  // pairs v_g 256 + v_(g+1): below 2^31
  auto two = [&](int g) {
    const uint32_t p = __float_as_uint(v[g] + 12582912.0f), q = __float_as_uint(v[g + 1] + 12582912.0f);
    return int(p * 256u + q - 0x4b400000u * 257u);
  };
  uint32_t w2, w1, w0;
  const uint32_t sign = magnitude((long long)two(0) * 65536 + two(2), (long long)two(4) * 65536 + two(6),
                                  w2, w1, w0) ^ sgn;
  const int lz = __clz(w2);
  const uint32_t th = __funnelshift_l(w1, w2, lz), tl = __funnelshift_l(w0, w1, lz);
  const int field = E - lz + 16 + 63 + 1023;
  if (big > 4194304.0f || w2 == 0 || unsigned(field - 1) >= 2045u)
    return join_any(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], E, sgn);
  // 53 bits of th:tl (top bit set), rounded; the carry runs into the exponent
  unsigned long long t = ((static_cast<unsigned long long>(th) << 32) | tl) >> 11;
  t += (tl >> 10) & 1u;
  t += static_cast<unsigned long long>(uint32_t(field - 1) << 20 | (sign & 0x80000000u)) << 32;
  return __longlong_as_double((long long)t);
}

constexpr int kMinExp = 64;  // smallest row exponent (2^-958): digits() needs it

// Larger of |re| and |im| of a row element, as its high word.
__device__ __forceinline__ uint32_t row_word(const double2* p) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(p);
  return max(hiabs(__ldg(w + 1)), hiabs(__ldg(w + 3)));
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

struct OzArgs {
  const double2 *A, *B;
  const long long *aM, *aK, *bN, *bK, *cM, *cN;
  double2* C;      // already moved by its offset
  double2* part;   // running sums over a CTA's segments, [split][n][m] (nseg > 1)
  int M, N, K;
  unsigned zrow, zspc;  // row blocks and segments a step of blockIdx.z stands for (one is 0)
  int seg, nseg, spc;
  int ash;         // alpha = (neg ? -1 : 1) 2^ash alpha_rest, neg = all ones or 0
  uint32_t neg;
  double alpha_rest, alpha_joined;  // alpha_joined = (neg ? -1 : 1) 2^ash
  int accumulate, splits, c_m;
  int* err;
  long long budget;
};

// Fixed point holds an element to a fraction of its row's largest, so a sum all
// of whose terms are small beside the product of the two rows' largest elements
// (rows graded in opposite directions, a row of the identity) would lose digits
// that FP64 arithmetic keeps.  With |a| <= 2^A, |b| <= 2^B and K complex terms a
// joined sum is off by at most 2 K (1 + 7.02) 2^-62 2^(A + B) in its real and
// imaginary parts (two roundings of half a unit of 2^-62, the products i + j >= 8
// left out), FP64 arithmetic by up to 2 K 2^-53 s, s = sum |a||b|.  So a sum is as
// accurate as that if s >= 2^-6 2^(A + B).  It is if the result has that size, or
// if the first 32 terms add up to it by their elements' weights (each 2^-16
// 2^(A + B) times the two weights); in dense products less than one in a thousand
// has neither.  Every other output is summed again here in FP64, and so are those
// whose rows have infinities or NaN, whose digit sums were not exact or whose
// scale is so small that a component below the normal range counts: they come
// out as they do in FP64 arithmetic.
constexpr int kSoundField = 1085;           // exponent field of 2^-6 2^(A + B) less E
constexpr uint32_t kSoundWeight = 1u << 10;  // the same in products of weights

// Bit j of todo: output z[j stride] of this lane's row lacks this segment's sum.
// Four outputs at a time, eight lanes each; bound by the FP64 pipe where many are
// left (8112 x 52 x 52 with a near-identity matrix, a tenth of its outputs: 28 us
// without, 79 with), by one round's latency where a few are.
__device__ __forceinline__ void settle(const OzArgs& P, uint32_t todo, double2* z, long long stride,
                                       const long long* am, const long long* bn, const long long* tk, int klen) {
  const int lane = threadIdx.x & 31, g = lane >> 3;
#pragma unroll 1
  while (const uint32_t lanes = __ballot_sync(0xffffffffu, todo != 0)) {
    uint32_t t = lanes;
    int r = -1;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (u == g) r = __ffs(t) - 1;
      t &= t - 1;
    }
    const int mine = __ffs(todo) - 1, j = __shfl_sync(0xffffffffu, mine, r & 31);
    double sr = 0.0, si = 0.0;
    if (r >= 0) {
      const char* pa = reinterpret_cast<const char*>(P.A + am[r]);
      const char* pb = reinterpret_cast<const char*>(P.B + bn[j]);
#pragma unroll 1
      for (int k0 = 0; k0 < klen; k0 += 32) {
        double2 a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int k = k0 + 8 * u + (lane & 7);
          a[u] = b[u] = make_double2(0.0, 0.0);
          if (k < klen) {
            a[u] = *reinterpret_cast<const double2*>(pa + tk[k]);
            b[u] = *reinterpret_cast<const double2*>(pb + tk[kSegMax + k]);
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (k0 + 8 * u < klen) {
            sr = fma(-a[u].y, b[u].y, fma(a[u].x, b[u].x, sr));
            si = fma(a[u].y, b[u].x, fma(a[u].x, b[u].y, si));
          }
      }
    }
    __syncwarp();
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) {
      sr += __shfl_xor_sync(0xffffffffu, sr, d);
      si += __shfl_xor_sync(0xffffffffu, si, d);
    }
    const int rank = __popc(lanes & ((1u << lane) - 1)), src = 8 * (rank & 3);  // this lane's of the four
    sr = __shfl_sync(0xffffffffu, sr, src);
    si = __shfl_sync(0xffffffffu, si, src);
    if (todo && rank < 4) {
      double2 v = z[mine * stride];
      v.x += P.alpha_joined * sr;
      v.y += P.alpha_joined * si;
      z[mine * stride] = v;
      todo &= todo - 1;
    }
  }
}

// Whether a low word of a row's elements k = k0, k0 + step, ... is set.
__device__ __noinline__ uint32_t low_words(const char* row, const long long* tk, int k0, int step, int klen) {
  uint32_t any = 0;
#pragma unroll 1
  for (int k = k0; k < klen; k += step) {
    const uint4 v = *reinterpret_cast<const uint4*>(row + tk[k]);
    any |= v.x | v.z;
  }
  return any ? 1u : 0u;
}

template <int NT, bool AKC, bool BKC>
__global__ void __launch_bounds__(32 * kWorkers + 32, 1) k_oz_gemm(const OzArgs P) {
  using L = OzSmem<NT>;
  constexpr int NB = NT / 2;   // complex columns
  constexpr int CPT = NT / 4;  // real columns a worker thread reads back
  constexpr int CU = 4;        // at a time (eight spill)
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
  uint64_t *full = bars, *empty = bars + 2, *done = bars + 4, *fin = bars + 5;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 6);
  int* sEA = reinterpret_cast<int*>(smem + L::kExpOff);
  long long* sK = reinterpret_cast<long long*>(smem + L::kTabOff);  // k offsets: A, then B
  uint8_t* sWA = smem + L::kWOff;
  uint8_t* sWB = sWA + kRows * kWPitch;
  long long* sAM = reinterpret_cast<long long*>(smem + L::kRowOff);
  long long* sBN = sAM + kRows;
  long long* sCM = sK + 4 * kSegMax;
  long long* sCN = sCM + kRows;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  const unsigned rb = blockIdx.y + blockIdx.z * P.zrow;
  if ((long long)rb * kRows >= P.M) return;
  const int m0 = int(rb) * kRows, n0 = blockIdx.x * NB;
  const int s0 = blockIdx.z * P.zspc, s1 = min(P.nseg, s0 + P.spc);

  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&full[s]), kWorkers);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    mbar_init(smem_u32(done), 1);
    mbar_init(smem_u32(fin), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kWorkers) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)), "r"(L::kCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else {
    if (tid < kRows) sAM[tid] = P.aM[min(m0 + tid, P.M - 1)];
    else if (tid < kRows + NB) sBN[tid - kRows] = P.bN[min(n0 + tid - kRows, P.N - 1)];
  }
  if (warp < kWorkers && P.splits == 1) {
    if (tid < kRows) sCM[tid] = m0 + tid < P.M ? P.cM[m0 + tid] : 0;
    else if (tid < kRows + NB) sCN[tid - kRows] = n0 + tid - kRows < P.N ? P.cN[n0 + tid - kRows] : 0;
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  bool ok = true;

  if (warp == kWorkers) {
    if (lane == 0) {
      int it = 0;
      for (int sg = s0; sg < s1 && ok; ++sg) {
        const int klen = min(P.K, (sg + 1) * P.seg) - sg * P.seg;
        const int nch = (klen + kKC - 1) / kKC;
        for (int c = 0; c < nch; ++c, ++it) {
          const int st = it & 1;
          ok = mbar_wait(smem_u32(&full[st]), (it >> 1) & 1, P.budget);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sa = smem_u32(smem + st * L::kStage), sb = sa + kSl * L::kASlice;
          const int ks = klen - c * kKC > 8 ? 2 : 1;  // 8 complex k per MMA
          for (int kk = 0; kk < ks; ++kk) {
            const uint32_t first = (c | kk) ? 1u : 0u;
#pragma unroll
            for (int i = 0; i < kSl; ++i) {
              const uint64_t da = desc64(sa + i * L::kASlice + kk * 32);
              // stacked digits 0 .. 7 - i, at most 256 columns per MMA
              constexpr int kMaxJ = 256 / NT < kSl ? 256 / NT : kSl;
#pragma unroll
              for (int j = 0; j < kSl - i; j += kMaxJ) {
                const int nj = (kSl - i - j) < kMaxJ ? (kSl - i - j) : kMaxJ;
                mma_f16(tmem + uint32_t((i + j) * NT), da, desc64(sb + j * L::kBSlice + kk * 32),
                        idesc_f16(nj * NT), i == 0 ? first : 1u);
              }
            }
          }
          mma_commit(smem_u32(&empty[st]));
        }
        mma_commit(smem_u32(done));
      }
      // every MMA issued has completed before tensor memory is freed (also
      // after giving up)
      mma_commit(smem_u32(fin));
      if (!mbar_wait(smem_u32(fin), 0, kDrainBudget)) ok = false;
    }
  } else {
    const int w = warp;
    // Element u of a thread in a stage.  A: warp w owns rows 8 w .. + 7; one
    // access covers two rows x 16 k (AKC) or 8 rows x 4 k.  B: 32 rows.
    constexpr int UA = 4, RA = AKC ? UA : 1;
    auto ar = [&](int u) { return AKC ? 8 * w + 2 * u + (lane >> 4) : 8 * w + (lane & 7); };
    auto ak = [&](int u) { return AKC ? (lane & 15) : 4 * u + (lane >> 3); };
    auto br = [&](int) { return BKC ? 2 * w + (lane >> 4) : 8 * (w >> 2) + (lane & 7); };
    auto bk = [&](int) { return BKC ? (lane & 15) : 4 * (w & 3) + (lane >> 3); };
    // Rows and k outside the matrix repeat the last one inside: such rows of the
    // result are not stored, and B's digits are zero beyond the last k.
    const char* arow[RA];
#pragma unroll
    for (int u = 0; u < RA; ++u)
      arow[u] = reinterpret_cast<const char*>(P.A + P.aM[min(m0 + ar(u), P.M - 1)]);
    const char* brow = reinterpret_cast<const char*>(P.B + P.bN[min(n0 + br(0), P.N - 1)]);
    auto aat = [&](int u, long long off) {
      return reinterpret_cast<const double2*>(arow[AKC ? u : 0] + off);
    };
    auto bat = [&](long long off) { return reinterpret_cast<const double2*>(brow + off); };
    // a warp whose rows all lie outside the matrix only clears them once
    const bool wact = m0 + 8 * w < P.M;
    const double2 zero = make_double2(0.0, 0.0);
    auto table = [&](int sg) {  // k offsets of a segment, in bytes
      if (tid >= 2 * kSegMax) return;
      const int k = min(sg * P.seg + min(tid & (kSegMax - 1), P.seg - 1), P.K - 1);
      sK[(sg & 1) * 2 * kSegMax + tid] = 16 * (tid < kSegMax ? P.aK[k] : P.bK[k]);
    };
    table(s0);
    int it = 0;
#pragma unroll 1
    for (int sg = s0; sg < s1; ++sg) {
      const int kb = sg * P.seg, klen = min(P.K, kb + P.seg) - kb;
      const long long* tk = sK + (sg & 1) * 2 * kSegMax;
      int* eA = sEA + (sg & 1) * (kRows + 32);
      int* eB = eA + kRows;
      if (tid < NB) eB[tid] = kNullRow;
      asm volatile("bar.sync 1, %0;" ::"r"(32 * kWorkers) : "memory");
      auto fetch = [&](int c, double2 (&na)[UA], double2& nb) {
#pragma unroll
        for (int u = 0; u < UA; ++u) na[u] = *aat(u, tk[c * kKC + ak(u)]);
        nb = *bat(tk[kSegMax + c * kKC + bk(0)]);
      };
      // the first two stages' elements, used for the exponents too
      double2 na0[UA], na1[UA], nb0, nb1;
      fetch(0, na0, nb0);
      fetch(1, na1, nb1);
      // ---- exponents of the segment's rows (later stages: read for them only,
      // the conversion finds them in L2 again) ------------------------------------
      auto word = [](double2 z) {
        return max(hiabs(uint32_t(__double2hiint(z.x))), hiabs(uint32_t(__double2hiint(z.y))));
      };
      // Weight 2^(7 - n) of an element n binades below its row's largest.
      auto weigh = [&](uint8_t* row, int k, double2 z, int f) {
        row[k] = uint8_t(__funnelshift_rc(128u, 0u, uint32_t(f - int(word(z) >> 20))));
      };
      int fa[RA], fb;
      {
        uint32_t ma[RA], mb = 0;
#pragma unroll
        for (int u = 0; u < RA; ++u) ma[u] = 0;
#pragma unroll 1
        for (int k0 = 2 * kKC; k0 < klen; k0 += 3 * kKC) {
          uint32_t x[3][UA], y[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int u = 0; u < UA; ++u) x[c][u] = row_word(aat(u, tk[k0 + c * kKC + ak(u)]));
            y[c] = row_word(bat(tk[kSegMax + k0 + c * kKC + bk(0)]));
          }
#pragma unroll
          for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int u = 0; u < UA; ++u) ma[AKC ? u : 0] = max(ma[AKC ? u : 0], x[c][u]);
            mb = max(mb, y[c]);
          }
        }
#pragma unroll
        for (int u = 0; u < UA; ++u)
          ma[AKC ? u : 0] = max(ma[AKC ? u : 0], max(word(na0[u]), word(na1[u])));
        mb = max(mb, max(word(nb0), word(nb1)));
        // the lanes of one row: 16 neighbours (k contiguous) or every eighth lane
        auto row_max = [](uint32_t v, bool kc) {
#pragma unroll
          for (int d = 16; d >= 1; d >>= 1)
            if (kc ? d < 16 : d >= 8) v = max(v, __shfl_xor_sync(0xffffffffu, v, d));
          return v;
        };
        bool nil = false;
#pragma unroll
        for (int u = 0; u < RA; ++u) nil |= (ma[u] = row_max(ma[u], AKC)) == 0;
        mb = row_max(mb, BKC);
        if (__any_sync(0xffffffffu, nil || mb == 0)) {
          // no high word but zeros: zeros, unless a low word says that there
          // are the smallest of the subnormal numbers
#pragma unroll
          for (int u = 0; u < RA; ++u)
            ma[u] = max(ma[u], row_max(low_words(arow[u], tk, AKC ? lane & 15 : lane >> 3, AKC ? 16 : 4, klen), AKC));
          mb = max(mb, row_max(low_words(brow, tk + kSegMax, bk(0), kKC, klen), BKC));
        }
        auto exponent = [](uint32_t word) {
          const int f = int(word >> 20);
          return word == 0 ? kNullRow : (f == 2047 ? kNanExp : max(f, kMinExp));
        };
#pragma unroll
        for (int u = 0; u < RA; ++u) {
          fa[u] = max(int(ma[u] >> 20), kMinExp);
          if (AKC ? (lane & 15) == 0 : lane < 8) eA[ar(u)] = exponent(ma[u]);
        }
#pragma unroll
        for (int u = 0; u < UA; ++u) {
          weigh(sWA + ar(u) * kWPitch, ak(u), na0[u], fa[AKC ? u : 0]);
          weigh(sWA + ar(u) * kWPitch, ak(u) + kKC, na1[u], fa[AKC ? u : 0]);
        }
        if ((BKC ? (lane & 15) == 0 : lane < 8) && br(0) < NB) atomicMax(&eB[br(0)], exponent(mb));
      }
      asm volatile("bar.sync 1, %0;" ::"r"(32 * kWorkers) : "memory");
      fb = br(0) < NB ? min(max(eB[br(0)], kMinExp), 2047) : kMinExp;
      if (br(0) < NB) {
        weigh(sWB + br(0) * kWPitch, bk(0), nb0, fb);
        weigh(sWB + br(0) * kWPitch, bk(0) + kKC, nb1, fb);
      }
      if (sg + 1 < s1) table(sg + 1);

      // ---- conversion: elements fetched two stages ahead ----------------------------
      const int nch = (klen + kKC - 1) / kKC;
      auto convert = [&](int c, double2 (&na)[UA], double2& nb) {
        const int st = it & 1;
        if (sg + 1 < s1 && wact && c > 0) {
          // the same places of the next segment, for its exponents
#pragma unroll
          for (int u = 0; u < UA; ++u) {
            const int k = kb + P.seg + (c - 1) * kKC + ak(u);
            if (k < P.K) prefetch_l2(aat(u, 16 * P.aK[k]));
          }
        }
        // (lanes run out of their budgets one by one; what follows takes a whole warp)
        if (it >= 2)
          ok = __all_sync(0xffffffffu, ok && mbar_wait(smem_u32(&empty[st]), ((it >> 1) - 1) & 1, P.budget));
        if (ok) {
          const uint32_t sa = smem_u32(smem + st * L::kStage), sb = sa + kSl * L::kASlice;
          if (wact || it < 2) {
#pragma unroll
            for (int u = 0; u < UA; ++u) {
              const int r = ar(u), k = ak(u);
              const uint32_t at = sa + uint32_t(r * 64 + (((k >> 2) ^ ((r >> 1) & 3)) << 4) + (k & 3) * 4);
              store_a<0, L::kASlice>(at, DigitPairs(na[u], fa[AKC ? u : 0]));
            }
          }
          const int n = br(0), k = bk(0);
          if (n < NB) {
            const uint32_t at = sb + uint32_t(n * 128 + (((k >> 2) ^ (n & 3)) << 4) + (k & 3) * 4);
            const DigitPairs d(nb, c * kKC + k < klen ? fb : kZeroExp);
            // lanes of both kinds share a store instruction without a bank conflict
            const bool h = BKC ? (lane >> 4) != 0 : ((n >> 2) & 1) != 0;
            store_b<0, L::kBSlice>(at + (h ? 64 : 0), d, RowPairs(d, h));
            store_b<0, L::kBSlice>(at + (h ? 0 : 64), d, RowPairs(d, !h));
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&full[st]));
        }
        ++it;
        if (c + 2 < nch) fetch(c + 2, na, nb);
      };
#pragma unroll 1
      for (int c = 0; c < nch; c += 2) {
        convert(c, na0, nb0);
        if (c + 1 < nch) convert(c + 1, na1, nb1);
      }

      // ---- read the accumulators back ---------------------------------------------
      asm volatile("bar.sync 1, %0;" ::"r"(32 * kWorkers) : "memory");  // sWA, sWB are whole
      if (ok) ok = mbar_wait(smem_u32(done), (sg - s0) & 1, P.budget);
      ok = __all_sync(0xffffffffu, ok);
      const int q = w & 3, c0 = (w >> 2) * CPT;
      // The CTA's segments are summed here, between segments in global memory
      // (read back from L2 by the thread that wrote it).  The sum of the last one
      // is staged where the stages were: every MMA has completed, and no warp
      // converts any more.
      const bool more = sg > s0, stage = sg + 1 == s1 && P.splits == 1;
      double* stg = reinterpret_cast<double*>(smem) + (q * 32 + lane) * (2 * L::kPitch) + c0;
      const int m = m0 + q * 32 + lane;
      const int ncol = min(NB, P.N - n0) - (c0 >> 1);
      double2* prow = P.part + ((long long)(P.zspc ? blockIdx.z : 0) * P.N + n0 + (c0 >> 1)) * P.M + m;
      if (ok && m0 + q * 32 < P.M && 2 * n0 + c0 < 2 * P.N) {  // else: no output here
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int F = eA[q * 32 + lane] - 2112 + P.ash;
        const uint32_t tq = tmem + (uint32_t(q * 32) << 16) + uint32_t(c0);
        uint32_t todo = 0;
        // rolled: the code of one tile has to fit the instruction cache
        // (unrolled, fetching it cost more than the work)
#pragma unroll 1
        for (int cc = 0; cc < CPT; cc += CU) {
          uint32_t v[kSl][CU];
#pragma unroll
          for (int g = 0; g < kSl; ++g) tmem_ld(tq + uint32_t(g * NT + cc), v[g]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < CU / 2; ++j) {
            const int E = F + eB[(c0 + cc) / 2 + j];
            double d[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              float x[kSl];
#pragma unroll
              for (int g = 0; g < kSl; ++g) x[g] = __uint_as_float(v[g][2 * j + i]);
              d[i] = join(x, E, P.neg);
            }
            double2 z = make_double2(d[0], d[1]);
            const bool in = m < P.M && cc / 2 + j < ncol;
            const int f = int(max(hiabs(uint32_t(__double2hiint(d[0]))), hiabs(uint32_t(__double2hiint(d[1])))) >> 20);
            const bool off = f == 2047 || E + kSoundField < 54;
            if ((off || f < E + kSoundField) && E > kNullRow / 2 && in) {
              const uint4* wa = reinterpret_cast<const uint4*>(sWA + (q * 32 + lane) * kWPitch);
              const uint4* wb = reinterpret_cast<const uint4*>(sWB + ((c0 + cc) / 2 + j) * kWPitch);
              uint32_t sum = 0;
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const uint4 x = wa[u], y = wb[u];
                sum = __dp4a(x.x, y.x, __dp4a(x.y, y.y, __dp4a(x.z, y.z, __dp4a(x.w, y.w, sum))));
              }
              if (off || sum < kSoundWeight) {
                todo |= 1u << (cc / 2 + j);
                z = zero;
              }
            }
            double2* pz = prow + (long long)(cc / 2 + j) * P.M;
            if (more && in) { const double2 o = *pz; z.x += o.x; z.y += o.y; }
            if (stage) *reinterpret_cast<double2*>(stg + cc + 2 * j) = z;
            else if (in) *pz = z;
          }
        }
        if (__any_sync(0xffffffffu, todo != 0))
          settle(P, todo, stage ? reinterpret_cast<double2*>(stg) : prow, stage ? 1 : P.M, sAM + q * 32,
                 sBN + c0 / 2, tk, klen);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      }
    }
    if (P.splits == 1) {
      // ---- write the tile from shared memory along C's contiguous index
      asm volatile("bar.sync 1, %0;" ::"r"(32 * kWorkers) : "memory");
      const double2* sc = reinterpret_cast<const double2*>(smem);
      constexpr int kEl = kRows * NB / (32 * kWorkers);
      constexpr int kBatch = kEl % 4 == 0 ? 4 : (kEl % 3 == 0 ? 3 : kEl);
      static_assert(kEl % kBatch == 0, "store batches");
#pragma unroll 1
      for (int e0 = 0; e0 < kEl; e0 += kBatch) {
        double2 val[kBatch];
        long long at[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
          const int e = (e0 + u) * 32 * kWorkers + tid;
          const int r = P.c_m ? e % kRows : e / NB, c = P.c_m ? e / kRows : e % NB;
          const bool in = ok && m0 + r < P.M && n0 + c < P.N;
          val[u] = sc[r * L::kPitch + c];
          at[u] = in ? sCM[r] + sCN[c] : -1;
        }
        if (P.alpha_rest != 1.0) {
#pragma unroll
          for (int u = 0; u < kBatch; ++u) { val[u].x *= P.alpha_rest; val[u].y *= P.alpha_rest; }
        }
        if (P.accumulate) {
          double2 old[kBatch];
#pragma unroll
          for (int u = 0; u < kBatch; ++u) old[u] = at[u] >= 0 ? P.C[at[u]] : zero;
#pragma unroll
          for (int u = 0; u < kBatch; ++u) { val[u].x += old[u].x; val[u].y += old[u].y; }
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
          if (at[u] >= 0) P.C[at[u]] = val[u];
      }
    }
  }
  if (!ok && P.err) atomicExch(P.err, 1);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kWorkers) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(L::kCols)
                 : "memory");
  }
}

// C (+)= alpha sum_s part[s][n][m], the splits in a fixed order: LS lanes of a
// warp share one output (every LS-th split each, joined by shuffles).
template <int LS>
__global__ void __launch_bounds__(256)
k_oz_finish(const double2* __restrict__ part, int nsplit, int M, int N, double2* __restrict__ C,
            const long long* __restrict__ cM, const long long* __restrict__ cN, double alpha,
            int accumulate) {
  constexpr int PO = 32 / LS;  // outputs per warp
  const long long total = (long long)M * N;
  const int lane = threadIdx.x & 31;
  const long long t = ((long long)blockIdx.x * 8 + (threadIdx.x >> 5)) * PO + lane % PO;
  double sr = 0.0, si = 0.0;
  if (t < total) {
#pragma unroll 4
    for (int s = lane / PO; s < nsplit; s += LS) {
      const double2 p = part[(long long)s * total + t];
      sr += p.x;
      si += p.y;
    }
  }
#pragma unroll
  for (int d = PO; d < 32; d <<= 1) {
    sr += __shfl_xor_sync(0xffffffffu, sr, d);
    si += __shfl_xor_sync(0xffffffffu, si, d);
  }
  if (t >= total || lane >= PO) return;
  const long long idx = cM[t % M] + cN[t / M];
  double2 v = make_double2(alpha * sr, alpha * si);
  if (accumulate) { v.x += C[idx].x; v.y += C[idx].y; }
  C[idx] = v;
}

// The same for many splits of a small output: a block per four outputs.
__global__ void __launch_bounds__(512)
k_oz_finish_wide(const double2* __restrict__ part, int nsplit, int M, int N, double2* __restrict__ C,
                 const long long* __restrict__ cM, const long long* __restrict__ cN, double alpha,
                 int accumulate) {
  __shared__ double2 red[512];
  const long long total = (long long)M * N;
  const int o = threadIdx.x & 3;
  const long long t = (long long)blockIdx.x * 4 + o;
  double sr = 0.0, si = 0.0;
  if (t < total) {
#pragma unroll 8
    for (int s = threadIdx.x >> 2; s < nsplit; s += 128) {
      const double2 p = part[(long long)s * total + t];
      sr += p.x;
      si += p.y;
    }
  }
  red[threadIdx.x] = make_double2(sr, si);
  for (int d = 256; d >= 4; d >>= 1) {
    __syncthreads();
    if (threadIdx.x < d) {
      red[threadIdx.x].x += red[threadIdx.x + d].x;
      red[threadIdx.x].y += red[threadIdx.x + d].y;
    }
  }
  if (threadIdx.x >= 4 || t >= total) return;
  const long long idx = cM[t % M] + cN[t / M];
  double2 v = make_double2(alpha * red[o].x, alpha * red[o].y);
  if (accumulate) { v.x += C[idx].x; v.y += C[idx].y; }
  C[idx] = v;
}

template <int NT, bool AKC, bool BKC>
void launch_nt(const OzArgs& a, dim3 grid, cudaStream_t s) {
  using L = OzSmem<NT>;
  static PerDevice attr;
  allow_smem(attr, k_oz_gemm<NT, AKC, BKC>, L::kTotal);
  k_oz_gemm<NT, AKC, BKC><<<grid, 32 * kWorkers + 32, L::kTotal, s>>>(a);
  RTCC3_CUDA(cudaGetLastError());
}

}  // namespace

OzPlan oz_plan(long long M, long long N, long long K) {
  OzPlan best;
  best.cost = 1e300;
  const double slots = 152.0;
  for (int sw = 0; sw < 2; ++sw) {
    const long long Mg = sw ? N : M, Ng = sw ? M : N;
    for (const int nt : {64, 48, 32, 16}) {
      const long long tiles = ((Mg + kRows - 1) / kRows) * ((2 * Ng + nt - 1) / nt);
      // segments: short enough that the tiles fill the GPU, at least 32 k, at
      // most the exactness bound
      long long seg = K * tiles / 152;
      seg = std::min<long long>(kSegMax, std::max<long long>(32, seg));
      long long nseg = (K + seg - 1) / seg;
      seg = ((K + nseg - 1) / nseg + 7) / 8 * 8;
      nseg = (K + seg - 1) / seg;
      // CTAs: one per SM is resident; a CTA takes several segments in turn and
      // sums them once the tiles fill two waves.  So the running sums are one
      // per output, or at most 304 tiles of them (20 MB): a partial sum per
      // segment was v / 128 of a triples tensor, 4.5 GB at (15, 57).
      long long zs = std::min(nseg, std::max<long long>(1, (2 * 152) / tiles));
      const long long spc = (nseg + zs - 1) / zs;
      zs = (nseg + spc - 1) / spc;
      // clocks of one segment of one tile: fixed latencies (row maxima,
      // read-back) and 8 complex k at a time, fitted to measurements at
      // K = 7 .. 5e6 with every tile width
      const double per = 14000.0 + double((seg + 7) / 8) * (1500.0 + 8.0 * nt) + 60.0 * nt;
      const double waves = std::ceil(double(tiles * zs) / slots);
      double cost = waves * double(spc) * per + 6000.0;
      if (spc > 1) cost += waves * double(spc) * 70.0 * nt;  // the adds
      if (zs > 1) cost += 6000.0 + double(zs) * double(M) * double(N) / slots;
      if (cost < best.cost) {
        best.swap = sw != 0;
        best.nt = nt;
        best.seg = int(seg);
        best.nseg = int(nseg);
        best.spc = int(spc);
        best.nsplit = int(zs);
        best.cost = cost;
      }
    }
  }
  return best;
}

int oz_gemm(const OzPlan& p, const OzOperand& A, const OzOperand& B, int M, int N, int K, double2* C,
            long long coff, const long long* cM, const long long* cN, bool c_m, double alpha,
            bool accumulate, double2* part, int* err, long long wait_budget, cudaStream_t s) {
  OzArgs a{};
  a.A = A.p + A.off;
  a.B = B.p + B.off;
  a.aM = A.rows;
  a.aK = A.ks;
  a.bN = B.rows;
  a.bK = B.ks;
  a.cM = cM;
  a.cN = cN;
  a.M = M;
  a.N = N;
  a.K = K;
  a.seg = p.seg;
  a.nseg = p.nseg;
  a.spc = p.spc;
  a.err = err;
  a.budget = wait_budget > 0 ? wait_budget : kWaitBudget;
  a.alpha_rest = a.alpha_joined = 1.0;
  const bool split = p.nsplit > 1;
  a.splits = p.nsplit;
  a.accumulate = !split && accumulate ? 1 : 0;
  a.c_m = !split && c_m ? 1 : 0;
  a.C = C + coff;
  a.part = part;
  if (!split) {
    // alpha as a sign, a power of two (joined without FP64 work) and the rest
    int e = 0;
    const double f = std::frexp(alpha, &e);
    if (std::fabs(f) == 0.5) {
      a.ash = e - 1;
      a.alpha_joined = alpha;
      a.neg = alpha < 0 ? 0xffffffffu : 0u;
    } else {
      a.alpha_rest = alpha;
    }
  }
  // more row blocks than the grid's y axis holds (a triples tensor has them):
  // they go on along z, which is free then, because so many tiles are not split
  constexpr unsigned kMaxY = 65535;
  const unsigned rows = unsigned((M + kRows - 1) / kRows), splits = unsigned(p.nsplit);
  RTCC3_CHECK(rows <= kMaxY || splits == 1, kErrArg, "sliced product: splits of a long output");
  a.zrow = splits == 1 ? kMaxY : 0;
  a.zspc = splits == 1 ? 0 : unsigned(p.spc);
  const dim3 grid(unsigned((2LL * N + p.nt - 1) / p.nt), std::min(rows, kMaxY),
                  splits == 1 ? (rows + kMaxY - 1) / kMaxY : splits);
#define RTCC3_OZ(NTV)                                                  \
  if (A.kc && B.kc) launch_nt<NTV, true, true>(a, grid, s);            \
  else if (A.kc) launch_nt<NTV, true, false>(a, grid, s);              \
  else if (B.kc) launch_nt<NTV, false, true>(a, grid, s);              \
  else launch_nt<NTV, false, false>(a, grid, s)
  if (p.nt == 64) { RTCC3_OZ(64); }
  else if (p.nt == 48) { RTCC3_OZ(48); }
  else if (p.nt == 32) { RTCC3_OZ(32); }
  else { RTCC3_OZ(16); }
#undef RTCC3_OZ
  if (!split) return 1;
  const long long total = (long long)M * N;
  auto blocks = [&](int po) { return (unsigned)((total + 8LL * po - 1) / (8LL * po)); };
  if (p.nsplit >= 256 && total <= 65536)
    k_oz_finish_wide<<<(unsigned)((total + 3) / 4), 512, 0, s>>>(part, p.nsplit, M, N, C + coff, cM, cN, alpha, accumulate ? 1 : 0);
  else if (p.nsplit >= 32)
    k_oz_finish<8><<<blocks(4), 256, 0, s>>>(part, p.nsplit, M, N, C + coff, cM, cN, alpha, accumulate ? 1 : 0);
  else
    k_oz_finish<1><<<blocks(32), 256, 0, s>>>(part, p.nsplit, M, N, C + coff, cM, cN, alpha, accumulate ? 1 : 0);
  RTCC3_CUDA(cudaGetLastError());
  return 2;
}

}  // namespace rtcc3
