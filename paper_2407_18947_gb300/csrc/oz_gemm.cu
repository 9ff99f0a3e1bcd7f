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
// integer ones.  Bound by the integer work and its latencies (3800 x 14440 x
// 48: ALU pipe 42 % busy, tensor pipe 15 %, 50000 clocks per tile; 17.6 ms on
// the FP64 cores before, 2.17 ms now).
#include "oz_gemm.h"

#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "tc_ptx.h"

namespace rtcc3 {

namespace {

constexpr int kSl = 8;              // digits
constexpr int kRows = 128;          // A rows per tile
constexpr int kKC = 16;             // complex k per stage (64-byte FP16 rows)
constexpr int kWorkers = 16;        // worker warps
constexpr int kSegMax = 128;        // complex k per segment (256 real: see oz_gemm.h)
constexpr unsigned long long kBias = 0x8080808080808080ULL;

template <int NT>
struct OzSmem {
  static constexpr int kASlice = kRows * 64, kBSlice = NT * 64;
  static constexpr int kStage = kSl * (kASlice + kBSlice);
  static constexpr int kPitch = NT / 2 + 1;  // complex per staged output row
  static constexpr int kBarOff = 2 * kStage;
  static constexpr int kExpOff = kBarOff + 64;                 // row exponents
  static constexpr int kTotal = kExpOff + (kRows + NT / 2) * 4 + 1024;
  static constexpr int kCols = kSl * NT < 32 ? 32 : kSl * NT;  // TMEM columns
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

__device__ __forceinline__ void tmem_ld4(uint32_t t, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(t));
}

// |x| as a sortable word whose top 11 bits are its exponent field.
__device__ __forceinline__ uint32_t hiabs(double x) { return uint32_t(__double2hiint(x)) & 0x7fffffffu; }

// a (|a| < 2^(F - 1022)) as the biased digits of its 62-bit fixed-point form:
// byte 7 - s of the result is digit s plus 128.
__device__ __forceinline__ unsigned long long digits(double a, int F) {
  const uint32_t hi = uint32_t(__double2hiint(a)), lo = uint32_t(__double2loint(a));
  const int ex = int((hi >> 20) & 0x7ffu);
  const unsigned long long m =
      (static_cast<unsigned long long>((hi & 0xfffffu) | (ex ? 0x100000u : 0u)) << 32) | lo;
  const int n = min(max(F - max(ex, 1), 0), 63);
  const unsigned long long x = (((m << 10) >> n) + 1ULL) >> 1;
  return (hi >> 31) ? kBias - x : kBias + x;
}

// Digit s of (re, im) as a pair of halves (1024 + u has the bits 0x6400 | u).
template <int S>
__device__ __forceinline__ uint32_t digit_pair(unsigned long long yr, unsigned long long yi) {
  const uint32_t r = S < 4 ? uint32_t(yr >> 32) : uint32_t(yr);
  const uint32_t i = S < 4 ? uint32_t(yi >> 32) : uint32_t(yi);
  constexpr uint32_t b = 3 - (S & 3);
  uint32_t u = __byte_perm(r, i, b | (b << 4) | ((4 + b) << 8) | ((4 + b) << 12));
  u = (u & 0x00ff00ffu) | 0x64006400u;
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&u),
                            __half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480)));
  return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

template <int S, int STRIDE>
__device__ __forceinline__ void store_a(uint32_t addr, unsigned long long yr, unsigned long long yi) {
  if constexpr (S < kSl) {
    sts32(addr + S * STRIDE, digit_pair<S>(yr, yi));
    store_a<S + 1, STRIDE>(addr, yr, yi);
  }
}

// Both rows of B's embedding, (re, -im) at row 2n and (im, re) at row 2n + 1;
// h: which of the two is stored first (lanes of both kinds share a store
// instruction without a bank conflict).
template <int S, int STRIDE>
__device__ __forceinline__ void store_b(uint32_t addr, uint32_t h, unsigned long long yr,
                                        unsigned long long yi) {
  if constexpr (S < kSl) {
    const uint32_t d = digit_pair<S>(yr, yi);
    const uint32_t even = d ^ 0x80000000u, odd = __byte_perm(d, d, 0x1032);
    sts32(addr + S * STRIDE + (h ? 64 : 0), h ? odd : even);
    sts32(addr + S * STRIDE + (h ? 0 : 64), h ? even : odd);
    store_b<S + 1, STRIDE>(addr, h, yr, yi);
  }
}

// sum_g v_g 2^(56 - 8 g) 2^E, the v_g integers held in FP32, rounded to nearest.
// ash, neg: times 2^ash and -1.
__device__ __forceinline__ double join(const uint32_t* v, int E, int neg) {
  auto iv = [&](int g) { return (long long)__float2int_rn(__uint_as_float(v[g])); };
  long long hi = iv(0) * (1LL << 24) + iv(1) * (1LL << 16) + iv(2) * 256 + iv(3);
  const long long lo = iv(4) * (1LL << 24) + iv(5) * (1LL << 16) + iv(6) * 256 + iv(7);
  // value = hi 2^32 + lo as a 96-bit integer
  hi += lo >> 32;
  uint32_t w0 = uint32_t(lo);
  if (hi < 0) {
    neg ^= 1;
    w0 = 0u - w0;
    hi = w0 ? ~hi : -hi;
  }
  uint32_t w1 = uint32_t(hi), w2 = uint32_t(static_cast<unsigned long long>(hi) >> 32);
  int e = E + 32;
  if (w2 == 0) { w2 = w1; w1 = w0; w0 = 0; e -= 32; }
  if (w2 == 0) { w2 = w1; w1 = w0; w0 = 0; e -= 32; }
  if (w2 == 0) return 0.0;
  const int lz = __clz(w2);
  const unsigned long long top =
      (static_cast<unsigned long long>(__funnelshift_l(w1, w2, lz)) << 32) | __funnelshift_l(w0, w1, lz);
  const unsigned long long t = (top >> 11) + ((top >> 10) & 1ULL);  // 53 bits
  const int field = e - lz + 63 + 1023;
  unsigned long long bits;
  if (field <= 0) bits = 0ULL;
  else bits = (static_cast<unsigned long long>(field - 1) << 52) + t;
  if (field >= 2047 || bits > 0x7ff0000000000000ULL) bits = 0x7ff0000000000000ULL;
  bits |= static_cast<unsigned long long>(neg) << 63;
  return __longlong_as_double((long long)bits);
}

struct OzArgs {
  const double2 *A, *B;
  const long long *aM, *aK, *bN, *bK, *cM, *cN;
  double2* C;      // already moved by its offset; the partials when nsplit > 1
  int M, N, K;
  int seg, nseg, spc;
  int ash, neg;    // alpha = (neg ? -1 : 1) 2^ash alpha_rest
  double alpha_rest;
  int accumulate, to_part, c_m;
  int* err;
  long long budget;
};

template <int NT, bool AKC, bool BKC>
__global__ void __launch_bounds__(32 * kWorkers + 32, 1) k_oz_gemm(const OzArgs P) {
  using L = OzSmem<NT>;
  constexpr int NB = NT / 2;   // complex columns
  constexpr int CPT = NT / 4;  // real columns a worker thread reads back
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
  uint64_t *full = bars, *empty = bars + 2, *done = bars + 4, *fin = bars + 5;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 6);
  int* sEA = reinterpret_cast<int*>(smem + L::kExpOff);
  int* sEB = sEA + kRows;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * kRows, n0 = blockIdx.x * NB;
  const int s0 = blockIdx.z * P.spc, s1 = min(P.nseg, s0 + P.spc);

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
    // rows this thread reads: AKC two rows x 16 k per warp access, else 8 rows x 4 k
    constexpr int UA = 4;
    long long arow[AKC ? UA : 1];
    bool aok[AKC ? UA : 1];
    if (AKC) {
#pragma unroll
      for (int u = 0; u < UA; ++u) {
        const int m = m0 + 8 * w + 2 * u + (lane >> 4);
        aok[u] = m < P.M;
        arow[u] = aok[u] ? P.aM[m] : 0;
      }
    } else {
      const int m = m0 + 8 * w + (lane & 7);
      aok[0] = m < P.M;
      arow[0] = aok[0] ? P.aM[m] : 0;
    }
    const int bn = BKC ? 2 * w + (lane >> 4) : 8 * (w >> 2) + (lane & 7);
    const int bk = BKC ? (lane & 15) : 4 * (w & 3) + (lane >> 3);
    const bool bact = bn < NB;
    const bool bok = bact && n0 + bn < P.N;
    const long long brow = bok ? P.bN[n0 + bn] : 0;
    const double2 zero = make_double2(0.0, 0.0);
    double acc[CPT];
    int it = 0;
    for (int sg = s0; sg < s1; ++sg) {
      const int kb = sg * P.seg, ke = min(P.K, kb + P.seg);
      // ---- exponents of the segment's rows ------------------------------------
      if (threadIdx.x < NB) sEB[threadIdx.x] = 1;
      asm volatile("bar.sync 1, %0;" ::"r"(32 * kWorkers) : "memory");
      int fa[AKC ? UA : 1];
      if (AKC) {
        uint32_t mx[UA] = {0, 0, 0, 0};
#pragma unroll 2
        for (int k = kb + (lane & 15); k < ke; k += 16) {
          const long long ok_ = P.aK[k];
#pragma unroll
          for (int u = 0; u < UA; ++u) {
            const double2 x = aok[u] ? P.A[arow[u] + ok_] : zero;
            mx[u] = max(mx[u], max(hiabs(x.x), hiabs(x.y)));
          }
        }
#pragma unroll
        for (int u = 0; u < UA; ++u) {
#pragma unroll
          for (int d = 8; d > 0; d >>= 1) mx[u] = max(mx[u], __shfl_xor_sync(0xffffffffu, mx[u], d));
          fa[u] = max(int(mx[u] >> 20), 1);
          if ((lane & 15) == 0) sEA[8 * w + 2 * u + (lane >> 4)] = fa[u];
        }
      } else {
        uint32_t mx = 0;
#pragma unroll 8
        for (int k = kb + (lane >> 3); k < ke; k += 4) {
          const double2 x = aok[0] ? P.A[arow[0] + P.aK[k]] : zero;
          mx = max(mx, max(hiabs(x.x), hiabs(x.y)));
        }
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
        fa[0] = max(int(mx >> 20), 1);
        if (lane < 8) sEA[8 * w + lane] = fa[0];
      }
      if (bok) {
        uint32_t mx = 0;
#pragma unroll 4
        for (int k = kb + bk; k < ke; k += 16) {
          const double2 x = P.B[brow + P.bK[k]];
          mx = max(mx, max(hiabs(x.x), hiabs(x.y)));
        }
        atomicMax(&sEB[bn], int(mx >> 20));
      }
      asm volatile("bar.sync 1, %0;" ::"r"(32 * kWorkers) : "memory");
      const int fb = bact ? sEB[bn] : 1;

      // ---- conversion, one stage ahead of the MMAs ------------------------------
      const int nch = (ke - kb + kKC - 1) / kKC;
      double2 na[UA], nbv;
      auto fetch = [&](int c) {
        const int k0 = kb + c * kKC;
        if (AKC) {
          const int k = k0 + (lane & 15);
          const long long o = k < ke ? P.aK[k] : 0;
#pragma unroll
          for (int u = 0; u < UA; ++u) na[u] = (aok[u] && k < ke) ? P.A[arow[u] + o] : zero;
        } else {
#pragma unroll
          for (int u = 0; u < UA; ++u) {
            const int k = k0 + 4 * u + (lane >> 3);
            na[u] = (aok[0] && k < ke) ? P.A[arow[0] + P.aK[k]] : zero;
          }
        }
        const int k = k0 + bk;
        nbv = (bok && k < ke) ? P.B[brow + P.bK[k]] : zero;
      };
      fetch(0);
      for (int c = 0; c < nch; ++c, ++it) {
        const int st = it & 1;
        double2 ca[UA];
#pragma unroll
        for (int u = 0; u < UA; ++u) ca[u] = na[u];
        const double2 cb = nbv;
        if (c + 1 < nch) fetch(c + 1);
        if (it >= 2 && ok) ok = mbar_wait(smem_u32(&empty[st]), ((it >> 1) - 1) & 1, P.budget);
        if (!ok) continue;
        const uint32_t sa = smem_u32(smem + st * L::kStage), sb = sa + kSl * L::kASlice;
#pragma unroll
        for (int u = 0; u < UA; ++u) {
          const int r = AKC ? 8 * w + 2 * u + (lane >> 4) : 8 * w + (lane & 7);
          const int k = AKC ? (lane & 15) : 4 * u + (lane >> 3);
          const uint32_t at = sa + uint32_t(r * 64 + (((k >> 2) ^ ((r >> 1) & 3)) << 4) + (k & 3) * 4);
          const int F = AKC ? fa[u] : fa[0];
          store_a<0, L::kASlice>(at, digits(ca[u].x, F), digits(ca[u].y, F));
        }
        if (bact) {
          const uint32_t at = sb + uint32_t(bn * 128 + (((bk >> 2) ^ (bn & 3)) << 4) + (bk & 3) * 4);
          store_b<0, L::kBSlice>(at, uint32_t(BKC ? (lane >> 4) : ((bn >> 2) & 1)), digits(cb.x, fb),
                                 digits(cb.y, fb));
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&full[st]));
      }

      // ---- read the accumulators back ---------------------------------------------
      if (ok) ok = mbar_wait(smem_u32(done), (sg - s0) & 1, P.budget);
      ok = __all_sync(0xffffffffu, ok);
      if (ok) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int q = w & 3, c0 = (w >> 2) * CPT;
        const int F = sEA[q * 32 + lane];
        const uint32_t tq = tmem + (uint32_t(q * 32) << 16) + uint32_t(c0);
#pragma unroll
        for (int cc = 0; cc < CPT; cc += 4) {
          uint32_t v[kSl][4];
#pragma unroll
          for (int g = 0; g < kSl; ++g) tmem_ld4(tq + uint32_t(g * NT + cc), v[g]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int G = sEB[(c0 + cc + j) >> 1];
            uint32_t x[kSl];
#pragma unroll
            for (int g = 0; g < kSl; ++g) x[g] = v[g][j];
            double d = join(x, F + G - 2112 + P.ash, P.neg);
            if (F == 2047 || G == 2047) d = __longlong_as_double(0x7ff8000000000000LL);
            if (sg == s0) acc[cc + j] = d;
            else acc[cc + j] += d;
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      }
      // sEA / sEB are rewritten by the next segment
      if (sg + 1 < s1) asm volatile("bar.sync 1, %0;" ::"r"(32 * kWorkers) : "memory");
    }
    // ---- write the tile, through shared memory so that stores run along C's
    // contiguous index (the stages are free: every MMA has completed)
    asm volatile("bar.sync 1, %0;" ::"r"(32 * kWorkers) : "memory");
    double* stg = reinterpret_cast<double*>(smem);
    if (ok) {
      const int q = w & 3, c0 = (w >> 2) * CPT;
#pragma unroll
      for (int cc = 0; cc < CPT; cc += 2)
        *reinterpret_cast<double2*>(&stg[(q * 32 + lane) * (2 * L::kPitch) + c0 + cc]) =
            make_double2(acc[cc], acc[cc + 1]);
    }
    asm volatile("bar.sync 1, %0;" ::"r"(32 * kWorkers) : "memory");
    const double2* sc = reinterpret_cast<const double2*>(smem);
    constexpr int kEl = kRows * NB / (32 * kWorkers);
    double2 val[kEl];
    long long at[kEl];
#pragma unroll
    for (int u = 0; u < kEl; ++u) {
      const int e = u * 32 * kWorkers + int(threadIdx.x);
      const int r = P.c_m ? e % kRows : e / NB, c = P.c_m ? e / kRows : e % NB;
      const int m = m0 + r, n = n0 + c;
      const bool in = ok && m < P.M && n < P.N;
      val[u] = sc[r * L::kPitch + c];
      if (P.alpha_rest != 1.0) { val[u].x *= P.alpha_rest; val[u].y *= P.alpha_rest; }
      at[u] = !in ? -1
                  : (P.to_part ? ((long long)blockIdx.z * P.M + m) * P.N + n : P.cM[m] + P.cN[n]);
    }
    if (P.accumulate) {
      double2 old[kEl];
#pragma unroll
      for (int u = 0; u < kEl; ++u) old[u] = at[u] >= 0 ? P.C[at[u]] : zero;
#pragma unroll
      for (int u = 0; u < kEl; ++u) { val[u].x += old[u].x; val[u].y += old[u].y; }
    }
#pragma unroll
    for (int u = 0; u < kEl; ++u)
      if (at[u] >= 0) P.C[at[u]] = val[u];
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

// C (+)= alpha sum_s part[s][m][n], the splits in a fixed order: LS lanes of a
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
  const long long idx = cM[t / N] + cN[t % N];
  double2 v = make_double2(alpha * sr, alpha * si);
  if (accumulate) { v.x += C[idx].x; v.y += C[idx].y; }
  C[idx] = v;
}

template <int NT, bool AKC, bool BKC>
void launch_nt(const OzArgs& a, dim3 grid, cudaStream_t s) {
  using L = OzSmem<NT>;
  // per device and process; set again by a second thread without harm
  static std::atomic<bool> attr{false};
  if (!attr.load(std::memory_order_acquire)) {
    RTCC3_CUDA(cudaFuncSetAttribute(k_oz_gemm<NT, AKC, BKC>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, L::kTotal));
    attr.store(true, std::memory_order_release);
  }
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
    for (int nt = 64; nt >= 16; nt /= 2) {
      const long long tiles = ((Mg + kRows - 1) / kRows) * ((2 * Ng + nt - 1) / nt);
      // segments: short enough that the tiles fill the GPU, at least 32 k, at
      // most the exactness bound
      long long seg = K * tiles / 152;
      seg = std::min<long long>(kSegMax, std::max<long long>(32, seg));
      long long nseg = (K + seg - 1) / seg;
      seg = ((K + nseg - 1) / nseg + 7) / 8 * 8;
      nseg = (K + seg - 1) / seg;
      // CTAs: one per SM is resident; split the segments while tiles are fewer
      // than two waves
      long long zs = std::min(nseg, std::max<long long>(1, (2 * 152) / tiles));
      const long long spc = (nseg + zs - 1) / zs;
      zs = (nseg + spc - 1) / spc;
      // clocks of one segment of one tile: fixed latencies (row maxima,
      // read-back) and 8 complex k at a time, fitted to measurements at
      // K = 48 .. 1.4e6 with tiles of 32 and 64 columns
      const double per = double((seg + 7) / 8) * (1900.0 + 18.0 * nt) + 24000.0 + 130.0 * nt;
      const double waves = std::ceil(double(tiles * zs) / slots);
      double cost = waves * double(spc) * per + 4000.0;
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
  a.alpha_rest = 1.0;
  const bool split = p.nsplit > 1;
  a.to_part = split ? 1 : 0;
  a.accumulate = !split && accumulate ? 1 : 0;
  a.c_m = !split && c_m ? 1 : 0;
  a.C = split ? part : C + coff;
  if (!split) {
    // alpha as a sign, a power of two (joined without FP64 work) and the rest
    int e = 0;
    const double f = std::frexp(alpha, &e);
    if (std::fabs(f) == 0.5) {
      a.ash = e - 1;
      a.neg = alpha < 0 ? 1 : 0;
    } else {
      a.alpha_rest = alpha;
    }
  }
  const long long gx = (2LL * N + p.nt - 1) / p.nt, gy = (M + kRows - 1) / kRows;
  RTCC3_CHECK(gy < 65536 && p.nsplit < 65536, kErrArg, "sliced product: grid too large");
  dim3 grid((unsigned)gx, (unsigned)gy, (unsigned)p.nsplit);
#define RTCC3_OZ(NTV)                                                  \
  if (A.kc && B.kc) launch_nt<NTV, true, true>(a, grid, s);            \
  else if (A.kc) launch_nt<NTV, true, false>(a, grid, s);              \
  else if (B.kc) launch_nt<NTV, false, true>(a, grid, s);              \
  else launch_nt<NTV, false, false>(a, grid, s)
  if (p.nt == 64) { RTCC3_OZ(64); }
  else if (p.nt == 32) { RTCC3_OZ(32); }
  else { RTCC3_OZ(16); }
#undef RTCC3_OZ
  if (!split) return 1;
  const long long total = (long long)M * N;
  auto blocks = [&](int po) { return (unsigned)((total + 8LL * po - 1) / (8LL * po)); };
  if (p.nsplit >= 32)
    k_oz_finish<8><<<blocks(4), 256, 0, s>>>(part, p.nsplit, M, N, C + coff, cM, cN, alpha, accumulate ? 1 : 0);
  else
    k_oz_finish<1><<<blocks(32), 256, 0, s>>>(part, p.nsplit, M, N, C + coff, cM, cN, alpha, accumulate ? 1 : 0);
  RTCC3_CUDA(cudaGetLastError());
  return 2;
}

}  // namespace rtcc3
