// Small-output and single-column contractions (see contract_small.h).
#include "contract_small.h"

#include <algorithm>

namespace rtcc3 {

namespace {

constexpr int kThreads = 256;

template <typename R>
__device__ __forceinline__ void cfma(R& ar, R& ai, Cx<R> a, Cx<R> b) {
  ar = fma(a.x, b.x, ar);
  ar = fma(-a.y, b.y, ar);
  ai = fma(a.x, b.y, ai);
  ai = fma(a.y, b.x, ai);
}

// RM x RN threads own UM x UN outputs each (rows rm + RM i, columns rn + RN j);
// the remaining G = 256 / (RM RN) thread groups take interleaved k of every
// slice and are summed in a fixed order at the end.
template <typename R, int RM, int RN, int UM, int UN>
struct SmallShape {
  static constexpr int MP = RM * UM, NP = RN * UN, G = kThreads / (RM * RN);
  static constexpr int EB = int(sizeof(Cx<R>));
  static constexpr int BK0 = 40960 / ((MP + NP + 2) * EB);
  // deep slices keep more loads in flight per thread (128 for the 16 x 16 tile)
  static constexpr int BK = BK0 >= 128 ? 128 : (BK0 >= 64 ? 64 : (BK0 >= 32 ? 32 : (BK0 >= 16 ? 16 : (BK0 >= 8 ? 8 : 4))));
  // thread groups sharing a warp (summed by shuffles) and the rest (by shared memory)
  static constexpr int WG = RM * RN >= 32 ? 1 : 32 / (RM * RN);
  static constexpr int GS = G / WG;
  // slices are stored [k][m] with an odd row pitch so that the transposing
  // stores of K-contiguous loads do not hit one bank
  static constexpr int MS = MP + 1, NS = NP + 1;
  static constexpr int TILE_BYTES = BK * (MS + NS) * EB;
  static constexpr int RED_BYTES = GS > 1 ? MP * NP * EB : 0;
  static constexpr int SMEM = TILE_BYTES > RED_BYTES ? TILE_BYTES : RED_BYTES;
  static_assert(G >= 1 && BK >= G, "slice shallower than the thread groups");
  static_assert(SMEM <= 48 * 1024, "static shared memory");
};

template <typename R, bool A_KC, bool B_KC, int RM, int RN, int UM, int UN>
__global__ void __launch_bounds__(kThreads)
k_reduce_small(const Cx<R>* __restrict__ A, long long aoff, const long long* __restrict__ aM,
               const long long* __restrict__ aK, const Cx<R>* __restrict__ B, long long boff,
               const long long* __restrict__ bN, const long long* __restrict__ bK,
               Cx<R>* __restrict__ Cp, long long coff, const long long* __restrict__ cM,
               const long long* __restrict__ cN, int M, int N, int K, int kchunk, R alpha,
               int accumulate, Cx<R>* __restrict__ part) {
  using S = SmallShape<R, RM, RN, UM, UN>;
  constexpr int MP = S::MP, NP = S::NP, G = S::G, BK = S::BK;
  __shared__ __align__(16) unsigned char smem[S::SMEM];
  constexpr int MS = S::MS, NS = S::NS;
  Cx<R>* As = reinterpret_cast<Cx<R>*>(smem);  // [BK][MS]
  Cx<R>* Bs = As + BK * MS;                      // [BK][NS]
  const int tid = threadIdx.x;
  const int rn = tid % RN, rm = (tid / RN) % RM, g = tid / (RM * RN);
  const int split = blockIdx.x;
  const int kbeg = split * kchunk;
  const int kend = min(K, kbeg + kchunk);
  R accr[UM][UN], acci[UM][UN];
#pragma unroll
  for (int i = 0; i < UM; ++i)
#pragma unroll
    for (int j = 0; j < UN; ++j) { accr[i][j] = R(0); acci[i][j] = R(0); }
  const Cx<R> zero = cmake<R>(R(0), R(0));
  const Cx<R>* Ab = A + aoff;
  const Cx<R>* Bb = B + boff;
  // the next slice is fetched into registers while the current one is used
  constexpr int LA = (MP * BK + kThreads - 1) / kThreads, LB = (NP * BK + kThreads - 1) / kThreads;
  Cx<R> ra[LA], rb[LB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < LA; ++u) {
      const int e = tid + u * kThreads;
      int mm, kk;
      if (A_KC) { kk = e % BK; mm = e / BK; } else { mm = e % MP; kk = e / MP; }
      const int k = k0 + kk;
      ra[u] = (e < MP * BK && mm < M && k < kend) ? Ab[aM[mm] + aK[k]] : zero;
    }
#pragma unroll
    for (int u = 0; u < LB; ++u) {
      const int e = tid + u * kThreads;
      int nn, kk;
      if (B_KC) { kk = e % BK; nn = e / BK; } else { nn = e % NP; kk = e / NP; }
      const int k = k0 + kk;
      rb[u] = (e < NP * BK && nn < N && k < kend) ? Bb[bN[nn] + bK[k]] : zero;
    }
  };
  if (kbeg < kend) fetch(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int u = 0; u < LA; ++u) {
      const int e = tid + u * kThreads;
      int mm, kk;
      if (A_KC) { kk = e % BK; mm = e / BK; } else { mm = e % MP; kk = e / MP; }
      if (e < MP * BK) As[kk * MS + mm] = ra[u];
    }
#pragma unroll
    for (int u = 0; u < LB; ++u) {
      const int e = tid + u * kThreads;
      int nn, kk;
      if (B_KC) { kk = e % BK; nn = e / BK; } else { nn = e % NP; kk = e / NP; }
      if (e < NP * BK) Bs[kk * NS + nn] = rb[u];
    }
    __syncthreads();
    if (k0 + BK < kend) fetch(k0 + BK);
#pragma unroll 4
    for (int kk = g; kk < BK; kk += G) {
      Cx<R> a[UM], b[UN];
#pragma unroll
      for (int i = 0; i < UM; ++i) a[i] = As[kk * MS + rm + RM * i];
#pragma unroll
      for (int j = 0; j < UN; ++j) b[j] = Bs[kk * NS + rn + RN * j];
#pragma unroll
      for (int i = 0; i < UM; ++i)
#pragma unroll
        for (int j = 0; j < UN; ++j) cfma<R>(accr[i][j], acci[i][j], a[i], b[j]);
    }
    __syncthreads();
  }
  // fixed-order sum over the thread groups: shuffles within a warp, then
  // shared memory across warps
  if (S::WG > 1) {
#pragma unroll
    for (int off = RM * RN; off < 32; off <<= 1)
#pragma unroll
      for (int i = 0; i < UM; ++i)
#pragma unroll
        for (int j = 0; j < UN; ++j) {
          accr[i][j] += __shfl_xor_sync(0xffffffffu, accr[i][j], off);
          acci[i][j] += __shfl_xor_sync(0xffffffffu, acci[i][j], off);
        }
  }
  auto store = [&](int m, int n, R re, R im) {
    if (m >= M || n >= N) return;
    if (part) {
      part[(size_t(m) * N + n) * gridDim.x + split] = cmake<R>(re, im);
    } else {
      const long long idx = coff + cM[m] + cN[n];
      Cx<R> v = cmake<R>(alpha * re, alpha * im);
      if (accumulate) { v.x += Cp[idx].x; v.y += Cp[idx].y; }
      Cp[idx] = v;
    }
  };
  if (S::GS == 1) {
    if (g != 0) return;
#pragma unroll
    for (int i = 0; i < UM; ++i)
#pragma unroll
      for (int j = 0; j < UN; ++j) store(rm + RM * i, rn + RN * j, accr[i][j], acci[i][j]);
    return;
  }
  // one [MP][NP] tile in shared memory, the warp-level partials added into it
  // one group after another (fixed order)
  Cx<R>* red = reinterpret_cast<Cx<R>*>(smem);
  for (int gs = 0; gs < S::GS; ++gs) {
    if (g % S::WG == 0 && g / S::WG == gs) {
#pragma unroll
      for (int i = 0; i < UM; ++i)
#pragma unroll
        for (int j = 0; j < UN; ++j) {
          Cx<R>& r = red[(rm + RM * i) * NP + rn + RN * j];
          r = gs == 0 ? cmake<R>(accr[i][j], acci[i][j])
                      : cmake<R>(r.x + accr[i][j], r.y + acci[i][j]);
        }
    }
    __syncthreads();
  }
  for (int t = tid; t < MP * NP; t += kThreads) store(t / NP, t % NP, red[t].x, red[t].y);
}

// C[cM[m] + cN[n]] (+)= alpha sum_s part[m][n][s]: one warp per output, the
// splits summed in a fixed order (lane-strided, then a shuffle tree).
template <typename R>
__global__ void __launch_bounds__(kThreads)
k_split_sum(const Cx<R>* __restrict__ part, int nsplit, Cx<R>* __restrict__ Cp, long long coff,
            const long long* __restrict__ cM, const long long* __restrict__ cN, int M, int N,
            R alpha, int accumulate) {
  const int lane = threadIdx.x & 31;
  const long long w0 = (long long)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
  const long long nw = (long long)gridDim.x * (kThreads / 32);
  for (long long t = w0; t < (long long)M * N; t += nw) {
    const Cx<R>* p = part + t * nsplit;
    R re = 0, im = 0;
    for (int sp = lane; sp < nsplit; sp += 32) {
      re += p[sp].x;
      im += p[sp].y;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      re += __shfl_xor_sync(0xffffffffu, re, off);
      im += __shfl_xor_sync(0xffffffffu, im, off);
    }
    if (lane == 0) {
      const int m = int(t / N), n = int(t - (long long)m * N);
      const long long idx = coff + cM[m] + cN[n];
      Cx<R> v = cmake<R>(alpha * re, alpha * im);
      if (accumulate) { v.x += Cp[idx].x; v.y += Cp[idx].y; }
      Cp[idx] = v;
    }
  }
}

// One output per warp (A contiguous along k: lanes stride k) or per thread.
template <typename R, bool A_KC>
__global__ void __launch_bounds__(kThreads)
k_gemv(const Cx<R>* __restrict__ A, long long aoff, const long long* __restrict__ aM,
       const long long* __restrict__ aK, const Cx<R>* __restrict__ B, long long boff,
       const long long* __restrict__ bK, Cx<R>* __restrict__ Cp, long long coff,
       const long long* __restrict__ cM, int M, int K, R alpha, int accumulate) {
  const Cx<R>* Ab = A + aoff;
  const Cx<R>* Bb = B + boff;
  if (A_KC) {
    const int lane = threadIdx.x & 31;
    const long long w0 = (long long)(blockIdx.x * (kThreads / 32)) + (threadIdx.x >> 5);
    const long long nw = (long long)gridDim.x * (kThreads / 32);
    for (long long m = w0; m < M; m += nw) {
      const Cx<R>* row = Ab + aM[m];
      R re = 0, im = 0;
      for (int k = lane; k < K; k += 32) cfma<R>(re, im, row[aK[k]], Bb[bK[k]]);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, off);
        im += __shfl_xor_sync(0xffffffffu, im, off);
      }
      if (lane == 0) {
        const long long idx = coff + cM[m];
        Cx<R> v = cmake<R>(alpha * re, alpha * im);
        if (accumulate) { v.x += Cp[idx].x; v.y += Cp[idx].y; }
        Cp[idx] = v;
      }
    }
  } else {
    for (long long m = (long long)blockIdx.x * kThreads + threadIdx.x; m < M;
         m += (long long)gridDim.x * kThreads) {
      const Cx<R>* row = Ab + aM[m];
      R re = 0, im = 0;
#pragma unroll 4
      for (int k = 0; k < K; ++k) cfma<R>(re, im, row[aK[k]], Bb[bK[k]]);
      const long long idx = coff + cM[m];
      Cx<R> v = cmake<R>(alpha * re, alpha * im);
      if (accumulate) { v.x += Cp[idx].x; v.y += Cp[idx].y; }
      Cp[idx] = v;
    }
  }
}

template <typename R>
__global__ void __launch_bounds__(kThreads)
k_outer(const Cx<R>* __restrict__ A, long long aoff, const long long* __restrict__ aM,
        const long long* __restrict__ aK, const Cx<R>* __restrict__ B, long long boff,
        const long long* __restrict__ bN, const long long* __restrict__ bK, Cx<R>* __restrict__ Cp,
        long long coff, const long long* __restrict__ cM, const long long* __restrict__ cN, int M,
        int N, R alpha, int accumulate) {
  const long long ak = aK[0], bk = bK[0];
  for (int m = blockIdx.y; m < M; m += gridDim.y) {
    const Cx<R> a = A[aoff + aM[m] + ak];
    const R ar = alpha * a.x, ai = alpha * a.y;
    const long long cm = coff + cM[m];
    for (int n = blockIdx.x * kThreads + threadIdx.x; n < N; n += gridDim.x * kThreads) {
      const Cx<R> b = B[boff + bN[n] + bk];
      const long long idx = cm + cN[n];
      Cx<R> v = cmake<R>(ar * b.x - ai * b.y, ar * b.y + ai * b.x);
      if (accumulate) {
        const Cx<R> c = Cp[idx];
        v.x += c.x;
        v.y += c.y;
      }
      Cp[idx] = v;
    }
  }
}

template <typename R, int RM, int RN, int UM, int UN>
void launch_cfg(bool a_kc, bool b_kc, const Cx<R>* A, long long aoff, const long long* aM,
                const long long* aK, const Cx<R>* B, long long boff, const long long* bN,
                const long long* bK, Cx<R>* C, long long coff, const long long* cM,
                const long long* cN, int M, int N, int K, int nsplit, int kchunk, double alpha,
                bool accumulate, Cx<R>* part, cudaStream_t s) {
  Cx<R>* p = nsplit > 1 ? part : nullptr;
#define RTCC3_RS(AK, BK_)                                                                        \
  k_reduce_small<R, AK, BK_, RM, RN, UM, UN><<<nsplit, kThreads, 0, s>>>(                        \
      A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K, kchunk, R(alpha),              \
      accumulate ? 1 : 0, p)
  if (a_kc && b_kc) RTCC3_RS(true, true);
  else if (a_kc) RTCC3_RS(true, false);
  else if (b_kc) RTCC3_RS(false, true);
  else RTCC3_RS(false, false);
#undef RTCC3_RS
  RTCC3_CUDA(cudaGetLastError());
  if (nsplit > 1) {
    const long long warps = (long long)M * N;
    const int grid = int(std::max<long long>(1, std::min<long long>((warps * 32 + kThreads - 1) / kThreads,
                                                                     152LL * 16)));
    k_split_sum<R><<<grid, kThreads, 0, s>>>(part, nsplit, C, coff, cM, cN, M, N, R(alpha),
                                             accumulate ? 1 : 0);
    RTCC3_CUDA(cudaGetLastError());
  }
}

// ---- small products spread over the GPU (FineArgs) ----------------------------
// The tiled kernels give a 38 x 38 x 38 product to one or a few CTAs, which
// multiply a zero-padded tile: in FP64 that is 40 to 270 us on an SM with two
// FP64 lanes per clock, in FP32 ten dependent load-barrier-multiply rounds.
// Here every lane owns a few terms of one output and all its loads are
// independent, so a product takes about the latency of one load chain
// (tables, operands): bound by latency below about 1e5 terms, by the FP64
// pipe (two terms per SM and 4 clocks) above.
template <typename R>
__device__ __forceinline__ void fine_sum(const FineArgs<R>& a, const Cx<R>* pa, const Cx<R>* pb,
                                         int k, int step, R& sr, R& si) {
  R r0 = R(0), i0 = R(0), r1 = R(0), i1 = R(0);
  const bool lin = a.aks >= 0 && a.bks >= 0;
  auto at = [&](int kk, Cx<R>& x, Cx<R>& y) {
    x = pa[lin ? kk * a.aks : a.aK[kk]];
    y = pb[lin ? kk * a.bks : a.bK[kk]];
  };
  for (; k + 3 * step < a.K; k += 4 * step) {
    Cx<R> x[4], y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) at(k + u * step, x[u], y[u]);
    cfma<R>(r0, i0, x[0], y[0]);
    cfma<R>(r1, i1, x[1], y[1]);
    cfma<R>(r0, i0, x[2], y[2]);
    cfma<R>(r1, i1, x[3], y[3]);
  }
  {
    const Cx<R> zero = cmake<R>(R(0), R(0));
    Cx<R> x[3] = {zero, zero, zero}, y[3] = {zero, zero, zero};
#pragma unroll
    for (int u = 0; u < 3; ++u)
      if (k + u * step < a.K) at(k + u * step, x[u], y[u]);
#pragma unroll
    for (int u = 0; u < 3; ++u)
      if (k + u * step < a.K) cfma<R>(u & 1 ? r1 : r0, u & 1 ? i1 : i0, x[u], y[u]);
  }
  sr = r0 + r1;
  si = i0 + i1;
}

template <typename R>
__device__ __forceinline__ void fine_store(const FineArgs<R>& a, long long idx, R sr, R si) {
  Cx<R> v = cmake<R>(a.alpha * sr, a.alpha * si);
  if (a.accumulate) {
    const Cx<R> o = a.C[idx];
    v.x += o.x;
    v.y += o.y;
  }
  a.C[idx] = v;
}

template <typename R>
__device__ __forceinline__ void fine_decode(const FineArgs<R>& a, unsigned o, unsigned& b, unsigned& m,
                                            unsigned& n) {
  const unsigned M = unsigned(a.M), N = unsigned(a.N);
  if (a.n_fast) {
    n = o % N;
    o /= N;
    m = o % M;
    b = o / M;
  } else {
    m = o % M;
    o /= M;
    n = o % N;
    b = o / N;
  }
}

template <typename R>
__global__ void __launch_bounds__(128) k_contract_fine(const FineArgs<R> a, unsigned total) {
  const unsigned idx = blockIdx.x * 128u + threadIdx.x;
  const unsigned o = idx >> a.ls_log, ks = idx & ((1u << a.ls_log) - 1u);
  R sr = R(0), si = R(0);
  unsigned b = 0, m = 0, n = 0;
  const bool in = o < total;
  if (in) {
    fine_decode(a, o, b, m, n);
    fine_sum<R>(a, a.A + a.aB[b] + a.aM[m], a.B + a.bB[b] + a.bN[n], int(ks), 1 << a.ls_log, sr, si);
  }
  for (int d = (1 << a.ls_log) >> 1; d > 0; d >>= 1) {
    sr += __shfl_down_sync(0xffffffffu, sr, d);
    si += __shfl_down_sync(0xffffffffu, si, d);
  }
  if (in && ks == 0) fine_store(a, a.cB[b] + a.cM[m] + a.cN[n], sr, si);
}

// One output per block: few outputs with long sums.
template <typename R>
__global__ void __launch_bounds__(256) k_contract_fine_block(const FineArgs<R> a) {
  __shared__ R red[16];
  unsigned b, m, n;
  fine_decode(a, blockIdx.x, b, m, n);
  R sr, si;
  fine_sum<R>(a, a.A + a.aB[b] + a.aM[m], a.B + a.bB[b] + a.bN[n], int(threadIdx.x), 256, sr, si);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    sr += __shfl_down_sync(0xffffffffu, sr, d);
    si += __shfl_down_sync(0xffffffffu, si, d);
  }
  if ((threadIdx.x & 31) == 0) {
    red[2 * (threadIdx.x >> 5)] = sr;
    red[2 * (threadIdx.x >> 5) + 1] = si;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  sr = red[0];
  si = red[1];
#pragma unroll
  for (int w = 1; w < 8; ++w) {
    sr += red[2 * w];
    si += red[2 * w + 1];
  }
  fine_store(a, a.cB[b] + a.cM[m] + a.cN[n], sr, si);
}

}  // namespace

template <typename R>
void launch_outer(const Cx<R>* A, long long aoff, const long long* aM, const long long* aK,
                  const Cx<R>* B, long long boff, const long long* bN, const long long* bK,
                  Cx<R>* C, long long coff, const long long* cM, const long long* cN, int M, int N,
                  double alpha, bool accumulate, cudaStream_t s) {
  // about four outputs per thread along n, rows spread over grid.y
  const int gx = std::max(1, std::min(1024, (N + 4 * kThreads - 1) / (4 * kThreads)));
  const int gy = std::max(1, std::min(M, std::max(1, 152 * 32 / gx)));
  k_outer<R><<<dim3(gx, gy), kThreads, 0, s>>>(A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN,
                                               M, N, R(alpha), accumulate ? 1 : 0);
  RTCC3_CUDA(cudaGetLastError());
}

int small_output_config(long long M, long long N) {
  if (M <= 6 && N <= 6) return kSmall6;
  if (M <= 8 && N <= 8) return kSmall8;
  if (M <= 10 && N <= 10) return kSmall10;
  if (M <= 16 && N <= 16) return kSmall16;
  // 20, 24, 32: the arithmetic goes with the tile's square, so a 20 x 20 output on
  // the 40 tile did four times its work ((20, 76) occ x occ density, complex64:
  // 5.8 -> 2.2 ms per slab of two; 27 x 27 on 40: 0.153 -> 0.101 ms).
  if (M <= 20 && N <= 20) return kSmall20;
  if (M <= 24 && N <= 24) return kSmall24;
  if (M <= 32 && N <= 32) return kSmall32;
  if (M <= 40 && N <= 40) return kSmall40;
  if (M <= 48 && N <= 48) return kSmall48;
  if (M <= 64 && N <= 64) return kSmall64;
  // 76 x 76 on a 2 x 2 grid of 64 x 64 tiles computed 2.8 times its output and read
  // both operands twice: 12.1 -> 4.9 ms per slab of two of (20, 76).
  // Tiles of 80 and 96 only where both sides need them: an output of few columns
  // (M = 95, N = 1) pays for the whole square (0.59 ms instead of 0.02 at 1e6 terms).
  if (M <= 80 && N <= 80 && N > 40) return kSmall80;
  if (M <= 96 && N <= 96 && N > 48) return kSmall96;
  if (N == 1 && M <= 256) return kSmallCol256;
  if (N == 1 && M <= 512) return kSmallCol512;
  return kSmallNone;
}

double small_output_tile(int cfg) {
  switch (cfg) {
    case kSmall6: return 36.0;
    case kSmall8: return 64.0;
    case kSmall10: return 100.0;
    case kSmall16: return 256.0;
    case kSmall20: return 400.0;
    case kSmall24: return 576.0;
    case kSmall32: return 1024.0;
    case kSmall80: return 6400.0;
    case kSmall96: return 9216.0;
    case kSmall40: return 1600.0;
    case kSmall48: return 2304.0;
    case kSmall64: return 4096.0;
    case kSmallCol256: return 256.0;
    case kSmallCol512: return 512.0;
    default: return 0.0;
  }
}

int small_output_bk(int cfg, int elem_bytes) {
  const bool d = elem_bytes == 16;
  switch (cfg) {
    case kSmall6: return d ? SmallShape<double, 2, 1, 3, 6>::BK : SmallShape<float, 2, 1, 3, 6>::BK;
    case kSmall8: return d ? SmallShape<double, 2, 2, 4, 4>::BK : SmallShape<float, 2, 2, 4, 4>::BK;
    case kSmall10: return d ? SmallShape<double, 2, 2, 5, 5>::BK : SmallShape<float, 2, 2, 5, 5>::BK;
    case kSmall16: return d ? SmallShape<double, 4, 4, 4, 4>::BK : SmallShape<float, 4, 4, 4, 4>::BK;
    case kSmall20: return d ? SmallShape<double, 4, 4, 5, 5>::BK : SmallShape<float, 4, 4, 5, 5>::BK;
    case kSmall24: return d ? SmallShape<double, 8, 8, 3, 3>::BK : SmallShape<float, 8, 8, 3, 3>::BK;
    case kSmall32: return d ? SmallShape<double, 8, 8, 4, 4>::BK : SmallShape<float, 8, 8, 4, 4>::BK;
    case kSmall80: return d ? SmallShape<double, 16, 16, 5, 5>::BK : SmallShape<float, 16, 16, 5, 5>::BK;
    case kSmall96: return d ? SmallShape<double, 16, 16, 6, 6>::BK : SmallShape<float, 16, 16, 6, 6>::BK;
    case kSmall40: return d ? SmallShape<double, 8, 8, 5, 5>::BK : SmallShape<float, 8, 8, 5, 5>::BK;
    case kSmall48: return d ? SmallShape<double, 16, 16, 3, 3>::BK : SmallShape<float, 16, 16, 3, 3>::BK;
    case kSmall64: return d ? SmallShape<double, 16, 16, 4, 4>::BK : SmallShape<float, 16, 16, 4, 4>::BK;
    case kSmallCol256: return d ? SmallShape<double, 64, 1, 4, 1>::BK : SmallShape<float, 64, 1, 4, 1>::BK;
    case kSmallCol512: return d ? SmallShape<double, 128, 1, 4, 1>::BK : SmallShape<float, 128, 1, 4, 1>::BK;
    default: return 0;
  }
}

template <typename R>
void launch_reduce_small(int cfg, bool a_kc, bool b_kc, const Cx<R>* A, long long aoff,
                         const long long* aM, const long long* aK, const Cx<R>* B, long long boff,
                         const long long* bN, const long long* bK, Cx<R>* C, long long coff,
                         const long long* cM, const long long* cN, int M, int N, int K, int nsplit,
                         int kchunk, double alpha, bool accumulate, Cx<R>* part, cudaStream_t s) {
  switch (cfg) {
    case kSmall6:
      launch_cfg<R, 2, 1, 3, 6>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K,
                                nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmall8:
      launch_cfg<R, 2, 2, 4, 4>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K,
                                nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmall10:
      launch_cfg<R, 2, 2, 5, 5>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K,
                                nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmall20:
      launch_cfg<R, 4, 4, 5, 5>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K,
                                nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmall24:
      launch_cfg<R, 8, 8, 3, 3>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K,
                                nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmall32:
      launch_cfg<R, 8, 8, 4, 4>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K,
                                nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmall80:
      launch_cfg<R, 16, 16, 5, 5>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K,
                                nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmall96:
      launch_cfg<R, 16, 16, 6, 6>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K,
                                nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmall40:
      launch_cfg<R, 8, 8, 5, 5>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K,
                                nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmall16:
      launch_cfg<R, 4, 4, 4, 4>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K,
                                nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmall48:
      launch_cfg<R, 16, 16, 3, 3>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N,
                                  K, nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmall64:
      launch_cfg<R, 16, 16, 4, 4>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N,
                                  K, nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmallCol256:
      launch_cfg<R, 64, 1, 4, 1>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N, K,
                                 nsplit, kchunk, alpha, accumulate, part, s);
      break;
    case kSmallCol512:
      launch_cfg<R, 128, 1, 4, 1>(a_kc, b_kc, A, aoff, aM, aK, B, boff, bN, bK, C, coff, cM, cN, M, N,
                                  K, nsplit, kchunk, alpha, accumulate, part, s);
      break;
    default:
      throw Error(kErrArg, "reduce_small: unsupported output shape");
  }
}

template <typename R>
void launch_gemv(bool a_kc, const Cx<R>* A, long long aoff, const long long* aM, const long long* aK,
                 const Cx<R>* B, long long boff, const long long* bK, Cx<R>* C, long long coff,
                 const long long* cM, int M, int K, double alpha, bool accumulate, cudaStream_t s) {
  const long long units = a_kc ? (long long)M * 32 : (long long)M;
  const int grid = int(std::max<long long>(1, std::min<long long>((units + kThreads - 1) / kThreads,
                                                                   152LL * 16)));
  if (a_kc)
    k_gemv<R, true><<<grid, kThreads, 0, s>>>(A, aoff, aM, aK, B, boff, bK, C, coff, cM, M, K, R(alpha),
                                              accumulate ? 1 : 0);
  else
    k_gemv<R, false><<<grid, kThreads, 0, s>>>(A, aoff, aM, aK, B, boff, bK, C, coff, cM, M, K, R(alpha),
                                               accumulate ? 1 : 0);
  RTCC3_CUDA(cudaGetLastError());
}

#define RTCC3_INST(R)                                                                              \
  template void launch_reduce_small<R>(int, bool, bool, const Cx<R>*, long long, const long long*,  \
                                       const long long*, const Cx<R>*, long long, const long long*, \
                                       const long long*, Cx<R>*, long long, const long long*,       \
                                       const long long*, int, int, int, int, int, double, bool,     \
                                       Cx<R>*, cudaStream_t);                                       \
  template void launch_gemv<R>(bool, const Cx<R>*, long long, const long long*, const long long*,   \
                               const Cx<R>*, long long, const long long*, Cx<R>*, long long,        \
                               const long long*, int, int, double, bool, cudaStream_t);         \
  template void launch_outer<R>(const Cx<R>*, long long, const long long*, const long long*,       \
                                const Cx<R>*, long long, const long long*, const long long*,       \
                                Cx<R>*, long long, const long long*, const long long*, int, int,   \
                                double, bool, cudaStream_t);
RTCC3_INST(float)
RTCC3_INST(double)
#undef RTCC3_INST

void fine_split(long long outputs, long long K, int* ls_log, bool* block_wide) {
  // fewer than about 8 warps' worth of outputs per SM and a long sum: a block
  // each; else lanes until the GPU is covered (1024 lanes per SM) or a lane
  // holds at most four terms
  *block_wide = outputs * 32 < 152 * 256 && K >= 512;
  int l = 0;
  while (l < 5 && (outputs << l) < 152LL * 1024 && (K >> l) > 4) ++l;
  *ls_log = l;
}

template <typename R>
void launch_fine(const FineArgs<R>& a, cudaStream_t s) {
  const long long total = (long long)a.M * a.N * a.nb;
  if (a.block_wide) {
    k_contract_fine_block<R><<<unsigned(total), 256, 0, s>>>(a);
  } else {
    const long long lanes = total << a.ls_log;
    k_contract_fine<R><<<unsigned((lanes + 127) / 128), 128, 0, s>>>(a, unsigned(total));
  }
  RTCC3_CUDA(cudaGetLastError());
}

template void launch_fine<float>(const FineArgs<float>&, cudaStream_t);
template void launch_fine<double>(const FineArgs<double>&, cudaStream_t);

}  // namespace rtcc3
