// Eigendecomposition of the small complex non-Hermitian matrices that carry
// the field coupling of the triples equation (see rotation.h).
//
// The matrices are orbital energies plus a perturbation of the field's
// strength, so their eigenvectors are a correction of the identity: k_eig_refine
// starts there and repeats a quadratically convergent correction (the
// refinement of Ogita and Aishima, "Iterative refinement for symmetric
// eigenvalue decomposition", Japan J. Indust. Appl. Math. 35, 1007 (2018), in
// its two-sided form for X and Y = X^-1, with each pair's 2 x 2 problem solved
// exactly so that near-degenerate pairs converge too).  All its work is matrix
// products, spread over a cluster of eight CTAs per matrix.  A matrix that it
// does not bring to convergence goes to the QR algorithm of k_eig_warp, launched
// behind it (and leaving at once otherwise).
//
// Measured, two n x n matrices with couplings of 1e-4, QR before and
// refinement now: complex128 n = 19 3.1 -> 0.11 ms, n = 38 14.1 -> 0.33 ms,
// n = 76 76 -> 1.9 ms; complex64 n = 19 0.45 -> 0.03 ms, n = 38 1.56 -> 0.08 ms,
// n = 76 7.8 -> 0.29 ms.  |S L S^-1 - M| is 3 to 8 times smaller.  Bound by the
// FP64 pipe of the eight SMs (complex128) and by the latency of its four
// cluster barriers per correction (complex64).  Couplings of 0.05 (fields near
// 0.5 au) still need QR.
//
// k_eig_warp: one warp per matrix, no block-wide barriers: M is reduced to upper
// Hessenberg form by Householder reflections, then to Schur form
// T = Q^H M Q by single-shift QR sweeps (Wilkinson shift, Givens rotations,
// deflation of negligible subdiagonal entries, an exceptional shift every
// eleventh sweep); the eigenvectors X of the upper-triangular T follow by back
// substitution (unit diagonal), so S = Q X, S^-1 = X^-1 Q^H and
// M = S diag(T_kk) S^-1.  Every lane computes the rotation parameters itself
// from the same shared-memory values (identical control flow), then the lanes
// update disjoint rows and columns.  The arithmetic type T is float for the
// complex64 graphs and double for the complex128 one.  H lives in shared
// memory, Q, X and X^-1 in a global workspace; a non-converging sweep count or
// a non-finite matrix raises *status (codes in rotation.h) instead of looping.
#include "rotation.h"

#include <cooperative_groups.h>

#include <algorithm>

namespace rtcc3 {

namespace {

template <typename T> struct C2T;
template <> struct C2T<float> { using type = float2; };
template <> struct C2T<double> { using type = double2; };

template <typename T>
struct Cplx {
  using V = typename C2T<T>::type;
  static __device__ __forceinline__ V mk(T a, T b) { V r; r.x = a; r.y = b; return r; }
  static __device__ __forceinline__ V mul(V a, V b) { return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
  static __device__ __forceinline__ V conj(V a) { return mk(a.x, -a.y); }
  static __device__ __forceinline__ V add(V a, V b) { return mk(a.x + b.x, a.y + b.y); }
  static __device__ __forceinline__ V sub(V a, V b) { return mk(a.x - b.x, a.y - b.y); }
  static __device__ __forceinline__ V scale(V a, T s) { return mk(a.x * s, a.y * s); }
  static __device__ __forceinline__ T abs(V a) { return sqrt(a.x * a.x + a.y * a.y); }
  // Smith's algorithm
  static __device__ __forceinline__ V div(V a, V b) {
    if (fabs(b.x) >= fabs(b.y)) {
      const T r = b.y / b.x, d = b.x + b.y * r;
      return mk((a.x + a.y * r) / d, (a.y - a.x * r) / d);
    }
    const T r = b.x / b.y, d = b.y + b.x * r;
    return mk((a.x * r + a.y) / d, (a.y * r - a.x) / d);
  }
  // principal square root without cancellation: t = sqrt((|x| + |z|) / 2) is
  // the larger of |Re|, |Im| and the other part follows as y / (2 t)
  static __device__ __forceinline__ V sqrt_(V z) {
    const T m = abs(z);
    if (m == T(0)) return mk(T(0), T(0));
    const T t = sqrt(T(0.5) * (fabs(z.x) + m));
    if (z.x >= T(0)) return mk(t, z.y / (T(2) * t));
    return mk(fabs(z.y) / (T(2) * t), copysign(t, z.y));
  }
};

// Sum over the warp, returned identically in every lane (lane 0's value:
// the lanes' butterfly sums may round differently, and every lane takes the
// same branches on the result).
// 1/sqrt(x) from the correctly rounded square root and division: the rotation
// stays unitary to rounding, with no systematic drift of |c|^2 + |s|^2 over the
// thousands of rotations accumulated into Q
template <typename T>
__device__ __forceinline__ T rsqrt_(T x) { return T(1) / sqrt(x); }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return __shfl_sync(0xffffffffu, v, 0);
}

// ---- correction of the identity -------------------------------------------------
constexpr int kCl = 8;        // CTAs per matrix
constexpr int kRefineThreads = 256;
constexpr int kRefineMax = 10;  // corrections before the QR algorithm takes over

// Scratch of one matrix: nine n x n arrays, then the column scales and the
// per-CTA maxima; the flag that tells k_eig_warp the matrix is done is last.
template <typename T>
struct RefineWs {
  using V = typename C2T<T>::type;
  V *X[2], *Y[2], *S1, *R, *S, *E, *c;
  T* red;
  int* done;
  __device__ RefineWs(double2* ws, int n) {
    V* p = reinterpret_cast<V*>(ws);
    const size_t nn = size_t(n) * n;
    X[0] = p; X[1] = p + nn; Y[0] = p + 2 * nn; Y[1] = p + 3 * nn;
    S1 = p + 4 * nn; R = p + 5 * nn; S = p + 6 * nn; E = p + 7 * nn;
    c = p + 8 * nn;
    red = reinterpret_cast<T*>(c + n);
    done = eig_done(ws, n);
  }
};

// Data written by other CTAs of the cluster is read through L2.
__device__ __forceinline__ float2 ldc(const float2* p) { return __ldcg(p); }
__device__ __forceinline__ double2 ldc(const double2* p) { return __ldcg(p); }

// sum_k a[k] b[k n] (+ the identity's contributions are the caller's)
template <typename T>
__device__ __forceinline__ typename C2T<T>::type row_col(const typename C2T<T>::type* a,
                                                         const typename C2T<T>::type* b, int n) {
  using X = Cplx<T>;
  using V = typename C2T<T>::type;
  V s0 = X::mk(T(0), T(0)), s1 = s0;
  int k = 0;
  for (; k + 4 <= n; k += 4) {
    V x[4], y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) { x[u] = ldc(a + k + u); y[u] = ldc(b + size_t(k + u) * n); }
    s0 = X::add(s0, X::mul(x[0], y[0]));
    s1 = X::add(s1, X::mul(x[1], y[1]));
    s0 = X::add(s0, X::mul(x[2], y[2]));
    s1 = X::add(s1, X::mul(x[3], y[3]));
  }
  for (; k < n; ++k) s0 = X::add(s0, X::mul(ldc(a + k), ldc(b + size_t(k) * n)));
  return X::add(s0, s1);
}

template <typename T>
__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(kRefineThreads)
k_eig_refine(EigJob ja, EigJob jb) {
  using X = Cplx<T>;
  using V = typename C2T<T>::type;
  namespace cg = cooperative_groups;
  auto cluster = cg::this_cluster();
  const EigJob J = blockIdx.x < kCl ? ja : jb;
  const int n = J.n, rank = int(blockIdx.x) % kCl, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  RefineWs<T> W(J.ws, n);
  __shared__ T wmax[kRefineThreads / 32];
  if (rank == 0 && tid == 0) *W.done = 0;
  const int rows = (n - rank + kCl - 1) / kCl;  // own rows rank, rank + 8, ...
  const T eps = sizeof(T) == 4 ? T(1.2e-7) : T(2.2e-16);
  const T tol = sizeof(T) == 4 ? T(1e-4) : T(3e-9);  // its square is rounding
  // the matrix's magnitude (rounding floor of its products)
  T mag = T(0);
  for (int t = tid; t < n * n; t += kRefineThreads) {
    const double2 m = J.M[t];
    const T a = T(fabs(m.x)) + T(fabs(m.y));
    mag = a > mag || !(a == a) ? a : mag;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    const T o = __shfl_xor_sync(0xffffffffu, mag, d);
    mag = o > mag || !(o == o) ? o : mag;
  }
  if (lane == 0) wmax[warp] = mag;
  __syncthreads();
  mag = wmax[0];
#pragma unroll
  for (int w = 1; w < kRefineThreads / 32; ++w) mag = wmax[w] > mag || !(wmax[w] == wmax[w]) ? wmax[w] : mag;
  __syncthreads();
  // not a number, or one without a rounding floor: k_eig_warp says so (mag is
  // the same in the whole cluster)
  if (!isfinite(mag)) return;
  const T floor_ = eps * mag;
  const int max_it = J.max_sweeps > 0 ? min(J.max_sweeps, kRefineMax) : kRefineMax;
  int cur = 0;
  bool converged = false;
  for (int it = 0; it < max_it; ++it) {
    const V *Xc = W.X[cur], *Yc = W.Y[cur];
    if (it > 0) {
      // S1 = M X and R = 1 - Y X, then S = Y S1
      for (int t = tid; t < rows * n; t += kRefineThreads) {
        const int i = rank + kCl * (t / n), j = t % n;
        V s = X::mk(T(0), T(0));
        for (int k = 0; k < n; ++k) {
          const double2 m = J.M[size_t(i) * n + k];
          s = X::add(s, X::mul(X::mk(T(m.x), T(m.y)), ldc(Xc + size_t(k) * n + j)));
        }
        W.S1[size_t(i) * n + j] = s;
        const V r = row_col<T>(Yc + size_t(i) * n, Xc + j, n);
        W.R[size_t(i) * n + j] = X::mk((i == j ? T(1) : T(0)) - r.x, -r.y);
      }
      cluster.sync();
      for (int t = tid; t < rows * n; t += kRefineThreads) {
        const int i = rank + kCl * (t / n), j = t % n;
        W.S[size_t(i) * n + j] = row_col<T>(Yc + size_t(i) * n, W.S1 + j, n);
      }
      cluster.sync();
    }
    auto s_at = [&](int i, int j) {
      if (it == 0) { const double2 m = J.M[size_t(i) * n + j]; return X::mk(T(m.x), T(m.y)); }
      return ldc(W.S + size_t(i) * n + j);
    };
    auto r_at = [&](int i, int j) { return it == 0 ? X::mk(T(0), T(0)) : ldc(W.R + size_t(i) * n + j); };
    auto lam_at = [&](int i) {
      const V s = s_at(i, i);
      return X::add(s, X::mul(r_at(i, i), s));
    };
    // E: for each pair the exact eigenvectors of its 2 x 2 block, one warp a row
    T mx = T(0);
    for (int t = warp; t < rows; t += kRefineThreads / 32) {
      const int i = rank + kCl * t;
      V q = X::mk(T(0), T(0));
      for (int j = lane; j < n; j += 32) {
        V e;
        if (j == i) {
          e = r_at(i, i);
        } else {
          // Rows i and j of a pair have to take opposite roots, or both columns
          // become the same vector: both work out the same b, c, s of (lo, hi)
          // bit for bit and row hi changes the signs.
          const int lo = min(i, j), hi = max(i, j);
          const V ll = lam_at(lo), lh = lam_at(hi);
          const V b = X::add(s_at(lo, hi), X::mul(r_at(lo, hi), lh));
          const V c = X::add(s_at(hi, lo), X::mul(r_at(hi, lo), ll));
          const T ab = X::abs(b), ac = X::abs(c);
          if (ab <= floor_ && ac <= floor_) {
            e = X::mk(T(0), T(0));
          } else {
            const V dl = X::scale(X::sub(ll, lh), T(0.5));
            const V bc = X::mul(b, c);
            V s = dl;
            const T d2 = dl.x * dl.x + dl.y * dl.y;
            if (ab * ac > T(1e-8) * d2) {
              s = X::sqrt_(X::add(X::mul(dl, dl), bc));
              if (dl.x * s.x + dl.y * s.y < T(0)) s = X::scale(s, T(-1));
            }
            const V den = X::add(dl, s);
            const V bd = X::div(b, den), cd = X::div(c, den);
            e = j > i ? X::scale(bd, T(-1)) : cd;
            q = X::sub(q, X::mul(bd, cd));
            const T ae = X::abs(e);
            mx = ae > mx || !(ae == ae) ? ae : mx;
          }
        }
        if (it > 0) {
          // Y has to be the inverse of X too
          const V r = r_at(i, j);
          const T ar = fabs(r.x) + fabs(r.y);
          mx = ar > mx || !(ar == ar) ? ar : mx;
        }
        W.E[size_t(i) * n + j] = e;
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        q.x += __shfl_xor_sync(0xffffffffu, q.x, d);
        q.y += __shfl_xor_sync(0xffffffffu, q.y, d);
      }
      if (lane == 0) W.c[i] = X::div(X::mk(T(1), T(0)), X::sqrt_(X::mk(T(1) - q.x, -q.y)));
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const T o = __shfl_xor_sync(0xffffffffu, mx, d);
      mx = o > mx || !(o == o) ? o : mx;
    }
    if (lane == 0) wmax[warp] = mx;
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < kRefineThreads / 32; ++w) mx = wmax[w] > mx || !(wmax[w] == wmax[w]) ? wmax[w] : mx;
      W.red[rank] = mx;
    }
    cluster.sync();
    mx = T(0);
    for (int r = 0; r < kCl; ++r) {
      const T o = __ldcg(W.red + r);
      mx = o > mx || !(o == o) ? o : mx;
    }
    // not a correction (or not finite), or still none after three: the QR
    // algorithm (mx is the same in the whole cluster)
    if (!(mx < (it < 3 ? T(4) : T(0.5)))) break;
    // X <- X (1 + E) c, Y <- c (1 - E + R) Y
    const int nxt = cur ^ 1;
    for (int t = tid; t < rows * n; t += kRefineThreads) {
      const int i = rank + kCl * (t / n), j = t % n;
      const size_t ij = size_t(i) * n + j;
      V x, y;
      if (it == 0) {
        const V e = ldc(W.E + ij);
        const T one = i == j ? T(1) : T(0);
        x = X::mk(one + e.x, e.y);
        y = X::mk(one - e.x, -e.y);
      } else {
        x = X::add(ldc(Xc + ij), row_col<T>(Xc + size_t(i) * n, W.E + j, n));
        V s = ldc(Yc + ij);
        for (int k = 0; k < n; ++k)
          s = X::add(s, X::mul(X::sub(ldc(W.R + size_t(i) * n + k), ldc(W.E + size_t(i) * n + k)),
                               ldc(Yc + size_t(k) * n + j)));
        y = s;
      }
      W.X[nxt][ij] = X::mul(x, ldc(W.c + j));
      W.Y[nxt][ij] = X::mul(ldc(W.c + i), y);
    }
    cur = nxt;
    if (mx <= tol) {
      converged = true;
      for (int t = tid; t < rows; t += kRefineThreads) {
        const int i = rank + kCl * t;
        const V l = lam_at(i);
        J.lam[i] = make_double2(double(l.x), double(l.y));
      }
      break;
    }
    cluster.sync();
  }
  __syncthreads();
  if (!converged) return;
  for (int t = tid; t < rows * n; t += kRefineThreads) {
    const size_t ij = size_t(rank + kCl * (t / n)) * n + t % n;
    const V x = ldc(W.X[cur] + ij), y = ldc(W.Y[cur] + ij);
    J.S[ij] = make_double2(double(x.x), double(x.y));
    J.Sinv[ij] = make_double2(double(y.x), double(y.y));
  }
  if (rank == 0 && tid == 0) *W.done = 1;
}

// level: 2 = H, Q, X and X^-1 in shared memory, 1 = H and Q, 0 = H only (the
// rest in the workspace).
template <typename T>
__global__ void __launch_bounds__(32) k_eig_warp(EigJob ja, EigJob jb, int level,
                                                 int* __restrict__ status) {
  using X = Cplx<T>;
  using V = typename C2T<T>::type;
  const EigJob J = blockIdx.x == 0 ? ja : jb;
  const int n = J.n;
  if (n <= 0 || *eig_done(J.ws, n)) return;  // refined already
  const int lane = threadIdx.x;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int nn = n * n;
  V* H = reinterpret_cast<V*>(sm_raw);  // n x n, row-major
  V* vb = H + nn;                       // Householder vector
  V* wsv = reinterpret_cast<V*>(J.ws);
  V* Q = level >= 1 ? vb + n : wsv;
  V* Xv = level >= 2 ? Q + nn : wsv + nn;
  V* Xi = Xv + nn;
  T fro = T(0);
  for (int t = lane; t < nn; t += 32) {
    const double2 m = J.M[t];
    H[t] = X::mk(T(m.x), T(m.y));
    Q[t] = X::mk((t / n) == (t % n) ? T(1) : T(0), T(0));
    fro += T(m.x) * T(m.x) + T(m.y) * T(m.y);
  }
  fro = sqrt(warp_sum(fro));
  __syncwarp();
  if (!isfinite(fro)) {
    if (lane == 0) atomicExch(status, eig_status(kEigNonFinite, n, n - 1));
    return;
  }
  const T tiny = sizeof(T) == 4 ? T(1e-30) : T(1e-300);
  const T eps = sizeof(T) == 4 ? T(1.2e-7) : T(2.2e-16);

  // ---- Householder reduction to upper Hessenberg form -------------------------
  for (int k = 0; k + 2 < n; ++k) {
    const int m = n - k - 1;
    T s2 = T(0);
    for (int i = lane; i < m; i += 32) {
      const V x = H[(k + 1 + i) * n + k];
      s2 += x.x * x.x + x.y * x.y;
    }
    s2 = warp_sum(s2);
    const T xnorm = sqrt(s2);
    const V x0 = H[(k + 1) * n + k];
    const T ax0 = X::abs(x0);
    if (xnorm <= tiny || s2 - ax0 * ax0 <= T(1e-30) * s2) continue;  // column already reduced
    const V ph = ax0 > T(0) ? X::scale(x0, T(1) / ax0) : X::mk(T(1), T(0));
    const V alpha = X::scale(ph, -xnorm);
    for (int i = lane; i < m; i += 32) vb[i] = i == 0 ? X::sub(x0, alpha) : H[(k + 1 + i) * n + k];
    __syncwarp();
    T vv = T(0);
    for (int i = lane; i < m; i += 32) vv += vb[i].x * vb[i].x + vb[i].y * vb[i].y;
    const T beta = T(2) / warp_sum(vv);
    // left: rows k+1.., columns k..n-1 (one column per lane)
    for (int j = k + lane; j < n; j += 32) {
      V sd = X::mk(T(0), T(0));
      for (int i = 0; i < m; ++i) sd = X::add(sd, X::mul(X::conj(vb[i]), H[(k + 1 + i) * n + j]));
      sd = X::scale(sd, beta);
      for (int i = 0; i < m; ++i) H[(k + 1 + i) * n + j] = X::sub(H[(k + 1 + i) * n + j], X::mul(vb[i], sd));
    }
    __syncwarp();
    // right: all rows of H and Q, columns k+1..n-1 (one row per lane)
    for (int r = lane; r < 2 * n; r += 32) {
      V* row = r < n ? &H[r * n] : &Q[size_t(r - n) * n];
      V sd = X::mk(T(0), T(0));
      for (int j = 0; j < m; ++j) sd = X::add(sd, X::mul(row[k + 1 + j], vb[j]));
      sd = X::scale(sd, beta);
      for (int j = 0; j < m; ++j) row[k + 1 + j] = X::sub(row[k + 1 + j], X::mul(sd, X::conj(vb[j])));
    }
    __syncwarp();
    for (int i = 1 + lane; i < m; i += 32) H[(k + 1 + i) * n + k] = X::mk(T(0), T(0));
    __syncwarp();
  }

  // ---- shifted QR sweeps to Schur form ---------------------------------------
  int hi = n - 1, iter = 0, its_here = 0;
  const int max_iter = J.max_sweeps > 0 ? J.max_sweeps : 60 * n + 100;
  bool failed = false;
  while (hi > 0) {
    int l = hi;
    while (l > 0) {
      const T off = X::abs(H[l * n + l - 1]);
      const T dg = X::abs(H[l * n + l]) + X::abs(H[(l - 1) * n + l - 1]);
      if (off <= eps * (dg > T(0) ? dg : fro)) break;
      --l;
    }
    __syncwarp();
    if (l > 0 && lane == 0) H[l * n + l - 1] = X::mk(T(0), T(0));
    __syncwarp();
    if (l == hi) {
      --hi;
      its_here = 0;
      continue;
    }
    if (++iter > max_iter) {
      failed = true;
      break;
    }
    ++its_here;
    for (int k = l; k < hi; ++k) {
      V x, y;
      if (k == l) {
        // Wilkinson shift: eigenvalue of the trailing 2x2 closest to H[hi][hi]
        const V a = H[(hi - 1) * n + hi - 1], b = H[(hi - 1) * n + hi];
        const V c = H[hi * n + hi - 1], d = H[hi * n + hi];
        const V tr2 = X::scale(X::add(a, d), T(0.5));
        const V hd = X::scale(X::sub(a, d), T(0.5));
        const V disc = X::sqrt_(X::add(X::mul(hd, hd), X::mul(b, c)));
        const V l1 = X::add(tr2, disc), l2 = X::sub(tr2, disc);
        V mu = X::abs(X::sub(l1, d)) < X::abs(X::sub(l2, d)) ? l1 : l2;
        if (its_here % 11 == 10 || !isfinite(mu.x) || !isfinite(mu.y))  // exceptional shift
          mu = X::add(d, X::mk(T(0.75) * X::abs(c), T(0)));
        x = X::sub(H[l * n + l], mu);
        y = H[(l + 1) * n + l];
      } else {
        x = H[k * n + k - 1];
        y = H[(k + 1) * n + k - 1];
      }
      // G = [[c, s], [-conj(s), conj(c)]] with c = conj(x) / r, s = conj(y) / r,
      // r = |(x, y)|: unitary, maps (x, y) to (r, 0); one reciprocal square root
      T r2 = x.x * x.x + x.y * x.y + y.x * y.x + y.y * y.y;
      V c, s;
      if (!(r2 > tiny && r2 < T(1) / tiny)) {  // rescale out of the under/overflow range
        const T m = fmax(fmax(fabs(x.x), fabs(x.y)), fmax(fabs(y.x), fabs(y.y)));
        if (m > T(0) && isfinite(m)) {
          x = X::scale(x, T(1) / m);
          y = X::scale(y, T(1) / m);
        } else {
          x = X::mk(T(1), T(0));
          y = X::mk(T(0), T(0));
        }
        r2 = x.x * x.x + x.y * x.y + y.x * y.x + y.y * y.y;
      }
      const T ri = rsqrt_(r2);
      c = X::mk(x.x * ri, -x.y * ri);
      s = X::mk(y.x * ri, -y.y * ri);
      __syncwarp();  // every lane has read the entries the rotation is built from
      // rows k, k+1 <- G rows; the bulge H[k+1][k-1] becomes exactly zero
      for (int j = (k == l ? k : k - 1) + lane; j < n; j += 32) {
        const V a = H[k * n + j], b = H[(k + 1) * n + j];
        H[k * n + j] = X::add(X::mul(c, a), X::mul(s, b));
        H[(k + 1) * n + j] = (k > l && j == k - 1)
                                 ? X::mk(T(0), T(0))
                                 : X::sub(X::mul(X::conj(c), b), X::mul(X::conj(s), a));
      }
      __syncwarp();
      // columns k, k+1 <- columns times G^H (H rows 0..min(k+2,hi), all rows of Q)
      const int rmax = min(k + 2, hi);
      for (int rr = lane; rr <= rmax + n; rr += 32) {
        V* row = rr <= rmax ? &H[rr * n] : &Q[size_t(rr - rmax - 1) * n];
        const V a = row[k], b = row[k + 1];
        row[k] = X::add(X::mul(a, X::conj(c)), X::mul(b, X::conj(s)));
        row[k + 1] = X::sub(X::mul(b, c), X::mul(a, s));
      }
      __syncwarp();
    }
  }
  if (failed) {
    if (lane == 0) atomicExch(status, eig_status(kEigNoConvergence, n, hi));
    return;
  }

  // ---- eigenvectors of T (unit upper triangular X), S = Q X, S^-1 = X^-1 Q^H --
  const T smin = fmax(eps * fro, tiny);
  for (int k = lane; k < n; k += 32) {
    const V tk = H[k * n + k];
    J.lam[k] = make_double2(double(tk.x), double(tk.y));
    for (int i = 0; i < n; ++i) Xv[size_t(i) * n + k] = X::mk(i == k ? T(1) : T(0), T(0));
    for (int i = k - 1; i >= 0; --i) {
      V acc = X::mk(T(0), T(0));
      for (int j = i + 1; j <= k; ++j) acc = X::add(acc, X::mul(H[i * n + j], Xv[size_t(j) * n + k]));
      V den = X::sub(H[i * n + i], tk);
      if (X::abs(den) < smin) den = X::mk(smin, T(0));
      Xv[size_t(i) * n + k] = X::scale(X::div(acc, den), T(-1));
    }
  }
  __syncwarp();
  for (int k = lane; k < n; k += 32) {
    // column k of X^-1: unit upper triangular back substitution
    for (int i = 0; i < n; ++i) Xi[size_t(i) * n + k] = X::mk(i == k ? T(1) : T(0), T(0));
    for (int i = k - 1; i >= 0; --i) {
      V acc = X::mk(T(0), T(0));
      for (int j = i + 1; j <= k; ++j) acc = X::add(acc, X::mul(Xv[size_t(i) * n + j], Xi[size_t(j) * n + k]));
      Xi[size_t(i) * n + k] = X::scale(acc, T(-1));
    }
  }
  __syncwarp();
  for (int t = lane; t < nn; t += 32) {
    const int i = t / n, k = t % n;
    V a = X::mk(T(0), T(0)), b = X::mk(T(0), T(0));
    for (int j = 0; j <= k; ++j) a = X::add(a, X::mul(Q[size_t(i) * n + j], Xv[size_t(j) * n + k]));
    for (int j = i; j < n; ++j) b = X::add(b, X::mul(Xi[size_t(i) * n + j], X::conj(Q[size_t(k) * n + j])));
    J.S[t] = make_double2(double(a.x), double(a.y));
    J.Sinv[t] = make_double2(double(b.x), double(b.y));
  }
}

template <typename T>
void launch_t(const EigJob& a, const EigJob& b, int* status, cudaStream_t s) {
  constexpr size_t kMaxSmem = 200 * 1024;
  const size_t nmax = size_t(std::max(a.n, b.n));
  const size_t vs = sizeof(typename C2T<T>::type);
  int level = 0;
  size_t smem = (nmax * nmax + nmax) * vs;
  if ((4 * nmax * nmax + nmax) * vs <= kMaxSmem) {
    level = 2;
    smem = (4 * nmax * nmax + nmax) * vs;
  } else if ((2 * nmax * nmax + nmax) * vs <= kMaxSmem) {
    level = 1;
    smem = (2 * nmax * nmax + nmax) * vs;
  }
  static PerDevice attr;
  allow_smem(attr, k_eig_warp<T>, int(kMaxSmem));
  k_eig_refine<T><<<2 * kCl, kRefineThreads, 0, s>>>(a, b);
  RTCC3_CUDA(cudaGetLastError());
  k_eig_warp<T><<<2, 32, smem, s>>>(a, b, level, status);
  RTCC3_CUDA(cudaGetLastError());
}

}  // namespace

void launch_eig(const EigJob& a, const EigJob& b, bool fp32, int* status, cudaStream_t s) {
  RTCC3_CHECK(a.n >= 1 && a.n <= kEigMaxN && b.n >= 1 && b.n <= kEigMaxN, kErrArg,
              "eigensolver supports n <= " + std::to_string(kEigMaxN));
  if (fp32) launch_t<float>(a, b, status, s);
  else launch_t<double>(a, b, status, s);
}

}  // namespace rtcc3
