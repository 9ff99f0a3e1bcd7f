// Contractions whose output is small or a single column, where the generic
// 64 x 64 tiled kernel wastes most of its tile and re-reads the long operand.
//
//   reduce_small: C[m,n] = sum_k A[m,k] B[n,k] with the whole M x N output held
//     by every CTA (M, N <= 96, or N = 1 and M <= 512); each CTA sums one K
//     chunk, so both operands stream from HBM exactly once.  Used for the
//     triples slot densities (ijkabc,ijkdbc->ad; ijkabc,ljkabc->li) and the
//     X1-type back-contractions (ijkabc,jkbc->ia).
//   gemv: C[m] = sum_k A[m,k] B[k] for a long output column (M > 512): one
//     warp per output when A is contiguous along k, else one thread per output
//     with consecutive threads on consecutive m.
// Addresses come from the contraction's offset tables (element offsets):
// A[aoff + aM[m] + aK[k]], B[boff + bN[n] + bK[k]], C[coff + cM[m] + cN[n]].
#pragma once

#include "common.h"

namespace rtcc3 {

// Output-tile configurations of reduce_small (0 = not applicable).
enum SmallCfg : int {
  kSmallNone = 0, kSmall48 = 1, kSmall16 = 2, kSmallCol256 = 3, kSmallCol512 = 4, kSmall64 = 5,
  kSmall10 = 6, kSmall40 = 7, kSmall6 = 8, kSmall8 = 9,
  kSmall20 = 10, kSmall24 = 11, kSmall32 = 12, kSmall80 = 13, kSmall96 = 14
};

// Configuration for an M x N output (N <= M expected; returns kSmallNone
// when the shape is not small).
int small_output_config(long long M, long long N);
// Outputs of a configuration's tile (what it computes, padding included).
double small_output_tile(int cfg);
// Depth of one K slice for a configuration (chunks are multiples of it).
int small_output_bk(int cfg, int elem_bytes);

// nsplit > 1: CTA s sums K range [s kchunk, (s+1) kchunk) into
// part[m][n][s] and a second kernel adds the splits in a fixed order into C
// (deterministic); nsplit == 1: C (+)= alpha * result directly.
template <typename R>
void launch_reduce_small(int cfg, bool a_kc, bool b_kc, const Cx<R>* A, long long aoff,
                         const long long* aM, const long long* aK, const Cx<R>* B, long long boff,
                         const long long* bN, const long long* bK, Cx<R>* C, long long coff,
                         const long long* cM, const long long* cN, int M, int N, int K, int nsplit,
                         int kchunk, double alpha, bool accumulate, Cx<R>* part, cudaStream_t s);

// Outer products (K = 1): C[coff + cM[m] + cN[n]] (+)= alpha A[aoff + aM[m] +
// aK[0]] B[boff + bN[n] + bK[0]], n along the output's contiguous index: a
// streaming pass over C (the reverse-pass products that spread a vector over
// the o^3 v^3 cotangent).
template <typename R>
void launch_outer(const Cx<R>* A, long long aoff, const long long* aM, const long long* aK,
                  const Cx<R>* B, long long boff, const long long* bN, const long long* bK,
                  Cx<R>* C, long long coff, const long long* cM, const long long* cN, int M, int N,
                  double alpha, bool accumulate, cudaStream_t s);

// Small products of any shape, spread over the whole GPU: 2^ls_log lanes of a
// warp (or, block_wide, one block of 256 threads) share one output, each
// summing every 2^ls_log-th k, joined by shuffles in a fixed order.  Offsets
// along k are k * aks / k * bks when those are >= 0, else from the tables.
// n_fast: consecutive outputs run along n (else along m).
template <typename R>
struct FineArgs {
  const Cx<R>*A = nullptr, *B = nullptr;
  Cx<R>* C = nullptr;
  const long long *aM = nullptr, *aK = nullptr, *bN = nullptr, *bK = nullptr, *cM = nullptr,
                  *cN = nullptr, *aB = nullptr, *bB = nullptr, *cB = nullptr;
  int M = 1, N = 1, K = 1, nb = 1;
  long long aks = -1, bks = -1;
  int ls_log = 0;
  bool n_fast = true, block_wide = false;
  R alpha = R(1);
  bool accumulate = false;
};
// Lane split of an outputs x K product (see FineArgs).
void fine_split(long long outputs, long long K, int* ls_log, bool* block_wide);
template <typename R>
void launch_fine(const FineArgs<R>& a, cudaStream_t s);

template <typename R>
void launch_gemv(bool a_kc, const Cx<R>* A, long long aoff, const long long* aM, const long long* aK,
                 const Cx<R>* B, long long boff, const long long* bK, Cx<R>* C, long long coff,
                 const long long* cM, int M, int K, double alpha, bool accumulate, cudaStream_t s);

}  // namespace rtcc3
