// FP64-accurate complex products on the tcgen05 tensor cores (sm_103a has 2
// FP64 FMA lanes per SM and clock; its FP16 tensor pipe does 4096).
//
// Splitting (Ozaki, Ogita, Oishi, Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 59, 95 (2012)):
// within one K segment every row of A and B is scaled by the power of two
// above its largest element and rounded to a 62-bit fixed-point number, which
// is cut into eight balanced 8-bit digits.  The digits are exact in FP16; the
// 36 digit products i + j <= 7 are formed by FP16 MMAs into eight FP32
// accumulators (one per i + j) whose partial sums are integers up to 2^24 and
// therefore exact for i + j <= 4 (K <= 256 real; beyond, sums that could have
// left that range are recognised).  The eight sums are joined in integer
// arithmetic and rounded once to a double.
//
// The error is a fraction of the product of the two rows' largest elements, not
// of the terms: at most 2 K 8.02 2^-62 of it for K complex terms.  Outputs for
// which that is not known to be within the bound of FP64 arithmetic, 2 K 2^-53
// sum |a||b| (opposite gradings, near-identity matrices, infinities and NaN,
// results below the normal range), are summed in FP64 instead, so that the bound
// of an FP64 chain holds for every output, |.| being the complex modulus.
//
// A complex product C[m,n] (+)= alpha sum_k A[m,k] B[n,k] runs as one real
// product: A rows interleave (re, im) along K, B is its 2x2 real embedding.
#pragma once

#include "common.h"

namespace rtcc3 {

// How one contraction runs: which operand takes the 128-row side (swap:
// the plan's B), the real columns per tile, the K segments (complex elements
// per segment, segments per CTA) and the number of CTAs that share a tile's
// segments, each with its own sum.
struct OzPlan {
  bool swap = false;
  int nt = 64;
  int seg = 128, nseg = 1, spc = 1, nsplit = 1;
  double cost = 0.0;  // estimated SM clocks of the whole product
};

// Plan of an M x N x K complex product.
OzPlan oz_plan(long long M, long long N, long long K);

struct OzOperand {
  const double2* p = nullptr;
  long long off = 0;
  const long long *rows = nullptr, *ks = nullptr;  // element offsets
  bool kc = false;                                 // contiguous along k
};

// C[coff + cM[m] + cN[n]] (+)= alpha sum_k A[m,k] B[n,k]; with p.nseg > 1 the
// sums of successive segments go through part (nsplit x N x M), with p.nsplit
// > 1 a second launch adds the CTAs' sums in a fixed order.  c_m: C's contiguous index is on the A side.  Returns the
// number of kernel launches.
int oz_gemm(const OzPlan& p, const OzOperand& A, const OzOperand& B, int M, int N, int K, double2* C,
            long long coff, const long long* cM, const long long* cN, bool c_m, double alpha,
            bool accumulate, double2* part, int* err, long long wait_budget, cudaStream_t s);

}  // namespace rtcc3
