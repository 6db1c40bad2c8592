// Split-precision ("error-free slice") FP64 contraction on the tcgen05 tensor
// cores, after Ozaki, Ogita, Oishi and Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and
// its applications" (Numer. Algorithms 59, 2012).
//
// Each row of A (and each column of B) is scaled by a power of two and cut
// into S balanced base-128 digits, x = 2^(e + 1) sum_t d_t 2^(-7t), |d_t| <= 64,
// each digit exact in BF16.  The digit pairs (t,u) of one level c = t + u are
// accumulated together by tcgen05.mma kind::f16, levels c <= S + 1 are kept;
// over a window of k whose level sums stay within 2^24 they are exact in FP32,
// and the windows are added in 64-bit integers.  The result carries about 7 S
// bits relative to the row/column maxima.
#pragma once
#include "engine.cuh"

namespace dsrg {

constexpr int kOzakiMaxSlices = 8;

// Error status of the split-precision kernels (device flag set when a bounded
// wait runs out); 0 = ok.  Synchronises st.
int ozaki_status(cudaStream_t st, const int* flag);

// C[m,n] += alpha * sum_k A[m,k] B[k,n] for the multi-index contraction g
// (nbatch must be 1) with `slices` digits per operand.  Scratch comes from ws.
void ozaki_gemm(Workspace& ws, const GemmArgs& g, int slices, int kind);
// sizes the split-precision path can index (32-bit packing work items)
bool ozaki_supported(const GemmArgs& g);

}  // namespace dsrg
