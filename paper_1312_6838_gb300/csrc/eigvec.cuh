// Internal interface of the eigenvector estimate (eigvec.cu) that the cyclic
// Jacobi rounds of lowrank.cu start from.
#pragma once

#include "css_common.cuh"

namespace css {

constexpr int kEstimateMinL = 17;   // see eigvec.cu

// Scratch of the estimate; G and H are lp x lp (leading dimension lp, l <= lp).
struct Estimate {
  float *A0, *A1, *X32, *Q;    // L x L each (L: l rounded up to 64), 64 x 64 per block pair
  double *X0, *X1, *Y, *E;     // l x l
  unsigned long long* log;     // the rotations of every block pair's sweep
  uint32_t *bar, *most;        // zeroed before the launch (kEstimateZeroed words from bar)
};
constexpr int kRotationWait = 46;   // id of the wait for a sweep's rotations
constexpr int kEstimateSweeps = 12;
constexpr int kEstimateZeroed = 32 + 2 * kEstimateSweeps;

inline bool estimate_fits(int l, int sms) { return l >= kEstimateMinL && 2 * ((l + 63) / 64) <= sms; }
Estimate carve_estimate(WsCarver& c, int l);
// X (l x l, orthogonal to FP64 rounding, returned in *X) with H = X^T G X
// diagonal as far as the estimate separates the eigenvalues; H is symmetric
// bit for bit.  Errors go to st.
cudaError_t estimate_eigvecs(const double* G, double* H, int l, int lp, const Estimate& w, DevStatus* st, int sms,
                             const double** X, cudaStream_t s);

}  // namespace css
