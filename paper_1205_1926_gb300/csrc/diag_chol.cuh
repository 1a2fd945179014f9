// Cholesky factor and inverse of a diagonal block in shared memory, shared by the banded factorisation and the
// Woodbury set-up.
#pragma once
#include "dev.h"

namespace tfeti {

constexpr int kDiagLd = kMaxNB + 1;   // row pitch of the blocks

// Cholesky of the jb x jb block D (lower, in shared memory) and its inverse X, all threads.
// The pivot's square root and reciprocal come from y = 1/sqrt(d) by Newton-Raphson,
// y <- y (3 - d y^2) / 2, two steps from an FP32 rsqrtf guess (2^-23 -> below FP64
// rounding): on this part every FP64 instruction of a lone thread occupies the
// sub-partition's FP64 pipe for a whole warp's worth of cycles, so the library
// square root and division sequences dominated the column step.  A pivot that is
// not positive sets `bit` of err and is replaced by 1.
__device__ inline void diag_factor_invert(double* D, double* X, int jb, int* err, int bit) {
  const int tid = threadIdx.x, nt = blockDim.x;
  __shared__ double s_rdiag[kMaxNB];
  // X = I; column c of the factor and row c of X = L^{-1} advance together: after the
  // pivot, column c of L and row c of X are scaled by 1/L[c][c]; then the trailing lower
  // triangle of D and the rows r > c of X (X[r][:] -= L[r][c] X[c][:]) are updated in the
  // same phase, three barriers per column
  for (int e = tid; e < jb * jb; e += nt) X[(e / jb) * kDiagLd + e % jb] = (e / jb == e % jb) ? 1.0 : 0.0;
  for (int c = 0; c < jb; ++c) {
    if (tid == 0) {
      double d = D[c * kDiagLd + c];
      if (!(d > 0.0)) {
        atomicOr(err, bit);
        d = 1.0;
      }
      double y = (double)rsqrtf((float)d);
      y = y * (1.5 - 0.5 * d * y * y);
      y = y * (1.5 - 0.5 * d * y * y);
      D[c * kDiagLd + c] = d * y;
      s_rdiag[c] = y;
    }
    __syncthreads();
    const double inv = s_rdiag[c];
    const int m = jb - c - 1;
    for (int e = tid; e < jb; e += nt) {
      if (e < m) D[(c + 1 + e) * kDiagLd + c] *= inv;
      else X[c * kDiagLd + (e - m)] *= inv;
    }
    __syncthreads();
    // trailing lower triangle, enumerated densely so that every lane of a warp has an entry,
    // followed by the m x (c + 1) update of X
    const int ntri = m * (m + 1) / 2;
    for (int e = tid; e < ntri + m * (c + 1); e += nt) {
      if (e < ntri) {
        int t = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
        while (t * (t + 1) / 2 > e) --t;
        while ((t + 1) * (t + 2) / 2 <= e) ++t;
        const int r = c + 1 + t, q = c + 1 + (e - t * (t + 1) / 2);
        D[r * kDiagLd + q] -= D[r * kDiagLd + c] * D[q * kDiagLd + c];
      } else {
        const int f = e - ntri, r = c + 1 + f / (c + 1), q = f % (c + 1);
        X[r * kDiagLd + q] -= D[r * kDiagLd + c] * X[c * kDiagLd + q];
      }
    }
    __syncthreads();
  }
}

}  // namespace tfeti
