// Thresholding of slices with few singular values above the threshold
// (svt_top.cu).
#pragma once

#include "tp_internal.cuh"

namespace tp {

constexpr int SVT_TOP_L = 32;   // vectors kept per slice

struct SvtTopArgs {
  // Gram matrices W^H W (q x q, column-major, both triangles), slice stride sG;
  // destroyed, then the rebuild's small operand
  float *gr, *gi;
  int64_t sG;
  float *hr, *hi;          // scratch of q x SVT_TOP_L per slice, slice stride sG
  float *xr, *xi;          // conj(X) of the kept vectors X: [h][q][SVT_TOP_L]
  const double* mu;
  int* attempt;            // per slice: this iteration tries (Gram needed)
  int* fast;               // per slice, set here: 1 = thresholded here, 0 = takes the Jacobi
  int* wait;               // per slice: iterations until the next attempt, and the
                           // failed attempts in a row from bit 16 on
  float* edge;             // per slice: smallest kept eigenvalue, 0 = no quadratic filter
  unsigned* above;         // per slice: bit j set = vector j is above the threshold
  int q;
};

bool svt_top_applies(int64_t q);
size_t svt_top_ws(int64_t q, size_t h);   // bytes of xr, xi and the flags of h slices
// Flags and vectors before a run's first iteration; V = I for the Jacobi.
int svt_top_init(const SvtTopArgs& g, int64_t h, float* vr, float* vi, cudaStream_t st);
int svt_top_launch(const SvtTopArgs& g, int64_t h, cudaStream_t st);
// From H = W X (p x SVT_TOP_L, slice stride sG): the operand that rebuilds the
// shrunk slice, into gr, gi: D X^H, or X D when transposed.
int svt_top_coef(const SvtTopArgs& g, int64_t h, const float* hr, const float* hi, int64_t p,
                 bool transpose, cudaStream_t st);

}  // namespace tp
