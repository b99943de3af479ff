// Householder QR of batched slices (householder.cu).
#pragma once

#include "tp_internal.cuh"

namespace tp {

constexpr int HQR_MAX_L = 96;   // columns of a slice

// Split planes (p0 non-null): Q also leaves as the hi/lo planes (bf16 or
// tf32, dftc::put_split) of the next tensor-core product's B operand,
// K-major with leading dimension ldk, p <= ldk <= 32 ceil(p / 32) (rows
// p .. ldk-1 and the columns from l on zero), slice stride ldk * lfull --
// the operand split fused.
struct HqrSplit {
  float* p0;
  float* p1;
  float* p2;
  float* p3;
  int64_t ldk;
  int bf16;
};

// Whether householder_launch takes slices of p x l (else householder_tall_launch).
bool householder_applies(int64_t p, int64_t l);

// Orthonormalises `batch` slices Y (p x l, column-major, slice stride sY) in
// place.  lcols (device, per slice, or null): only the first lcols[f] columns
// are factored, the others set to zero.  keep_phase: column j of Q is
// multiplied by sign(R(j, j)) (R's diagonal is real), so that for Y with
// nearly orthonormal columns Q(:, j) stays close to Y(:, j) instead of
// possibly flipping its sign.
int householder_launch(float* yr, float* yi, int64_t sY, int p, int l, const int32_t* lcols,
                       bool keep_phase, int64_t batch, cudaStream_t st, HqrSplit sp = HqrSplit{});

// The same QR of slices of at most 256 rows with the sums in the order of the
// shared-memory form (no split planes, no kept phase).
int householder_shared_launch(float* yr, float* yi, int64_t sY, int p, int l, const int32_t* lcols,
                              int64_t batch, cudaStream_t st);

// The same for contiguous slices of more than 256 rows (slice stride rows * l),
// with `scratch` of householder_tall_scratch() bytes, 256-byte aligned.  A
// slice that is all zero or not finite sets TP_DEV_BREAKDOWN and is left zero
// (not a number).
size_t householder_tall_scratch(int64_t rows, int64_t l, int64_t batch);
int householder_tall_launch(float* yr, float* yi, int64_t rows, int l, const int32_t* lcols,
                            int64_t batch, void* scratch, int32_t* status, cudaStream_t st);

// CholeskyQR2 in float64 (cholqr.cu) of contiguous slices of any number of rows
// >= l, with `scratch` of cholqr_scratch() bytes, 256-byte aligned.  A Gram
// matrix that is not positive definite even with a shift (an all-zero or not
// finite slice) sets TP_DEV_BREAKDOWN and leaves the slice as it is.  weak
// (device, or null) is set to 1 if some slice's diagonal of R leaves the rank in
// doubt: a Cholesky breakdown, or min R(j, j) <= CHOLQR_WEAK max R(j, j).  2^-16 is 256 times float32's rounding, and
// its square is far above float64's.  polish: one pass only, for slices that are
// nearly orthonormal; one that is not positive definite stays as it is.
constexpr float CHOLQR_WEAK = 1.f / 65536.f;
size_t cholqr_scratch(int64_t l, int64_t batch);
int cholqr_launch(float* yr, float* yi, int64_t rows, int l, const int32_t* lcols, int64_t batch,
                  void* scratch, int32_t* status, cudaStream_t st, int* weak = nullptr,
                  bool polish = false);

}  // namespace tp
