// Facewise complex GEMM of the half spectrum in plain FP32 (Algorithm 1 and
// Algorithm 2 loops over k: C_hat_k = A_hat_k B_hat_k).  Planar split-complex
// operands, four real products per complex multiply-add, each output summed
// over K in order.  The real slices (k = 0 and, for even n3, k = n3/2) skip
// the imaginary planes.
//
// Bound by the float32 FMA pipe (ncu: busy 70% of the time, the issue slots
// 44%).  Each thread owns a 4 x 4 complex block as row pairs and runs
// Blackwell's packed two-lane FMA: one instruction does two multiply-adds, so
// the operand loads fit in the free issue slots.  K tiles of 16 arrive by
// asynchronous 4-byte copies (any alignment, zero-filled past the edges, B
// transposed on the way) in a three-stage ring; holding B twice over in
// shared memory to save its register copies was slower (3.28 ms below).
// 600 x 500 x 1600, 33 slices: 3.62 ms (one multiply-add per instruction, two
// barriers per K tile) -> 2.68 ms, 45 of the nominal 80 TFLOP/s.
#include "tp_internal.cuh"

namespace tp {
namespace {

constexpr int BK = 16, STAGES = 3;

// 4-byte asynchronous copy, zero when !ok (the address is then not read).
__device__ __forceinline__ void copy4(uint32_t dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src),
               "r"(ok ? 4 : 0)
               : "memory");
}

// The tile shapes: BM x BN outputs by (BM / TM) x (BN / TN) threads.  Row
// pitches of the K tiles: A keeps 16-byte rows; B's four extra floats spread
// its transposing copies over the banks.
template <int BM_, int BN_, int TM_, int TN_>
struct Shape {
  static constexpr int BM = BM_, BN = BN_, TM = TM_, TN = TN_;
  static constexpr int TX = BM / TM, TY = BN / TN, NT = TX * TY;
  static constexpr int LA = BM, LB = BN + 4;
  static constexpr int STAGE = 2 * BK * (LA + LB);   // floats
  static constexpr size_t SMEM = size_t(STAGES) * STAGE * sizeof(float);
  static_assert(BM * BK % NT == 0 && BN * BK % NT == 0, "whole copies per thread");
};

template <class S, bool REAL, bool CONJ>
__device__ __forceinline__ void cgemm_tile(const CGemm& g, int64_t f, int64_t K, float* sm) {
  constexpr int BM = S::BM, BN = S::BN, TM = S::TM, TN = S::TN, NT = S::NT;
  const int tid = threadIdx.x;
  const int tx = tid % S::TX, ty = tid / S::TX;
  const int64_t m0 = int64_t(blockIdx.x) * BM;
  const int64_t n0 = int64_t(blockIdx.y) * BN;
  const float* ap[2] = {g.ar + f * g.sA, g.ai + f * g.sA};
  const float* bp[2] = {g.br + f * g.sB, g.bi + f * g.sB};
  const uint32_t sbase = uint32_t(__cvta_generic_to_shared(sm));

  // copies of one K tile into stage s: A by columns (rows fastest), B along k
  // (or along n when it is given as its conjugate transpose)
  auto load = [&](int64_t kt, int s) {
    const uint32_t da = sbase + uint32_t(s * S::STAGE) * 4;
    const uint32_t db = da + uint32_t(2 * BK * S::LA) * 4;
#pragma unroll
    for (int pl = 0; pl < (REAL ? 1 : 2); ++pl) {
#pragma unroll
      for (int u = 0; u < BM * BK / NT; ++u) {
        const int e = tid + NT * u, m = e % BM, k = e / BM;
        const bool ok = m0 + m < g.M && kt + k < K;
        copy4(da + uint32_t((pl * BK + k) * S::LA + m) * 4,
              ok ? ap[pl] + m0 + m + g.lda * (kt + k) : ap[pl], ok);
      }
#pragma unroll
      for (int u = 0; u < BN * BK / NT; ++u) {
        const int e = tid + NT * u;
        const int k = CONJ ? e / BN : e % BK, n = CONJ ? e % BN : e / BK;
        const bool ok = n0 + n < g.N && kt + k < K;
        const int64_t off = CONJ ? n0 + n + g.ldb * (kt + k) : kt + k + g.ldb * (n0 + n);
        copy4(db + uint32_t((pl * BK + k) * S::LB + n) * 4, ok ? bp[pl] + off : bp[pl], ok);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  // rows of the thread: groups of 4 consecutive, 4 TX apart; columns likewise
  float2 cr[TM / 2][TN], ci[TM / 2][TN];
#pragma unroll
  for (int i = 0; i < TM / 2; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) cr[i][j] = ci[i][j] = make_float2(0.f, 0.f);

  const int64_t nt = (K + BK - 1) / BK;
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < nt) load(int64_t(s) * BK, s);
    else asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int stage = 0;
  for (int64_t t = 0; t < nt; ++t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();   // tile t has landed; every thread is done with tile t - 1's stage
    const int64_t next = t + STAGES - 1;
    const int ns = stage == 0 ? STAGES - 1 : stage - 1;
    if (next < nt) load(next * BK, ns);
    else asm volatile("cp.async.commit_group;" ::: "memory");
    const float* As = sm + stage * S::STAGE;
    const float* Bs = As + 2 * BK * S::LA;
#pragma unroll 4
    for (int kk = 0; kk < BK; ++kk) {
      float2 a_r[TM / 2], a_i[TM / 2], a_n[TM / 2];
      float b_r[TN], b_i[TN];
#pragma unroll
      for (int i = 0; i < TM / 4; ++i) {
        const float4 x = *reinterpret_cast<const float4*>(As + kk * S::LA + i * 4 * S::TX + tx * 4);
        a_r[2 * i] = make_float2(x.x, x.y);
        a_r[2 * i + 1] = make_float2(x.z, x.w);
        if (!REAL) {
          const float4 y =
              *reinterpret_cast<const float4*>(As + (BK + kk) * S::LA + i * 4 * S::TX + tx * 4);
          a_i[2 * i] = make_float2(y.x, y.y);
          a_i[2 * i + 1] = make_float2(y.z, y.w);
        }
      }
#pragma unroll
      for (int j = 0; j < TN / 4; ++j) {
        const float4 x = *reinterpret_cast<const float4*>(Bs + kk * S::LB + j * 4 * S::TY + ty * 4);
        b_r[4 * j] = x.x; b_r[4 * j + 1] = x.y; b_r[4 * j + 2] = x.z; b_r[4 * j + 3] = x.w;
        if (!REAL) {
          const float4 y =
              *reinterpret_cast<const float4*>(Bs + (BK + kk) * S::LB + j * 4 * S::TY + ty * 4);
          b_i[4 * j] = y.x; b_i[4 * j + 1] = y.y; b_i[4 * j + 2] = y.z; b_i[4 * j + 3] = y.w;
        }
      }
      if (!REAL)   // -Im A, or -Re A against a conjugated B
#pragma unroll
        for (int i = 0; i < TM / 2; ++i)
          a_n[i] = CONJ ? make_float2(-a_r[i].x, -a_r[i].y) : make_float2(-a_i[i].x, -a_i[i].y);
      // two columns at a time and one product after the other, so that a
      // dependent update comes TM packed FMAs later
#pragma unroll
      for (int j = 0; j < TN; j += 2) {
        const float2 br[2] = {make_float2(b_r[j], b_r[j]), make_float2(b_r[j + 1], b_r[j + 1])};
#pragma unroll
        for (int e = 0; e < TM; ++e)
          cr[e / 2][j + (e & 1)] = __ffma2_rn(a_r[e / 2], br[e & 1], cr[e / 2][j + (e & 1)]);
        if (!REAL) {
          const float2 bi[2] = {make_float2(b_i[j], b_i[j]), make_float2(b_i[j + 1], b_i[j + 1])};
#pragma unroll
          for (int e = 0; e < TM; ++e)
            ci[e / 2][j + (e & 1)] =
                __ffma2_rn(CONJ ? a_n[e / 2] : a_r[e / 2], bi[e & 1], ci[e / 2][j + (e & 1)]);
#pragma unroll
          for (int e = 0; e < TM; ++e)
            cr[e / 2][j + (e & 1)] =
                __ffma2_rn(CONJ ? a_i[e / 2] : a_n[e / 2], bi[e & 1], cr[e / 2][j + (e & 1)]);
#pragma unroll
          for (int e = 0; e < TM; ++e)
            ci[e / 2][j + (e & 1)] = __ffma2_rn(a_i[e / 2], br[e & 1], ci[e / 2][j + (e & 1)]);
        }
      }
    }
    stage = stage + 1 == STAGES ? 0 : stage + 1;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");

  float* Cr = g.cr + f * g.sC;
  float* Ci = g.ci + f * g.sC;
#pragma unroll
  for (int j = 0; j < TN; ++j) {
    const int64_t n = n0 + (j / 4) * 4 * S::TY + ty * 4 + (j & 3);
    if (n >= g.N) continue;
#pragma unroll
    for (int i = 0; i < TM / 2; ++i) {
      const int64_t m = m0 + (i / 2) * 4 * S::TX + tx * 4 + 2 * (i & 1);
      const float2 r = cr[i][j];
      const float2 c = REAL ? make_float2(0.f, 0.f) : ci[i][j];
      if (m < g.M) {
        Cr[m + g.ldc * n] = r.x;
        Ci[m + g.ldc * n] = c.x;
      }
      if (m + 1 < g.M) {
        Cr[m + 1 + g.ldc * n] = r.y;
        Ci[m + 1 + g.ldc * n] = c.y;
      }
    }
  }
}

template <class S, bool CONJ>
__global__ void __launch_bounds__(S::NT) cgemm_simt_kernel(const __grid_constant__ CGemm g) {
  extern __shared__ __align__(16) float cg_sm[];
  const int64_t K = g.dynK ? *g.dynK : g.K;
  for (int64_t f = blockIdx.z; f < g.h; f += gridDim.z) {
    if (g.only && g.only[f] != g.only_val) continue;
    const bool real = (f == 0) || ((g.n3 % 2 == 0) && f == g.h - 1);
    if (real) cgemm_tile<S, true, CONJ>(g, f, K, cg_sm);
    else cgemm_tile<S, false, CONJ>(g, f, K, cg_sm);
    __syncthreads();
  }
}

using Wide = Shape<64, 64, 4, 4>;     // 256 threads, two CTAs per SM
using Small = Shape<32, 32, 4, 4>;    // 64 threads

template <class S>
int64_t tiles(const CGemm& g) {
  return ((g.M + S::BM - 1) / S::BM) * ((g.N + S::BN - 1) / S::BN) * g.h;
}

template <class S>
int launch_shape(const CGemm& g, cudaStream_t st) {
  const int64_t gx = (g.M + S::BM - 1) / S::BM, gy = (g.N + S::BN - 1) / S::BN;
  if (gx > 0x7fffffff || gy > 65535) {
    set_error("cgemm: output %lld x %lld too large for one launch", (long long)g.M, (long long)g.N);
    return TP_EUNSUPPORTED;
  }
  const int64_t gz = g.h < 65535 ? g.h : 65535;
  const dim3 grid{unsigned(gx), unsigned(gy), unsigned(gz)};
  KernelScope ks("cgemm_fp32", st);
  if (g.b_conj_trans) {
    TP_SET_SMEM((cgemm_simt_kernel<S, true>), S::SMEM);
    cgemm_simt_kernel<S, true><<<grid, S::NT, S::SMEM, st>>>(g);
  } else {
    TP_SET_SMEM((cgemm_simt_kernel<S, false>), S::SMEM);
    cgemm_simt_kernel<S, false><<<grid, S::NT, S::SMEM, st>>>(g);
  }
  return launch_status("cgemm_simt_kernel");
}

}  // namespace

// 64 x 64 tiles, or 32 x 32 ones where a short inner dimension (at most 256)
// leaves fewer than four of the former per SM: such launches end before their
// pipelines fill, and finer tiles use more SMs (256 x 144 x 144, 41 slices:
// 56 against 64 us; 64 x 32 x 48, 9 slices: 8.2 against 8.3; but 611 x 389 x
// 150, 23 slices, ten tiles per SM: 186 against 176).  Larger thread blocks
// of 8 x 8 outputs were no faster (2819 against 2677 us on the headline shape
// below).  32 x 32 ones too where C has at most 32 rows or columns, half of a 64
// x 64 tile or more being work for nothing: 10^6 x 4 x 4, 2 slices 254 -> 145 us, 2000 x 20 x
// 2000, 9 slices 405 -> 279, 5000 x 10 x 300, 17 slices 274 -> 170.  Both shapes sum
// in the same order.
int launch_cgemm_simt(const CGemm& g, cudaStream_t st) {
  if (g.M == 0 || g.N == 0 || g.h == 0) return TP_OK;
  const int64_t K = g.dynK ? g.kcap : g.K;
  const bool narrow = (g.N <= 32 || g.M <= 32) && g.N <= 32 * int64_t(65535);
  if (narrow || (K <= 256 && tiles<Wide>(g) < 4 * int64_t(sm_count())))
    return launch_shape<Small>(g, st);
  return launch_shape<Wide>(g, st);
}

}  // namespace tp
