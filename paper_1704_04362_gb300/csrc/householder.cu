// orth() of the randomized t-SVD and of the t-SVD's vectors: the Householder
// QR Y = Q R of a batch of slices (p x l, p >= l, l <= 96, planar float32,
// column-major) with reflectors H_j = I - tau_j v_j v_j^H (v_j(j) = 1, zero
// above) chosen as LAPACK's zlarfg chooses them, so that H_j^H maps rows j..
// of column j onto beta_j e_j with beta_j real; then Q = H_0 H_1 ... H_{l-1}
// [I_l; 0].  Householder QR is backward stable whatever the conditioning of
// Y: Q is orthonormal to float32 rounding in one pass and cannot break down,
// and it spans the columns of Y (completed by the reflectors where Y is rank
// deficient), which is all the range finder uses.
//
// One CTA holds a block of up to 256 rows in registers: every lane has rows
// of every column of its warp, warp w the columns w, w + W, ... ("slots").
// Only the reflectors pass through shared memory, one column per step: the
// owner of column j + 1 applies H_j to it first and publishes the next
// reflector (look-ahead), so a step of the factorisation costs one barrier.
// Forming Q needs none: every column of Q takes the reflectors in turn on its
// own.  Products run on the packed two-lane float32 FMA.
//
// Slices of more than 256 rows are factored as a tree (tall-skinny QR,
// Demmel, Grigori, Hoemmen and Langou 2012): the rows are cut into blocks of
// 128 .. 256, each block is factored by a CTA of its own, the blocks' R
// factors are stacked and factored in turn until one block is left, and Q is
// formed back down the tree by applying each block's reflectors to its rows
// of the parent's Q.  Scratch is the R stacks only (Y's own storage holds the
// reflectors meanwhile).  Blocks are scaled by powers of two, so that squares
// stay in float32's range whatever the magnitude of Y.
//
// What bounds it: the chain of l dependent reflectors per block (two warp
// sums, a square root, divisions, a barrier) and, where the slices are many
// and the SMs full, instruction issue.
// 33 slices of 1024 x 50 (the plain rank rule's sketch of a 1024 x 1024 x 64
// tensor): 0.24 ms, against 3.2 ms of the float64 CholeskyQR2 that the last
// orthonormalisation of a call takes (cholqr.cu).  1001 slices of 128 x 50: 0.35 ms (columns in shared
// memory, read and written every step) -> 0.335 ms; 8 lanes a column with 16
// rows each (fewer shuffles, a longer chain per reflector) 0.42 ms.
#include "householder.cuh"

#include "dft_common.cuh"

namespace tp {
namespace {

// A column of P = 64 R2 rows in a warp's registers: lane `lane` holds the row
// pairs r, r + 1 with r = 64 t + 2 lane, t < R2, real and imaginary parts
// apart, so that products run on the packed two-lane FMA without shuffling.
template <int R2>
struct HqrCol {
  float2 re[R2], im[R2];
};

__device__ __forceinline__ float hqr_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Two (four) warp sums at once by exchanging halves of the values at the
// first (two) levels instead of reducing each value separately: 5 + 2
// broadcasts (6 + 4) shuffles instead of 10 (20); every lane gets every sum.
__device__ __forceinline__ void hqr_sum2(float& a, float& b, int lane) {
  const bool up = lane & 16;
  float k = up ? b : a;
  k += __shfl_xor_sync(0xffffffffu, up ? a : b, 16);   // a in the low half, b in the high
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  a = __shfl_sync(0xffffffffu, k, 0);
  b = __shfl_sync(0xffffffffu, k, 16);
}
__device__ __forceinline__ void hqr_sum4(float (&d)[4], int lane) {
  const bool up = lane & 16, mid = lane & 8;
  float k0 = up ? d[2] : d[0], k1 = up ? d[3] : d[1];
  k0 += __shfl_xor_sync(0xffffffffu, up ? d[0] : d[2], 16);
  k1 += __shfl_xor_sync(0xffffffffu, up ? d[1] : d[3], 16);
  float k = mid ? k1 : k0;
  k += __shfl_xor_sync(0xffffffffu, mid ? k0 : k1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  // lanes 0-7 hold sum 0, 8-15 sum 1, 16-23 sum 2, 24-31 sum 3
#pragma unroll
  for (int u = 0; u < 4; ++u) d[u] = __shfl_sync(0xffffffffu, k, 8 * u);
}

// v^H x over this lane's rows.
template <int R2>
__device__ __forceinline__ void hqr_dot(const HqrCol<R2>& v, const HqrCol<R2>& x, float& dr,
                                        float& di) {
  float2 a = make_float2(0.f, 0.f), b = a, c = a;
#pragma unroll
  for (int t = 0; t < R2; ++t) {
    a = __ffma2_rn(v.re[t], x.re[t], a);
    b = __ffma2_rn(v.re[t], x.im[t], b);
    a = __ffma2_rn(v.im[t], x.im[t], a);
    c = __ffma2_rn(v.im[t], x.re[t], c);
  }
  dr = a.x + a.y;
  di = (b.x - c.x) + (b.y - c.y);
}
// x <- x - v (f d), d = v^H x (f = conj(tau) applies H^H, f = tau applies H)
template <int R2>
__device__ __forceinline__ void hqr_update(const HqrCol<R2>& v, HqrCol<R2>& x, float2 f, float dr,
                                           float di) {
  const float gr = f.x * dr - f.y * di, gi = f.x * di + f.y * dr;
  const float2 nr = make_float2(-gr, -gr), pi = make_float2(gi, gi), ni = make_float2(-gi, -gi);
#pragma unroll
  for (int t = 0; t < R2; ++t) {
    x.re[t] = __ffma2_rn(v.re[t], nr, x.re[t]);
    x.im[t] = __ffma2_rn(v.re[t], ni, x.im[t]);
    x.re[t] = __ffma2_rn(v.im[t], pi, x.re[t]);
    x.im[t] = __ffma2_rn(v.im[t], nr, x.im[t]);
  }
}

// A reflector column in shared memory: (re r, re r + 1, im r, im r + 1) of the
// row pairs in order, one 16-byte access per pair.
template <int R2>
__device__ __forceinline__ HqrCol<R2> hqr_load_v(const float4* vcol, int lane) {
  HqrCol<R2> v;
#pragma unroll
  for (int t = 0; t < R2; ++t) {
    const float4 a = vcol[32 * t + lane];
    v.re[t] = make_float2(a.x, a.y);
    v.im[t] = make_float2(a.z, a.w);
  }
  return v;
}

// Reflector of the register column x at row k, one warp: v (1 at row k, zeros
// above) goes to vcol, x keeps R's column (beta at row k, zeros below).
// Returns tau (0 when the column is already beta e_k with beta real).
template <int R2>
__device__ __forceinline__ float2 hqr_reflector(HqrCol<R2>& x, int k, float4* vcol, int lane,
                                                float& beta) {
  float s = 0.f, ax = 0.f, ay = 0.f;
#pragma unroll
  for (int t = 0; t < R2; ++t) {
    const int r = 64 * t + 2 * lane;
    if (r > k) s = fmaf(x.re[t].x, x.re[t].x, fmaf(x.im[t].x, x.im[t].x, s));
    if (r + 1 > k) s = fmaf(x.re[t].y, x.re[t].y, fmaf(x.im[t].y, x.im[t].y, s));
    if (r == k) {
      ax = x.re[t].x;
      ay = x.im[t].x;
    }
    if (r + 1 == k) {
      ax = x.re[t].y;
      ay = x.im[t].y;
    }
  }
  s = hqr_sum(s);
  const int src = (k >> 1) & 31;
  ax = __shfl_sync(0xffffffffu, ax, src);
  ay = __shfl_sync(0xffffffffu, ay, src);
  float2 tau = make_float2(0.f, 0.f);
  float sr = 0.f, si = 0.f;
  beta = ax;
  if (!(s == 0.f && ay == 0.f)) {
    const float nrm = sqrtf(fmaf(ax, ax, fmaf(ay, ay, s)));
    beta = ax >= 0.f ? -nrm : nrm;
    // v = x / (alpha - beta); |alpha - beta| >= nrm > 0 by the sign of beta
    const float dr = ax - beta, di = ay;
    const float den = fmaf(dr, dr, di * di);
    sr = dr / den;
    si = -di / den;
    tau = make_float2((beta - ax) / beta, -ay / beta);
  }
#pragma unroll
  for (int t = 0; t < R2; ++t) {
    const int r = 64 * t + 2 * lane;
    float4 v = make_float4(x.re[t].x * sr - x.im[t].x * si, x.re[t].y * sr - x.im[t].y * si,
                           x.re[t].x * si + x.im[t].x * sr, x.re[t].y * si + x.im[t].y * sr);
    if (r > k) x.re[t].x = x.im[t].x = 0.f;
    else v.x = r == k ? 1.f : 0.f, v.z = 0.f;
    if (r + 1 > k) x.re[t].y = x.im[t].y = 0.f;
    else v.y = r + 1 == k ? 1.f : 0.f, v.w = 0.f;
    if (r == k) x.re[t].x = beta, x.im[t].x = 0.f;
    if (r + 1 == k) x.re[t].y = beta, x.im[t].y = 0.f;
    vcol[32 * t + lane] = v;
  }
  return tau;
}

// The reflector (v, f) on this warp's columns k with lo < k < l in the slots
// from `first` on, two at a time (their sums interleave in the shuffles).
template <int R2, int W, int SLOTS>
__device__ __forceinline__ void hqr_apply(const HqrCol<R2>& v, HqrCol<R2> (&x)[SLOTS], int first,
                                          int lo, int l, float2 f, int warp, int lane) {
#pragma unroll
  for (int s = 0; s < SLOTS; s += 2) {
    constexpr int kLast = SLOTS - 1;
    if (s + 1 < first) continue;
    const int s1 = s < kLast ? s + 1 : s;
    const int k0 = warp + W * s, k1 = warp + W * s1;
    const bool a0 = k0 > lo && k0 < l;
    const bool a1 = s1 != s && k1 > lo && k1 < l;
    if (a0 && a1) {
      float d[4];
      hqr_dot<R2>(v, x[s], d[0], d[1]);
      hqr_dot<R2>(v, x[s1], d[2], d[3]);
      hqr_sum4(d, lane);
      hqr_update<R2>(v, x[s], f, d[0], d[1]);
      hqr_update<R2>(v, x[s1], f, d[2], d[3]);
    } else if (a0) {
      float dr, di;
      hqr_dot<R2>(v, x[s], dr, di);
      hqr_sum2(dr, di, lane);
      hqr_update<R2>(v, x[s], f, dr, di);
    } else if (a1) {
      float dr, di;
      hqr_dot<R2>(v, x[s1], dr, di);
      hqr_sum2(dr, di, lane);
      hqr_update<R2>(v, x[s1], f, dr, di);
    }
  }
}

// Binary exponent of |x| (0 for zero is excluded by the caller; infinities
// and NaN give 128).
__device__ __forceinline__ int hqr_exponent(float x) {
  return int((__float_as_uint(x) >> 23) & 0xffu) - 127;
}
constexpr int kZeroBlock = -1000000;   // exponent of a block of zeros

// HQR_WHOLE   a slice of at most 256 rows: Y becomes Q (and its split planes)
// HQR_FACTOR  a block of a taller slice: Y becomes the reflectors, R goes to
//             the stack of the next level
// HQR_TOP     the last level's stack (one block per slice): becomes its Q;
//             a slice whose R is all zero or not finite is flagged
enum HqrMode { HQR_WHOLE, HQR_FACTOR, HQR_TOP };

struct HqrParams {
  float *yr, *yi;          // element (r, c) of slice f at f*sY + r + rows*c
  int64_t sY;
  int rows, nb;            // rows of a slice, blocks per slice (balanced cut)
  int lfull;
  const int32_t* lcols;    // per-slice column counts or null
  int keep_phase;
  HqrSplit sp;
  // tree levels
  float2* tau;             // [slice][block][lfull]
  float *rr, *ri;          // FACTOR: the stack, (nb lfull) x lfull per slice
  int* ex_out;             // [slice][block]: exponent the block was scaled by
  const int* ex_in;        // exponents of this level's source blocks (lfull rows each) or null
  int* flag;               // [slice]: 0, 1 (zero), 2 (not finite)
  int32_t* status;
};

__device__ __forceinline__ void hqr_block(int rows, int nb, int b, int& r0, int& p) {
  const int base = rows / nb, rem = rows % nb;
  r0 = b * base + min(b, rem);
  p = base + (b < rem ? 1 : 0);
}

// Shared-memory index (in floats) of row r's real part in a reflector column;
// the imaginary part is 2 further.
__device__ __forceinline__ int hqr_vrow(int r) { return 4 * (r >> 1) + (r & 1); }

// CTAs per SM the registers are budgeted for: 64 a thread while the columns
// take at most half of them.
template <int R2, int W, int SLOTS>
struct HqrResident {
  static constexpr int v = 4 * R2 * SLOTS <= 32 ? 1024 / (32 * W) : 512 / (32 * W);
};

template <int R2, int W, int SLOTS, int MODE>
__global__ void __launch_bounds__(32 * W, HqrResident<R2, W, SLOTS>::v)
    hqr_kernel(const HqrParams g) {
  constexpr int PP = 32 * R2;                          // row pairs of a column
  extern __shared__ __align__(16) float4 hqr_v[];      // reflectors, l columns of PP pairs
  __shared__ float2 tau_s[HQR_MAX_L];
  __shared__ float beta_s[HQR_MAX_L];                  // R(j, j)
  __shared__ int amax_s, bits_s;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int f = int(blockIdx.x) / g.nb, b = int(blockIdx.x) - f * g.nb;
  const int lfull = g.lfull;
  // per-slice column count (the per-frequency sketch size): the columns from
  // l on are left zero
  const int l = g.lcols ? min(max(int(g.lcols[f]), 1), lfull) : lfull;
  int r0, p;
  hqr_block(g.rows, g.nb, b, r0, p);
  float* yr = g.yr + int64_t(f) * g.sY + r0;
  float* yi = g.yi + int64_t(f) * g.sY + r0;
  const int64_t ld = g.rows;

  HqrCol<R2> x[SLOTS];
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    const int k = warp + W * s;
#pragma unroll
    for (int t = 0; t < R2; ++t) {
      const int r = 64 * t + 2 * lane;
      const int64_t o = r + ld * k;
      const bool i0 = k < l && r < p, i1 = k < l && r + 1 < p;
      x[s].re[t] = make_float2(i0 ? yr[o] : 0.f, i1 ? yr[o + 1] : 0.f);
      x[s].im[t] = make_float2(i0 ? yi[o] : 0.f, i1 ? yi[o + 1] : 0.f);
    }
  }
  if (MODE != HQR_WHOLE) {
    // scale the block by 2^-E, E its largest exponent
    if (threadIdx.x == 0) {
      amax_s = kZeroBlock;
      bits_s = 0;
    }
    __syncthreads();
    const int* ex = g.ex_in ? g.ex_in + int64_t(f) * (g.rows / lfull) : nullptr;
    int top = kZeroBlock;
    int er[2 * R2];
#pragma unroll
    for (int i = 0; i < 2 * R2; ++i) {
      const int r = 64 * (i >> 1) + 2 * lane + (i & 1);
      er[i] = ex && r < p ? ex[(r0 + r) / lfull] : 0;
    }
    auto each = [&](auto&& fn) {
#pragma unroll
      for (int s = 0; s < SLOTS; ++s)
#pragma unroll
        for (int t = 0; t < R2; ++t) {
          fn(x[s].re[t].x, er[2 * t]);
          fn(x[s].re[t].y, er[2 * t + 1]);
          fn(x[s].im[t].x, er[2 * t]);
          fn(x[s].im[t].y, er[2 * t + 1]);
        }
    };
    each([&](float& a, int e) {
      if (a != 0.f) top = max(top, hqr_exponent(a) + e);
    });
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) atomicMax(&amax_s, top);
    __syncthreads();
    const int E = amax_s;
    each([&](float& a, int e) {
      if (a != 0.f) a = ldexpf(a, e - E);
    });
    if (MODE == HQR_FACTOR && threadIdx.x == 0) g.ex_out[int64_t(f) * g.nb + b] = E;
  }
  // factorisation: step kn - 1 applies H_{kn-1}^H to columns kn .. l-1 and
  // forms reflector kn (step -1 only forms the first).  The slot of column kn
  // is the outer, unrolled loop, so that every column is addressed by a
  // constant and stays in registers.
#pragma unroll
  for (int s0 = 0; s0 < SLOTS; ++s0) {
#pragma unroll 1
    for (int ww = 0; ww < W; ++ww) {
      const int kn = s0 * W + ww, j = kn - 1;
      if (kn >= l) break;
      HqrCol<R2> v;
      float2 fc = make_float2(0.f, 0.f);
      if (j >= 0) {
        v = hqr_load_v<R2>(hqr_v + j * PP, lane);
        fc = make_float2(tau_s[j].x, -tau_s[j].y);
      }
      const bool live = fc.x != 0.f || fc.y != 0.f;
      if (warp == ww) {   // look-ahead: column kn first, then its reflector
        if (live) {
          float dr, di;
          hqr_dot<R2>(v, x[s0], dr, di);
          hqr_sum2(dr, di, lane);
          hqr_update<R2>(v, x[s0], fc, dr, di);
        }
        float beta;
        const float2 t = hqr_reflector<R2>(x[s0], kn, hqr_v + kn * PP, lane, beta);
        if (lane == 0) {
          tau_s[kn] = t;
          beta_s[kn] = beta;
        }
      }
      if (live) hqr_apply<R2, W, SLOTS>(v, x, s0, kn, l, fc, warp, lane);
      __syncthreads();
    }
  }
  const float* vf = reinterpret_cast<const float*>(hqr_v);
  if (MODE == HQR_FACTOR) {
    float2* tau = g.tau + (int64_t(f) * g.nb + b) * lfull;
    for (int j = threadIdx.x; j < l; j += 32 * W) tau[j] = tau_s[j];
    const int64_t lr = int64_t(g.nb) * lfull;
    float* rr = g.rr + int64_t(f) * lr * lfull + int64_t(b) * lfull;
    float* ri = g.ri + int64_t(f) * lr * lfull + int64_t(b) * lfull;
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      const int k = warp + W * s;
      if (k >= lfull) continue;
#pragma unroll
      for (int i = 0; i < 2 * R2; ++i) {
        const int r = 64 * (i >> 1) + 2 * lane + (i & 1);
        if (r < lfull) {   // x is zero below the diagonal and in the columns from l on
          rr[r + lr * k] = (i & 1) ? x[s].re[i >> 1].y : x[s].re[i >> 1].x;
          ri[r + lr * k] = (i & 1) ? x[s].im[i >> 1].y : x[s].im[i >> 1].x;
        }
        if (k < l && r < p) {
          yr[r + ld * k] = vf[4 * k * PP + hqr_vrow(r)];
          yi[r + ld * k] = vf[4 * k * PP + hqr_vrow(r) + 2];
        }
      }
    }
    return;
  }
  if (MODE == HQR_TOP) {
    int bits = 0;
#pragma unroll
    for (int s = 0; s < SLOTS; ++s)
#pragma unroll
      for (int t = 0; t < R2; ++t) {
        const float2 a = x[s].re[t], c = x[s].im[t];
        if (a.x != 0.f || a.y != 0.f || c.x != 0.f || c.y != 0.f) bits |= 1;
        if (!isfinite(a.x) || !isfinite(a.y) || !isfinite(c.x) || !isfinite(c.y)) bits |= 2;
      }
    bits = __reduce_or_sync(0xffffffffu, bits);
    if (lane == 0 && bits) atomicOr(&bits_s, bits);
    __syncthreads();
    if (threadIdx.x == 0) {
      const int bad = (bits_s & 2) ? 2 : (bits_s & 1) ? 0 : 1;
      g.flag[f] = bad;
      if (bad && g.status) atomicOr(g.status, TP_DEV_BREAKDOWN);
    }
  }
  // Q's column k: H_k e_k = e_k - tau_k v_k, then H_{k-1}, ..., H_0
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    const int k = warp + W * s;
    if (k >= l) continue;
    const HqrCol<R2> v = hqr_load_v<R2>(hqr_v + k * PP, lane);
#pragma unroll
    for (int t = 0; t < R2; ++t) {
      const int r = 64 * t + 2 * lane;
      x[s].re[t] = make_float2(r == k ? 1.f : 0.f, r + 1 == k ? 1.f : 0.f);
      x[s].im[t] = make_float2(0.f, 0.f);
    }
    hqr_update<R2>(v, x[s], tau_s[k], 1.f, 0.f);
  }
#pragma unroll 1
  for (int i = l - 2; i >= 0; --i) {
    const float2 tau = tau_s[i];
    if (tau.x == 0.f && tau.y == 0.f) continue;
    const HqrCol<R2> v = hqr_load_v<R2>(hqr_v + i * PP, lane);
    hqr_apply<R2, W, SLOTS>(v, x, 0, i, l, tau, warp, lane);
  }
  const bool split = MODE == HQR_WHOLE && g.sp.p0 != nullptr;
  const int64_t sbase = split ? int64_t(f) * g.sp.ldk * lfull : 0;
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    const int k = warp + W * s;
    if (k >= lfull) continue;
    const float sg = (g.keep_phase && k < l && beta_s[k] < 0.f) ? -1.f : 1.f;
#pragma unroll
    for (int i = 0; i < 2 * R2; ++i) {
      const int r = 64 * (i >> 1) + 2 * lane + (i & 1);
      const bool in = k < l && r < p;
      const float qr = in ? sg * ((i & 1) ? x[s].re[i >> 1].y : x[s].re[i >> 1].x) : 0.f;
      const float qi = in ? sg * ((i & 1) ? x[s].im[i >> 1].y : x[s].im[i >> 1].x) : 0.f;
      if (r < p) {
        yr[r + ld * k] = qr;
        yi[r + ld * k] = qi;
      }
      if (split && r < g.sp.ldk) {
        const int64_t o = sbase + r + g.sp.ldk * k;
        dftc::put_split(g.sp.p0, g.sp.p1, g.sp.bf16 != 0, o, qr);
        dftc::put_split(g.sp.p2, g.sp.p3, g.sp.bf16 != 0, o, qi);
      }
    }
  }
}

// Q of one block of a tall slice: its reflectors (in Y) applied to its l rows
// of the parent's Q (in the stack), written over the reflectors.  A flagged
// slice is left zero (or not a number) instead.
template <int R2, int W, int SLOTS>
__global__ void __launch_bounds__(32 * W, HqrResident<R2, W, SLOTS>::v)
    hqr_form_kernel(const HqrParams g) {
  constexpr int PP = 32 * R2;
  extern __shared__ __align__(16) float4 hqr_v[];
  __shared__ float2 tau_s[HQR_MAX_L];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int f = int(blockIdx.x) / g.nb, b = int(blockIdx.x) - f * g.nb;
  const int lfull = g.lfull;
  const int l = g.lcols ? min(max(int(g.lcols[f]), 1), lfull) : lfull;
  int r0, p;
  hqr_block(g.rows, g.nb, b, r0, p);
  float* yr = g.yr + int64_t(f) * g.sY + r0;
  float* yi = g.yi + int64_t(f) * g.sY + r0;
  const int64_t ld = g.rows;
  const int bad = g.flag[f];
  const float2* tau = g.tau + (int64_t(f) * g.nb + b) * lfull;
  const int64_t lr = int64_t(g.nb) * lfull;
  const float* cr = g.rr + int64_t(f) * lr * lfull + int64_t(b) * lfull;
  const float* ci = g.ri + int64_t(f) * lr * lfull + int64_t(b) * lfull;
  for (int j = threadIdx.x; j < l; j += 32 * W) tau_s[j] = tau[j];
  HqrCol<R2> x[SLOTS];
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    const int k = warp + W * s;
#pragma unroll
    for (int t = 0; t < R2; ++t) {
      const int r = 64 * t + 2 * lane;
      const int64_t o = r + ld * k, c = r + lr * k;
      const bool in = k < l, q0 = in && r < l, q1 = in && r + 1 < l;
      if (in)
        hqr_v[k * PP + 32 * t + lane] =
            make_float4(r < p ? yr[o] : 0.f, r + 1 < p ? yr[o + 1] : 0.f, r < p ? yi[o] : 0.f,
                        r + 1 < p ? yi[o + 1] : 0.f);
      x[s].re[t] = make_float2(q0 ? cr[c] : 0.f, q1 ? cr[c + 1] : 0.f);
      x[s].im[t] = make_float2(q0 ? ci[c] : 0.f, q1 ? ci[c + 1] : 0.f);
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int i = l - 1; i >= 0; --i) {
    const float2 ti = tau_s[i];
    if (ti.x == 0.f && ti.y == 0.f) continue;
    const HqrCol<R2> v = hqr_load_v<R2>(hqr_v + i * PP, lane);
    hqr_apply<R2, W, SLOTS>(v, x, 0, -1, l, ti, warp, lane);
  }
  const float fill = bad == 2 ? __int_as_float(0x7fc00000) : 0.f;
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    const int k = warp + W * s;
    if (k >= lfull) continue;
#pragma unroll
    for (int i = 0; i < 2 * R2; ++i) {
      const int r = 64 * (i >> 1) + 2 * lane + (i & 1);
      if (r >= p) continue;
      const float qr = (i & 1) ? x[s].re[i >> 1].y : x[s].re[i >> 1].x;
      const float qi = (i & 1) ? x[s].im[i >> 1].y : x[s].im[i >> 1].x;
      yr[r + ld * k] = k >= l ? 0.f : bad ? fill : qr;
      yi[r + ld * k] = k >= l ? 0.f : bad ? fill : qi;
    }
  }
}

// Launch of MODE (or, FORM, of hqr_form_kernel) with the register shape that
// holds p rows and l columns.
constexpr int HQR_FORM = 3;

template <int R2, int W, int SLOTS, int MODE>
int hqr_launch(const HqrParams& g, int64_t blocks, cudaStream_t st) {
  const size_t smem = size_t(32 * R2) * g.lfull * sizeof(float4);
  if constexpr (MODE == HQR_FORM) {
    auto k = hqr_form_kernel<R2, W, SLOTS>;
    TP_SET_SMEM(k, smem);
    k<<<unsigned(blocks), 32 * W, smem, st>>>(g);
  } else {
    auto k = hqr_kernel<R2, W, SLOTS, MODE>;
    TP_SET_SMEM(k, smem);
    k<<<unsigned(blocks), 32 * W, smem, st>>>(g);
  }
  return launch_status("householder_qr");
}

template <int MODE>
int hqr_dispatch(const HqrParams& g, int p, int64_t blocks, cudaStream_t st) {
  const int l = g.lfull;
  KernelScope ks("householder_qr", st);
  if (p <= 64) {   // l <= p
    if (l <= 32) return hqr_launch<1, 8, 4, MODE>(g, blocks, st);
    return hqr_launch<1, 16, 4, MODE>(g, blocks, st);
  }
  if (p <= 128) {
    if (l <= 32) return hqr_launch<2, 8, 4, MODE>(g, blocks, st);
    if (l <= 64) return hqr_launch<2, 16, 4, MODE>(g, blocks, st);
    return hqr_launch<2, 16, 6, MODE>(g, blocks, st);
  }
  if (l <= 32) return hqr_launch<4, 16, 2, MODE>(g, blocks, st);
  if (l <= 64) return hqr_launch<4, 16, 4, MODE>(g, blocks, st);
  return hqr_launch<4, 16, 6, MODE>(g, blocks, st);
}

// ---------------------------------------------------------------- in shared memory
//
// The same QR of a slice of at most 256 rows held in shared memory, a step's
// reflector in registers (lane r % 32 holds rows r) and a warp per column.  It
// is a few percent slower than the registers' form above and rounds in another
// order.  Sketches with at most one power iteration take it: there the trailing
// singular values are set by the rounding of the core's Gram matrix (rsvd.cu),
// so that another order of the sums here moves them by more than rounding.
constexpr int HQS_THREADS = 256;
constexpr int HQS_WARPS = HQS_THREADS / 32;

// Reflector of column a (rows j .. p-1), one warp: rows j+1.. become v,
// row j becomes beta; returns tau (0 when the column is already beta e_j with
// beta real).
__device__ float2 hqs_reflector(float2* a, int j, int p, int lane) {
  const float2 al = a[j];
  float s = 0.f;
  for (int r = j + 1 + lane; r < p; r += 32) {
    const float2 x = a[r];
    s = fmaf(x.x, x.x, fmaf(x.y, x.y, s));
  }
  s = hqr_sum(s);
  if (s == 0.f && al.y == 0.f) return make_float2(0.f, 0.f);
  const float nrm = sqrtf(fmaf(al.x, al.x, fmaf(al.y, al.y, s)));
  const float beta = al.x >= 0.f ? -nrm : nrm;
  // v = x / (alpha - beta); |alpha - beta| >= nrm > 0 by the sign of beta
  const float dr = al.x - beta, di = al.y;
  const float den = fmaf(dr, dr, di * di);
  const float sr = dr / den, si = -di / den;
  for (int r = j + 1 + lane; r < p; r += 32) {
    const float2 x = a[r];
    a[r] = make_float2(x.x * sr - x.y * si, x.x * si + x.y * sr);
  }
  __syncwarp();
  if (lane == 0) a[j] = make_float2(beta, 0.f);
  return make_float2((beta - al.x) / beta, -al.y / beta);
}

// v_j of column a into registers: row r = lane + 32 t, 1 at row j, 0 above.
template <int RPL>
__device__ __forceinline__ void hqs_load_v(const float2* a, int j, int p, int lane,
                                           float2 (&v)[RPL]) {
#pragma unroll
  for (int t = 0; t < RPL; ++t) {
    const int r = lane + 32 * t;
    v[t] = (r <= j || r >= p) ? make_float2(r == j ? 1.f : 0.f, 0.f) : a[r];
  }
}

// c <- c - f v (v^H c) on rows j .. p-1 (f = conj(tau) applies H^H, f = tau H)
template <int RPL>
__device__ __forceinline__ void hqs_apply(const float2 (&v)[RPL], float2* c, int j, int p, float2 f,
                                          int lane) {
  float2 x[RPL];
  float dr = 0.f, di = 0.f;
#pragma unroll
  for (int t = 0; t < RPL; ++t) {
    const int r = lane + 32 * t;
    x[t] = (r >= j && r < p) ? c[r] : make_float2(0.f, 0.f);
    dr = fmaf(v[t].x, x[t].x, fmaf(v[t].y, x[t].y, dr));    // Re(conj(v) x)
    di = fmaf(v[t].x, x[t].y, fmaf(-v[t].y, x[t].x, di));   // Im(conj(v) x)
  }
  hqr_sum2(dr, di, lane);
  const float gr = f.x * dr - f.y * di, gi = f.x * di + f.y * dr;
#pragma unroll
  for (int t = 0; t < RPL; ++t) {
    const int r = lane + 32 * t;
    if (r >= j && r < p)
      c[r] = make_float2(x[t].x - (v[t].x * gr - v[t].y * gi),
                         x[t].y - (v[t].x * gi + v[t].y * gr));
  }
}

// Column k of Q from its reflector (stored in place): H_k e_k restricted to
// rows k.. -- 1 - tau at row k, -tau v below -- and zeros above.
__device__ __forceinline__ void hqs_materialize(float2* a, int k, int p, float2 tau, int lane) {
  for (int r = lane; r < p; r += 32) {
    float2 y;
    if (r < k) {
      y = make_float2(0.f, 0.f);
    } else if (r == k) {
      y = make_float2(1.f - tau.x, -tau.y);
    } else {
      const float2 v = a[r];
      y = make_float2(-(tau.x * v.x - tau.y * v.y), -(tau.x * v.y + tau.y * v.x));
    }
    a[r] = y;
  }
}

// One CTA per slice; RPL rows per lane (p <= 32 RPL).
template <int RPL>
__global__ void __launch_bounds__(HQS_THREADS) householder_shared_kernel(float* y_re, float* y_im,
                                                                         int64_t sY, int p,
                                                                         int lfull,
                                                                         const int32_t* lcols) {
  extern __shared__ __align__(16) float2 hqs_a[];   // Y, then Q: p x l column-major
  __shared__ float2 tau_s[HQR_MAX_L];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int l = lcols ? min(max(int(lcols[blockIdx.x]), 1), lfull) : lfull;
  float* yr = y_re + int64_t(blockIdx.x) * sY;
  float* yi = y_im + int64_t(blockIdx.x) * sY;
  float2* A = hqs_a;
  for (int e = threadIdx.x; e < p * l; e += HQS_THREADS) A[e] = make_float2(yr[e], yi[e]);
  __syncthreads();
  if (warp == 0) {
    const float2 t = hqs_reflector(A, 0, p, lane);
    if (lane == 0) tau_s[0] = t;
  }
  __syncthreads();
  // factorisation: step j applies H_j^H to columns j+1 .. l-1
  for (int j = 0; j + 1 < l; ++j) {
    const float2 tau = tau_s[j];
    float2 v[RPL];
    hqs_load_v<RPL>(A + int64_t(j) * p, j, p, lane, v);
    const bool live = tau.x != 0.f || tau.y != 0.f;
    const float2 f = make_float2(tau.x, -tau.y);
    int k = j + 1 + warp;
    if (warp == 0) {   // look-ahead: column j + 1 first, then its reflector
      float2* c = A + int64_t(k) * p;
      if (live) hqs_apply<RPL>(v, c, j, p, f, lane);
      __syncwarp();
      const float2 t = hqs_reflector(c, k, p, lane);
      if (lane == 0) tau_s[k] = t;
      k += HQS_WARPS;
    }
    if (live)
      for (; k < l; k += HQS_WARPS) hqs_apply<RPL>(v, A + int64_t(k) * p, j, p, f, lane);
    __syncthreads();
  }
  // Q = H_0 ... H_{l-1} [I; 0]: step i applies H_i to columns i+1 .. l-1,
  // whose first (column i + 1) its owner first turns from reflector storage
  // into H_{i+1} e_{i+1}
  for (int i = l - 2; i >= 0; --i) {
    const float2 tau = tau_s[i];
    float2 v[RPL];
    hqs_load_v<RPL>(A + int64_t(i) * p, i, p, lane, v);
    int k = i + 1 + warp;
    if (warp == 0) {
      hqs_materialize(A + int64_t(k) * p, k, p, tau_s[k], lane);
      __syncwarp();
    }
    if (tau.x != 0.f || tau.y != 0.f)
      for (; k < l; k += HQS_WARPS) hqs_apply<RPL>(v, A + int64_t(k) * p, i, p, tau, lane);
    __syncthreads();
  }
  if (warp == 0) hqs_materialize(A, 0, p, tau_s[0], lane);
  __syncthreads();
  for (int e = threadIdx.x; e < p * lfull; e += HQS_THREADS) {
    const float2 q = e < p * l ? A[e] : make_float2(0.f, 0.f);
    yr[e] = q.x;
    yi[e] = q.y;
  }
}

template <int RPL>
int hqs_launch(float* yr, float* yi, int64_t sY, int p, int l, const int32_t* lcols, int64_t batch,
               cudaStream_t st) {
  const size_t smem = size_t(p) * l * sizeof(float2);
  TP_SET_SMEM(householder_shared_kernel<RPL>, smem);
  {
    KernelScope ks("householder_qr", st);
    householder_shared_kernel<RPL><<<unsigned(batch), HQS_THREADS, smem, st>>>(yr, yi, sY, p, l,
                                                                              lcols);
  }
  return launch_status("householder_shared_kernel");
}

constexpr int HQR_BLOCK = 256;

}  // namespace

bool householder_applies(int64_t p, int64_t l) { return p <= HQR_BLOCK && l <= HQR_MAX_L; }

int householder_launch(float* yr, float* yi, int64_t sY, int p, int l, const int32_t* lcols,
                       bool keep_phase, int64_t batch, cudaStream_t st, HqrSplit sp) {
  if (p > HQR_BLOCK || l > HQR_MAX_L || l > p) {
    set_error("householder: needs l <= p <= %d and l <= %d", HQR_BLOCK, HQR_MAX_L);
    return TP_EUNSUPPORTED;
  }
  if (batch <= 0 || l <= 0) return TP_OK;
  HqrParams g{};
  g.yr = yr;
  g.yi = yi;
  g.sY = sY;
  g.rows = p;
  g.nb = 1;
  g.lfull = l;
  g.lcols = lcols;
  g.keep_phase = keep_phase ? 1 : 0;
  g.sp = sp;
  return hqr_dispatch<HQR_WHOLE>(g, p, batch, st);
}

int householder_shared_launch(float* yr, float* yi, int64_t sY, int p, int l, const int32_t* lcols,
                              int64_t batch, cudaStream_t st) {
  if (p > HQR_BLOCK || l > HQR_MAX_L || l > p) {
    set_error("householder_shared: needs l <= p <= %d and l <= %d", HQR_BLOCK, HQR_MAX_L);
    return TP_EUNSUPPORTED;
  }
  if (batch <= 0 || l <= 0) return TP_OK;
  if (p <= 64) return hqs_launch<2>(yr, yi, sY, p, l, lcols, batch, st);
  if (p <= 128) return hqs_launch<4>(yr, yi, sY, p, l, lcols, batch, st);
  return hqs_launch<8>(yr, yi, sY, p, l, lcols, batch, st);
}

// Scratch of householder_tall_launch: per level below the top the R stack
// (two float planes), the taus and the exponents, and the flags.
size_t householder_tall_scratch(int64_t rows, int64_t l, int64_t batch) {
  size_t total = ws_bytes(size_t(batch), 4);
  while (rows > HQR_BLOCK) {
    const int64_t nb = (rows + HQR_BLOCK - 1) / HQR_BLOCK;
    total += 2 * ws_bytes(size_t(nb) * l * l * batch, 4) + ws_bytes(size_t(nb) * l * batch, 8) +
             ws_bytes(size_t(nb) * batch, 4);
    rows = nb * l;
  }
  return total;
}

int householder_tall_launch(float* yr, float* yi, int64_t rows, int l, const int32_t* lcols,
                            int64_t batch, void* scratch, int32_t* status, cudaStream_t st) {
  constexpr int kMaxLevels = 24;   // each level shrinks the rows by 256 / 96 at least
  if (l < 1 || l > HQR_MAX_L || rows <= HQR_BLOCK || rows > 0x7fffffff) {
    set_error("householder_tall: needs more than %d rows and l <= %d", HQR_BLOCK, HQR_MAX_L);
    return TP_EUNSUPPORTED;
  }
  Arena ws;
  ws.base = static_cast<char*>(scratch);
  int* flag = ws.take<int>(size_t(batch));
  HqrParams lev[kMaxLevels];
  int n = 0, rc = TP_OK;
  float *cr = yr, *ci = yi;
  const int* ex = nullptr;
  auto block_rows = [](const HqrParams& g) { return (g.rows + g.nb - 1) / g.nb; };
  while (rc == TP_OK) {
    HqrParams g{};
    g.yr = cr;
    g.yi = ci;
    g.sY = rows * l;
    g.rows = int(rows);
    g.nb = int((rows + HQR_BLOCK - 1) / HQR_BLOCK);
    g.lfull = l;
    g.lcols = lcols;
    g.ex_in = ex;
    g.flag = flag;
    g.status = status;
      if (batch * g.nb > 0x7fffffff || (g.nb > 1 && n == kMaxLevels)) {
      set_error("householder_tall: too many blocks");
      return TP_EUNSUPPORTED;
    }
    if (g.nb == 1) {
      rc = hqr_dispatch<HQR_TOP>(g, block_rows(g), batch, st);
      break;
    }
    g.rr = ws.take<float>(size_t(g.nb) * l * l * batch);
    g.ri = ws.take<float>(size_t(g.nb) * l * l * batch);
    g.tau = ws.take<float2>(size_t(g.nb) * l * batch);
    g.ex_out = ws.take<int>(size_t(g.nb) * batch);
    rc = hqr_dispatch<HQR_FACTOR>(g, block_rows(g), batch * g.nb, st);
    lev[n++] = g;
    cr = g.rr;
    ci = g.ri;
    ex = g.ex_out;
    rows = int64_t(g.nb) * l;
  }
  while (rc == TP_OK && n > 0) {
    const HqrParams& g = lev[--n];
    rc = hqr_dispatch<HQR_FORM>(g, block_rows(g), batch * g.nb, st);
  }
  return rc;
}

}  // namespace tp
