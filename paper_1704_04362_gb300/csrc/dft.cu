// Mode-3 DFT of real tubes kept to the half spectrum, and its inverse
// (Section 2, "Operators": fft(X,[],3) / ifft(X,[],3); Algorithm 1 steps 2-3
// and the final inverse).
//
// The transforms of lengths that neither rfft_reg.cu (registers) nor fft.cu
// (primes up to 13) takes, and the choice among the three.  Both directions
// are small dense contractions per tube.  The t <-> n3 - t
// symmetry halves them: with e_t = x_t + x_{n3-t} and o_t = x_t - x_{n3-t}
// (t = 1 .. n3/2; e_0 = x_0 and, for even n3, e_{n3/2} = x_{n3/2}, o = 0 there),
//     Re X_k = sum_{t <= n3/2} e_t cos(2 pi k t / n3),
//     Im X_k = -sum_{t <= n3/2} o_t sin(2 pi k t / n3);
// and for the inverse, with P_t = sum_k w_k Re X_k cos, Q_t = sum_k w_k Im X_k sin
// (w_k = 1/n3 at k = 0 and k = n3/2, else 2/n3), x_t = P_t - Q_t and
// x_{n3-t} = P_t + Q_t.  Over all tubes these are two real matrix products
// with a common schedule (dft_product_kernel); each sum runs in order.
#include <algorithm>

#include "dft_common.cuh"

namespace tp {
namespace {
using namespace dftc;

constexpr int RB = 128;          // threads per block of the transposed kernel
constexpr int TU = 8;            // samples it loads ahead

// (cos, sin)(2 pi m / n3) for m < n3.  float sincospi (about 1 ulp; exact at
// quarter turns, m/n3 in {0, 1/4, 1/2, 3/4}) keeps the tables off the slow
// float64 pipe.  The argument 2m/n3 is formed exactly enough: 2m and n3 are
// small integers, and the quotient's rounding (2^-24 relative) moves the angle
// by less than the float result's own rounding.
__device__ __forceinline__ void build_twiddles(float2* tw, int n3) {
  for (int m = threadIdx.x; m < n3; m += blockDim.x) {
    float s, c;
    sincospif(float(2 * m) / float(n3), &s, &c);
    tw[m] = make_float2(c, s);
  }
}

// The transforms as matrix products: M = tubes, N = outputs (frequencies k of
// the forward, times t <= n3/2 of the inverse), K = folded samples t (or
// frequencies k), two products side by side (e cos | -o sin; w Re cos | w Im sin).
// A block of TX x TY threads owns 4 TX tubes and 4 TY outputs, a thread 4 tubes
// x 4 outputs of both products as tube pairs on the packed two-lane FMA.  The
// K x 4 TY table of the transform matrix stays in shared memory while the
// block walks its tubes; the tubes come in K tiles of 8, folded on the way from
// registers to shared memory, the next tile's samples loaded before the
// current one is used.  The whole half spectrum of a tube of up to 239 samples is
// produced by one block, so each sample is read once (longer tubes take the
// outputs in as many parts as their table needs shared memory).
// Bound by the float32 pipe for n3 above about 60, below by the tubes' traffic.
// 218880 tubes, one output per thread and tube group in chunks of 16 (table
// rebuilt per chunk) -> this: n3 = 67 forward 0.22 -> 0.11 ms, inverse 0.079 ->
// 0.065; n3 = 127 0.62 -> 0.18, 0.19 -> 0.12; n3 = 251 3.6 -> 0.87, 0.75 -> 0.47.
constexpr int DK = 8;                        // K tile
constexpr int DN = 4, DM = 4;                // outputs and tubes per thread
constexpr int TABLE_BYTES_MAX = 120 * 1024;
constexpr int DT_MAX = 480;                  // threads: 16 x 30 groups, n3 = 232 .. 239

struct DftArgs {
  DftGather g;                // forward
  const float *in_re, *in_im; // inverse
  float* out;
  int64_t rows, in_slice;
  int n3, K, N, parts;        // K terms, N outputs a part, parts of the outputs
  int tx_log, ty;             // block shape
};

// NP: K-tile samples per thread; MT, MB: threads a block and blocks per SM the
// registers are budgeted for (80 registers keep 22 to 24 warps on an SM).
template <bool INV, int NP, int MT, int MB>
__global__ void __launch_bounds__(MT, MB) dft_product_kernel(const __grid_constant__ DftArgs p) {
  extern __shared__ __align__(16) float dft_sm[];
  const int n3 = p.n3, h = n3 / 2 + 1, K = p.K, KP = (K + DK - 1) / DK * DK;
  const int TX = 1 << p.tx_log, BM = DM * TX, NO = DN * p.ty, nt = TX * p.ty;
  const int tid = threadIdx.x, tx = tid & (TX - 1), ty = tid >> p.tx_log;
  const int q0 = int(blockIdx.y) * p.N;      // first output of this part
  float2* W = reinterpret_cast<float2*>(dft_sm);                 // [KP][NO]
  float* Ab = dft_sm + 2 * KP * NO;                               // [2][2][DK][BM]
  const float** base = reinterpret_cast<const float**>(Ab + 4 * DK * BM);   // [BM]
  int64_t* offs = reinterpret_cast<int64_t*>(base + BM);         // [BM], -1 past the data
  float* scl = reinterpret_cast<float*>(offs + BM);              // [BM]
  float2* tw = reinterpret_cast<float2*>(scl + BM);              // [n3]
  build_twiddles(tw, n3);
  __syncthreads();
  const float inv = 1.0f / float(n3);
  for (int e = tid; e < KP * NO; e += nt) {
    const int t = e / NO, q = q0 + e - t * NO;
    float2 w = make_float2(0.f, 0.f);
    if (q < h && t < K) {
      w = tw[int((int64_t(q) * t) % n3)];
      if (INV) {
        const float wk = (t == 0 || 2 * t == n3) ? inv : 2.0f * inv;
        w = make_float2(wk * w.x, wk * w.y);
      } else {
        w.y = -w.y;
      }
    }
    W[e] = w;
  }
  Extent ex{};
  int64_t total;
  if (INV) {
    total = p.rows;
  } else {
    ex = extent_of(p.g);
    total = ex.rows_pad * ex.cols_pad;
  }
  const int64_t ss = INV ? p.in_slice : p.g.slice_stride;

  float v0[NP], v1[NP];
  // raw values of K tile k0 of the current tubes, into registers
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < NP; ++u) {
      const int e = tid + u * nt, m = e & (BM - 1), t = k0 + (e >> (p.tx_log + 2));
      v0[u] = v1[u] = 0.f;
      if (e >= DK * BM || t >= K) continue;
      const float* b = base[m];
      if (!b) continue;
      const float* a = b + int64_t(t) * ss;
      if (INV) {
        v0[u] = __ldg(a);
        // the imaginary parts of the real slices are ignored
        if (t > 0 && 2 * t != n3) v1[u] = __ldg(p.in_im + (a - p.in_re));
      } else {
        v0[u] = scl[m] * __ldg(a);
        if (t > 0 && 2 * t != n3) v1[u] = scl[m] * __ldg(b + int64_t(n3 - t) * ss);
      }
    }
  };
  auto stage = [&](int k0, float* A) {   // A: [2][DK][BM]
#pragma unroll
    for (int u = 0; u < NP; ++u) {
      const int e = tid + u * nt;
      if (e >= DK * BM) continue;
      const int t = k0 + (e >> (p.tx_log + 2));
      const bool lone = t == 0 || 2 * t == n3;
      A[e] = INV ? v0[u] : lone ? v0[u] : v0[u] + v1[u];
      A[DK * BM + e] = INV ? v1[u] : lone ? 0.f : v0[u] - v1[u];
    }
  };

  for (int64_t m0 = int64_t(blockIdx.x) * BM; m0 < total; m0 += int64_t(gridDim.x) * BM) {
    __syncthreads();   // the previous tubes' addresses and tiles are done with
    for (int m = tid; m < BM; m += nt) {
      const int64_t e = m0 + m;
      const bool in = e < total;
      if (INV) {
        base[m] = in ? p.in_re + e : nullptr;
        offs[m] = in ? e : -1;
      } else {
        const int64_t c = in ? e / ex.rows_pad : 0, r = in ? e - c * ex.rows_pad : 0;
        float s = 0.f;
        base[m] = in ? tube_ptr(p.g, ex, r, c, s) : nullptr;
        scl[m] = s;
        offs[m] = in ? r + p.g.out_ld * c : -1;
      }
    }
    __syncthreads();
    float2 a0[2][DN], a1[2][DN];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int q = 0; q < DN; ++q) a0[i][q] = a1[i][q] = make_float2(0.f, 0.f);
    fetch(0);
    int buf = 0;
    for (int k0 = 0; k0 < K; k0 += DK, buf ^= 1) {
      float* A = Ab + buf * 2 * DK * BM;
      stage(k0, A);
      __syncthreads();   // also: every thread is done with the other buffer's last use
      if (k0 + DK < K) fetch(k0 + DK);
#pragma unroll 2
      for (int kk = 0; kk < DK; ++kk) {   // zero samples past K
        const float4 x = *reinterpret_cast<const float4*>(A + kk * BM + DM * tx);
        const float4 y = *reinterpret_cast<const float4*>(A + (DK + kk) * BM + DM * tx);
        const float2 xe[2] = {make_float2(x.x, x.y), make_float2(x.z, x.w)};
        const float2 yo[2] = {make_float2(y.x, y.y), make_float2(y.z, y.w)};
        const float4* w4 = reinterpret_cast<const float4*>(W + (k0 + kk) * NO + DN * ty);
#pragma unroll
        for (int q = 0; q < DN; q += 2) {
          const float4 w = w4[q / 2];
          const float2 c0 = make_float2(w.x, w.x), s0 = make_float2(w.y, w.y);
          const float2 c1 = make_float2(w.z, w.z), s1 = make_float2(w.w, w.w);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            a0[i][q] = __ffma2_rn(xe[i], c0, a0[i][q]);
            a1[i][q] = __ffma2_rn(yo[i], s0, a1[i][q]);
            a0[i][q + 1] = __ffma2_rn(xe[i], c1, a0[i][q + 1]);
            a1[i][q + 1] = __ffma2_rn(yo[i], s1, a1[i][q + 1]);
          }
        }
      }
    }
    // outputs q of the thread's four tubes; four consecutive ones in one store
    // where their place is aligned
    const int64_t o0 = offs[DM * tx], o3 = offs[DM * tx + 3];
    const bool quad = o0 >= 0 && o3 == o0 + 3 && (o0 & 3) == 0;
    auto put4 = [&](float* dst, int64_t shift, bool aligned, const float (&v)[4]) {
      if (quad && aligned) {
        *reinterpret_cast<float4*>(dst + shift + o0) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int64_t o = offs[DM * tx + j];
          if (o >= 0) dst[shift + o] = v[j];
        }
      }
    };
#pragma unroll
    for (int q = 0; q < DN; ++q) {
      const int k = q0 + DN * ty + q;
      if (DN * ty + q >= p.N || k >= h) continue;
      const float u[4] = {a0[0][q].x, a0[0][q].y, a0[1][q].x, a0[1][q].y};
      const float v[4] = {a1[0][q].x, a1[0][q].y, a1[1][q].x, a1[1][q].y};
      if (INV) {
        const bool al = (p.rows & 3) == 0 && aligned16(p.out);
        float lo[4], hi[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          lo[j] = u[j] - v[j];
          hi[j] = u[j] + v[j];
        }
        put4(p.out, p.rows * int64_t(k), al, lo);
        if (k > 0 && n3 - k > n3 / 2) put4(p.out, p.rows * int64_t(n3 - k), al, hi);
      } else if (p.g.out_re_lo) {
        const int64_t shift = int64_t(k) * p.g.out_slice;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int64_t o = offs[DM * tx + j];
          if (o < 0) continue;
          put_split(p.g.out_re, p.g.out_re_lo, p.g.out_bf16 != 0, shift + o, u[j]);
          put_split(p.g.out_im, p.g.out_im_lo, p.g.out_bf16 != 0, shift + o, v[j]);
        }
      } else {
        const bool al = (p.g.out_slice & 3) == 0;
        const int64_t shift = int64_t(k) * p.g.out_slice;
        put4(p.g.out_re, shift, al && aligned16(p.g.out_re), u);
        put4(p.g.out_im, shift, al && aligned16(p.g.out_im), v);
      }
    }
  }
}

// Same transform, written transposed: element (r, c) of slice k goes to
// out[k*out_slice + c + out_ld*r], so that the picked-slice index (the
// facewise product's inner dimension) is contiguous.  A block owns a tile of
// 32 rows x 8 columns (rows fastest, so tube reads stay coalesced); each
// frequency chunk is staged through shared memory and stored as 32-byte runs
// along the column index.  This kernel runs the plain (unfolded) contraction:
// the folded form's extra live registers cost more occupancy than the
// arithmetic it saves here.
constexpr int TR = 32, TCOL = 8;
constexpr int TPTT = TCOL / (RB / TR);   // columns per thread in the transposed kernel (2)

template <int KC>
__global__ void __launch_bounds__(RB) rdft_t_kernel(DftGather g) {
  extern __shared__ float2 sm2[];
  const int n3 = int(g.n3);
  const int h = n3 / 2 + 1;
  const int n3p = (n3 + TU - 1) / TU * TU;
  float2* tw = sm2;
  float2* Wc = sm2 + n3;   // Wc[t*KC + q] = tw[(k0+q) t mod n3], zero for t >= n3
  float* stg = reinterpret_cast<float*>(Wc + n3p * KC);   // [KC][TR][TCOL + 1]
  build_twiddles(tw, n3);
  const Extent ex = extent_of(g);
  const int64_t r0 = int64_t(blockIdx.x) * TR;
  if (r0 >= ex.rows_pad) return;   // uniform over the block
  const int tid = threadIdx.x;
  const int lr = tid % TR, lc = tid / TR;   // this thread: row lr, columns lc and lc + 4
  const int64_t r = r0 + lr;

  for (int64_t c0 = int64_t(blockIdx.y) * TCOL; c0 < ex.cols_pad; c0 += int64_t(gridDim.y) * TCOL) {
    const float* p[TPTT];
    float s[TPTT];
#pragma unroll
    for (int j = 0; j < TPTT; ++j) p[j] = tube_ptr(g, ex, r, c0 + lc + 4 * j, s[j]);
    for (int k0 = 0; k0 < h; k0 += KC) {
      __syncthreads();
      for (int e = tid; e < n3p * KC; e += RB) {
        const int t = e / KC, q = e - t * KC;
        Wc[e] = t < n3 ? tw[int((int64_t(k0 + q) * t) % n3)] : make_float2(0.f, 0.f);
      }
      __syncthreads();
      float2 acc[TPTT][KC];   // (Re, Im), updated by packed two-lane FMAs
#pragma unroll
      for (int j = 0; j < TPTT; ++j)
#pragma unroll
        for (int q = 0; q < KC; ++q) acc[j][q] = make_float2(0.f, 0.f);
      for (int t0 = 0; t0 < n3; t0 += TU) {
        float x[TPTT][TU];
#pragma unroll
        for (int u = 0; u < TU; ++u)
#pragma unroll
          for (int j = 0; j < TPTT; ++j)
            x[j][u] = (p[j] && t0 + u < n3) ? s[j] * __ldg(p[j] + int64_t(t0 + u) * g.slice_stride)
                                            : 0.f;
#pragma unroll
        for (int u = 0; u < TU; ++u)
#pragma unroll
          for (int q = 0; q < KC; ++q) {
            const float2 w = Wc[(t0 + u) * KC + q];
#pragma unroll
            for (int j = 0; j < TPTT; ++j)
              acc[j][q] = __ffma2_rn(make_float2(x[j][u], -x[j][u]), w, acc[j][q]);
          }
      }
      // planes: 0 re (hi), 1 im (hi), 2 re lo, 3 im lo
      const int nplanes = g.out_re_lo ? 4 : 2;
      for (int pl = 0; pl < nplanes; ++pl) {
        __syncthreads();   // staging buffer free
#pragma unroll
        for (int j = 0; j < TPTT; ++j)
#pragma unroll
          for (int q = 0; q < KC; ++q) {
            const float v = (pl & 1) ? acc[j][q].y : acc[j][q].x;
            float o;
            if (!g.out_re_lo) {
              o = v;
            } else {   // hi, or lo = v - hi rounded to tf32 (a bf16 lo is rounded when stored)
              const float hi = g.out_bf16 ? __bfloat162float(__float2bfloat16_rn(v)) : tf32_rna(v);
              o = pl < 2 ? hi : (g.out_bf16 ? v - hi : tf32_rna(v - hi));
            }
            stg[(q * TR + lr) * (TCOL + 1) + lc + 4 * j] = o;
          }
        __syncthreads();
        float* dst = pl == 0 ? g.out_re : pl == 1 ? g.out_im : pl == 2 ? g.out_re_lo : g.out_im_lo;
        // thread -> (column wc, row wr); 16 rows per pass, two passes
        const int wc = tid % TCOL, wr = tid / TCOL;
        const int64_t c = c0 + wc;
        if (c < ex.cols_pad) {
          for (int q = 0; q < KC && k0 + q < h; ++q) {
#pragma unroll
            for (int pass = 0; pass < TR / (RB / TCOL); ++pass) {
              const int rr = wr + pass * (RB / TCOL);
              const int64_t rg = r0 + rr;
              if (rg < ex.rows_pad) {
                const int64_t o = int64_t(k0 + q) * g.out_slice + c + g.out_ld * rg;
                const float v = stg[(q * TR + rr) * (TCOL + 1) + wc];
                if (g.out_bf16 && g.out_re_lo)
                  reinterpret_cast<__nv_bfloat16*>(dst)[o] = __float2bfloat16_rn(v);
                else
                  dst[o] = v;
              }
            }
          }
        }
      }
    }
  }
}

// Chunk size among {16, 12, 8} that pads n the least (ties: larger).
int pick_kc(int64_t n) {
  const int cands[3] = {16, 12, 8};
  int best = 16;
  int64_t best_cost = -1;
  for (int kc : cands) {
    const int64_t cost = (n + kc - 1) / kc * kc;
    if (best_cost < 0 || cost < best_cost) {
      best = kc;
      best_cost = cost;
    }
  }
  return best;
}

// The transposed form (a tuned tile width KC).
template <int KC>
int launch_rdft_t(const DftGather& g, cudaStream_t st) {
  const int64_t n3p = (g.n3 + TU - 1) / TU * TU;
  const size_t smem = size_t(g.n3 + n3p * KC) * sizeof(float2) +
                      size_t(KC) * TR * (TCOL + 1) * sizeof(float);
  TP_SET_SMEM(rdft_t_kernel<KC>, smem);
  const int64_t bx = (g.rows + TR - 1) / TR;
  if (bx > 0x7fffffff) { set_error("rdft: too many rows"); return TP_EINVAL; }
  // the column tiles are walked grid-stride: with all rows live (no row
  // gather) about 16 blocks per SM suffice, and a column gather's capacity
  // can far exceed the picked count
  int64_t by = (g.cols + TCOL - 1) / TCOL;
  const int64_t by_cap = bx >= int64_t(sm_count()) * 16 ? 1 : int64_t(sm_count()) * 16 / bx;
  if (g.gather_dim != 1 && by > by_cap) by = by_cap;
  if (by > 65535) by = 65535;
  {
    KernelScope ks("rdft_t", st);
    rdft_t_kernel<KC><<<dim3(unsigned(bx), unsigned(by)), RB, smem, st>>>(g);
  }
  return launch_status("rdft_t_kernel");
}

// Block shape and grid of a product over `tubes` tubes: outputs in the fewest
// equal parts whose table fits, threads near 256 (more where the outputs of a
// part need them), as many blocks as are resident, each walking its tubes.
template <bool INV, int NP>
int launch_product_np(const DftArgs& p, int64_t tubes, size_t smem, const char* name,
                      cudaStream_t st) {
  const int nt = p.ty << p.tx_log;
  auto kernel = nt <= 256   ? dft_product_kernel<INV, NP, 256, 3>
                : nt <= 384 ? dft_product_kernel<INV, NP, 384, 2>
                            : dft_product_kernel<INV, NP, DT_MAX, 1>;
  TP_SET_SMEM(kernel, smem);
  if (nt > DT_MAX) {
    set_error("dft: %d threads a block", nt);
    return TP_EUNSUPPORTED;
  }
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, nt, smem) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  const int64_t bm = int64_t(DM) << p.tx_log;
  int64_t blocks = (tubes + bm - 1) / bm;
  const int64_t cap = std::max<int64_t>(1, int64_t(sm_count()) * per_sm / p.parts);
  if (blocks > cap) blocks = cap;
  {
    KernelScope ks(name, st);
    kernel<<<dim3(unsigned(blocks), unsigned(p.parts)), nt, smem, st>>>(p);
  }
  return launch_status("dft_product_kernel");
}

template <bool INV>
int launch_product(DftArgs& p, int64_t tubes, const char* name, cudaStream_t st) {
  const int h = p.n3 / 2 + 1;
  p.K = h;
  const size_t kp = size_t(h + DK - 1) / DK * DK;
  const int fit = std::max(1, int(TABLE_BYTES_MAX / (sizeof(float2) * kp * DN)));
  const int groups = (h + DN - 1) / DN;
  p.parts = (groups + fit - 1) / fit;
  // four groups of outputs at least (some may be past the spectrum), so that a
  // thread stages 8 samples of a K tile at most: n3 = 17, 19, 23 with three groups
  // and 11 samples, 220000 tubes, forward 28.8, 29.0, 31.7 -> 22.3, 22.7, 24.7 us,
  // inverse 21.1, 22.3, 22.5 -> 17.5, 17.8, 18.6
  p.ty = std::max(4, (groups + p.parts - 1) / p.parts);
  p.N = p.ty * DN;
  p.parts = (h + p.N - 1) / p.N;
  // 16 to 64 lanes along the tubes: small problems and many outputs take few
  p.tx_log = 4;
  while (p.tx_log < 6 && (p.ty << (p.tx_log + 1)) <= 256 &&
         tubes >= int64_t(sm_count()) * 2 * (DM << (p.tx_log + 1)))
    ++p.tx_log;
  const int nt = p.ty << p.tx_log;
  const size_t bm = size_t(DM) << p.tx_log;
  const size_t smem = kp * p.N * sizeof(float2) + 4 * DK * bm * sizeof(float) +
                      bm * (sizeof(float*) + sizeof(int64_t) + sizeof(float)) +
                      size_t(p.n3) * sizeof(float2);
  const int np = int((DK * bm + nt - 1) / nt);   // K-tile samples per thread: 32 / ty
  if (np <= 4) return launch_product_np<INV, 4>(p, tubes, smem, name, st);
  if (np <= 8) return launch_product_np<INV, 8>(p, tubes, smem, name, st);
  set_error("dft: %d samples a thread", np);
  return TP_EUNSUPPORTED;
}

}  // namespace

bool fft_supported(int64_t n3);
bool rfft_reg_supported(int64_t n3);
int launch_rfft_reg(const DftGather& g, cudaStream_t st);
int launch_irfft_reg(const float* in_re, const float* in_im, int64_t rows, int64_t in_slice,
                     int64_t n3, float* out, cudaStream_t st);
int launch_fft_fwd(const DftGather& g, cudaStream_t st);
int launch_fft_inv(const float* ire, const float* iim, int64_t rows, int64_t in_slice, int64_t n3,
                   float* out, cudaStream_t st);

// Longer tubes than this go through the mixed-radix FFT (fft.cu) when their
// length factors into primes up to 13; building with another value keeps
// shorter ones on the direct contraction.  218880 tubes, FFT against product,
// forward / inverse in us: n3 = 80 57 / 53 against 123 / 84; n3 = 225 (odd: a
// full complex transform) 183 / 247 against 657 / 419.
#ifndef TP_FFT_THRESHOLD
#define TP_FFT_THRESHOLD 16
#endif
constexpr int64_t kFftThreshold = TP_FFT_THRESHOLD;
int launch_rdft(const DftGather& g, cudaStream_t st) {
  const bool plain = g.gather_dim == 0 && !g.out_transposed && !g.out_re_lo &&
                     (g.cols == 1 || g.col_stride == g.rows) && g.out_ld == g.rows &&
                     g.out_slice == g.rows * g.cols && g.slice_stride == g.rows * g.cols &&
                     g.row_stride == 1;
  if (g.n3 < 1 || (g.n3 > 512 && !(plain && fft_supported(g.n3)))) {
    set_error("rdft: n3 = %lld: longer than 512 needs a plain (ungathered) transform and "
              "prime factors <= 13", (long long)g.n3);
    return TP_EUNSUPPORTED;
  }
  if (g.rows == 0 || g.cols == 0) return TP_OK;
  if (rfft_reg_supported(g.n3)) return launch_rfft_reg(g, st);
  if (g.n3 > kFftThreshold && fft_supported(g.n3)) return launch_fft_fwd(g, st);
  if (!g.out_transposed) {
    DftArgs p{};
    p.g = g;
    p.n3 = int(g.n3);
    return launch_product<false>(p, g.rows * g.cols, "rdft", st);
  }
  // transposed: tile width KC among {8, 12, 16} (each frequency sums its
  // samples in the same order whatever the width): autotuned, default the
  // least padding
  const auto run = [&](int c) {
    switch (c) {
      case 0: return launch_rdft_t<8>(g, st);
      case 1: return launch_rdft_t<12>(g, st);
      default: return launch_rdft_t<16>(g, st);
    }
  };
  const int kc = pick_kc(g.n3 / 2 + 1);
  const int64_t key[7] = {g.n3, size_class(g.rows), size_class(g.cols), g.gather_dim,
                          g.out_transposed, g.out_re_lo ? 1 : 0, g.out_bf16};
  int c = 0;
  const int rc = autotune_pick("rdft", key, 7, 3, kc == 8 ? 0 : kc == 12 ? 1 : 2, run, st, &c);
  return rc ? rc : run(c);
}

// The plain forward transform with every frequency's samples summed in order
// (tubes of up to 256 samples that are no power of two up to 128), for callers
// whose results hang on the rounding of its sums; else launch_rdft.
int launch_rdft_in_order(const DftGather& g, cudaStream_t st) {
  const bool pow2 = g.n3 <= 128 && (g.n3 & (g.n3 - 1)) == 0;
  if (g.n3 < 1 || g.n3 > 256 || pow2) return launch_rdft(g, st);
  if (g.rows == 0 || g.cols == 0) return TP_OK;
  DftArgs p{};
  p.g = g;
  p.n3 = int(g.n3);
  return launch_product<false>(p, g.rows * g.cols, "rdft", st);
}

int launch_irdft(const float* in_re, const float* in_im, int64_t rows, int64_t in_slice,
                 int64_t n3, float* out, cudaStream_t st) {
  if (n3 < 1 || (n3 > 512 && !fft_supported(n3))) {
    set_error("irdft: n3 = %lld: longer than 512 needs prime factors <= 13", (long long)n3);
    return TP_EUNSUPPORTED;
  }
  if (rows == 0) return TP_OK;
  if (rfft_reg_supported(n3))
    return launch_irfft_reg(in_re, in_im, rows, in_slice, n3, out, st);
  // An odd length is a full complex transform in the FFT, where many tubes leave
  // the product ahead.  FFT against product, us: n3 = 25, 39, 45 on 32768 tubes 10.4 /
  // 10.0, 12.5 / 12.4, 12.7 / 12.3, on 49152 11.2 / 9.8, 14.6 / 12.4, 14.5 / 13.7, on
  // 220000 23.6 / 18.2, 38.9 / 28.8, 41.4 / 32.3; n3 = 49, 63, 75 on 128000 25.6 / 28.1,
  // 30.8 / 26.5, 39.2 / 39.1, on 220000 43.2 / 44.3, 60.4 / 44.8, 76.1 / 64.6.
  const bool odd_product = n3 % 2 == 1 && ((n3 < 48 && rows >= 49152) || (n3 < 80 && rows >= 163840));
  if (n3 > kFftThreshold && fft_supported(n3) && !odd_product)
    return launch_fft_inv(in_re, in_im, rows, in_slice, n3, out, st);
  DftArgs p{};
  p.in_re = in_re;
  p.in_im = in_im;
  p.rows = rows;
  p.in_slice = in_slice;
  p.out = out;
  p.n3 = int(n3);
  return launch_product<true>(p, rows, "irdft", st);
}

}  // namespace tp
