// Mode-3 transforms (Section 2 "Operators", fft/ifft along the third
// dimension) of tubes whose length is a product of the primes 2 .. 13, by a
// mixed-radix FFT with the butterflies in registers and one shared buffer;
// lengths up to 16 and 32, 64, 128 stay with rfft_reg.cu.
//
// Every tube is transformed on its own (packing two into one complex sequence
// would halve an odd length's work, but the smaller tube would inherit the
// larger one's rounding, and its infinities).  Even N: z_n = x_{2n} + i x_{2n+1},
// M = N / 2, Z = FFT(z), and
//   X_k = (Z_k + conj(Z_{M-k})) / 2 - i w_N^k (Z_k - conj(Z_{M-k})) / 2;
// odd N: M = N, z = x.  The FFT decimates in frequency, in place:
// M = R_1 R_2 ... R_s (R <= 16, the fewest stages, then the smallest largest
// radix), stage i cuts its sub-transforms of length m into R_i of length
// L = m / R_i,
//   y_q(j) = w_m^{j q} sum_r x(j + r L) w_R^{r q},  stored at j + q L,
// so each butterfly reads and writes the same places and a stage costs one
// barrier.  Frequency k = q_1 + R_1 (q_2 + R_2 (...)) ends at place
// q_1 M/R_1 + q_2 M/(R_1 R_2) + ..., looked up in a 16-bit table.  The first
// stage of the forward transform reads the tubes from global memory into its
// registers and the last stage of the inverse stores the samples from its
// registers, so a sequence passes through shared memory s times.  The inverse
// rebuilds Z and runs the forward FFT on its conjugate.
//
// A block owns P neighbouring tubes (P M about 16 a thread), P innermost in shared memory: consecutive threads take consecutive
// tubes of the same butterfly, so global accesses are runs of 4P bytes and
// shared ones are free of conflicts from P = 16 on (below that an odd radix
// goes last).  The transposed form (picked-slice index
// contiguous, the tensor-core product's operand layout) owns tiles of rows x 8
// columns instead.
// Bound by the latency of a block's phases (load, stages, store) at 32 warps an
// SM: 40 to 45% of the copy bandwidth at N = 168, 33% at N = 2000.
// 16384 tubes of 2000: two tubes to a sequence, radices up to 5, out of place in
// two buffers 0.34 ms forward and 0.33 inverse -> 0.117 and 0.126 ms.  218880
// tubes of 168 by products with the transform matrix: 0.317 and 0.227 ms ->
// 0.099 and 0.100 ms.
#include <algorithm>
#include <type_traits>

#include "dft_common.cuh"

namespace tp {
namespace {
using namespace dftc;

// Threads of a block (NT): 256 with P M about 4096 and four blocks per SM, so
// that one block's loads overlap the others' stages; 512 and 8192 (two blocks)
// where 4096 would leave fewer than 8 tubes, less than a sector.
constexpr int FFT_NT = 256, FFT_NT_LONG = 512, FFT_M_LONG = 512;
constexpr int FFT_PER_THREAD = 16;   // P M aimed at, per thread
constexpr int FFT_LGP_MAX = 8;       // P divides the threads
constexpr int FFT_RMAX = 16;
constexpr int FFT_STAGES = 16;
constexpr int FFT_TCOLS = 8;         // columns of a transposed tile

struct FftPlan {
  int n3, n, s, lgP;                 // tube length N, transform length M, stages, log2 P
  int radix[FFT_STAGES];
  int sub[FFT_STAGES];               // L of each stage
  unsigned magic[FFT_STAGES];        // floor(2^32 / L) + 1: i / L for i, L < 2^16
  int step[FFT_STAGES];              // w_m = w_N^step
};

// cos and sin of 2 pi m / R by their Taylor series in float64, at compile time.
template <int R>
struct Roots {
  float c[R], s[R];
};
template <int R>
constexpr Roots<R> make_roots() {
  Roots<R> t{};
  for (int m = 0; m < R; ++m) {
    // reduce to [-1/8, 1/8] of a turn around the nearest quarter
    const int quarter = (8 * m + R) / (2 * R);
    const double x = 2.0 * 3.14159265358979323846 * (double(m) / R - 0.25 * quarter);
    double c = 1.0, s = x, tc = 1.0, ts = x;
    for (int i = 1; i < 12; ++i) {
      tc *= -x * x / ((2 * i - 1) * (2 * i));
      ts *= -x * x / ((2 * i) * (2 * i + 1));
      c += tc;
      s += ts;
    }
    const int q = quarter & 3;
    t.c[m] = float(q == 0 ? c : q == 1 ? -s : q == 2 ? -c : s);
    t.s[m] = float(q == 0 ? s : q == 1 ? c : q == 2 ? -s : -c);
  }
  return t;
}
template <int R>
__constant__ Roots<R> kRoots = make_roots<R>();

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -(a.y * b.y)), fmaf(a.x, b.y, a.y * b.x));
}

__host__ __device__ constexpr int first_factor(int r) {
  if (r % 4 == 0 && r > 4) return r == 8 ? 2 : 4;
  for (int f : {2, 3, 5, 7})
    if (r % f == 0 && r > f) return f;
  return r;
}

// x <- its R-point DFT (exp(-2 pi i r q / R)), natural order.
template <int R>
__device__ __forceinline__ void dft(float2 (&x)[R]) {
  constexpr int A = first_factor(R);
  if constexpr (R == 2) {
    const float2 a = x[0], b = x[1];
    x[0] = make_float2(a.x + b.x, a.y + b.y);
    x[1] = make_float2(a.x - b.x, a.y - b.y);
  } else if constexpr (R == 4) {
    const float2 a = make_float2(x[0].x + x[2].x, x[0].y + x[2].y);
    const float2 b = make_float2(x[0].x - x[2].x, x[0].y - x[2].y);
    const float2 c = make_float2(x[1].x + x[3].x, x[1].y + x[3].y);
    const float2 d = make_float2(x[1].x - x[3].x, x[1].y - x[3].y);   // times -i below
    x[0] = make_float2(a.x + c.x, a.y + c.y);
    x[2] = make_float2(a.x - c.x, a.y - c.y);
    x[1] = make_float2(b.x + d.y, b.y - d.x);
    x[3] = make_float2(b.x - d.y, b.y + d.x);
  } else if constexpr (A == R) {   // odd prime: sums and differences of r and R - r
    constexpr int H = (R - 1) / 2;
    const float2 x0 = x[0];
    float2 t[H], d[H];
#pragma unroll
    for (int r = 1; r <= H; ++r) {
      t[r - 1] = make_float2(x[r].x + x[R - r].x, x[r].y + x[R - r].y);
      d[r - 1] = make_float2(x[r].x - x[R - r].x, x[r].y - x[R - r].y);
    }
#pragma unroll
    for (int r = 0; r < H; ++r) x[0] = make_float2(x[0].x + t[r].x, x[0].y + t[r].y);
#pragma unroll
    for (int q = 1; q <= H; ++q) {
      float2 m = x0, n = make_float2(0.f, 0.f);
#pragma unroll
      for (int r = 1; r <= H; ++r) {
        const int e = q * r % R;
        m.x = fmaf(kRoots<R>.c[e], t[r - 1].x, m.x);
        m.y = fmaf(kRoots<R>.c[e], t[r - 1].y, m.y);
        n.x = fmaf(kRoots<R>.s[e], d[r - 1].x, n.x);
        n.y = fmaf(kRoots<R>.s[e], d[r - 1].y, n.y);
      }
      x[q] = make_float2(m.x + n.y, m.y - n.x);        // m - i n
      x[R - q] = make_float2(m.x - n.y, m.y + n.x);    // m + i n
    }
  } else {   // r = B a + b, q = qa + A qb
    constexpr int B = R / A;
    float2 y[R];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      float2 v[A];
#pragma unroll
      for (int a = 0; a < A; ++a) v[a] = x[B * a + b];
      dft<A>(v);
#pragma unroll
      for (int a = 0; a < A; ++a)
        y[B * a + b] =
            a * b == 0 ? v[a] : cmul(v[a], make_float2(kRoots<R>.c[a * b], -kRoots<R>.s[a * b]));
    }
#pragma unroll
    for (int a = 0; a < A; ++a) {
      float2 v[B];
#pragma unroll
      for (int b = 0; b < B; ++b) v[b] = y[B * a + b];
      dft<B>(v);
#pragma unroll
      for (int b = 0; b < B; ++b) x[a + A * b] = v[b];
    }
  }
}

// exp(-2 pi i m / N) for m < N, by float sincospi (off the float64 pipe), and
// the place of frequency k (or, INVERSE, the frequency at place p).
template <int NT>
__device__ __forceinline__ void build_tables(const FftPlan& plan, float2* tw, uint16_t* place,
                                             bool inverse) {
  for (int m = threadIdx.x; m < plan.n3; m += NT) {
    float s, c;
    sincospif(-float(2 * m) / float(plan.n3), &s, &c);
    tw[m] = make_float2(c, s);
  }
  for (int p = threadIdx.x; p < plan.n; p += NT) {
    int rest = p, k = 0, mul = 1;
    for (int i = 0; i < plan.s; ++i) {
      const int q = rest / plan.sub[i];
      rest -= q * plan.sub[i];
      k += q * mul;
      mul *= plan.radix[i];
    }
    if (inverse) place[p] = uint16_t(k);
    else place[k] = uint16_t(p);
  }
}

// Butterfly i of stage st: its first place and the sub-transform offset j.
__device__ __forceinline__ int butterfly(const FftPlan& plan, int st, int i, int& j) {
  const int L = plan.sub[st];
  const int b = L == 1 ? i : int(__umulhi(unsigned(i), plan.magic[st]));
  j = i - b * L;
  return b * L * plan.radix[st] + j;
}

// The q-th outputs' twiddles w_m^{j q}, and the outputs in place.
template <int R>
__device__ __forceinline__ void put_stage(const FftPlan& plan, int st, const float2* tw, float2* at,
                                          int j, float2 (&x)[R]) {
  const int stride = plan.sub[st] << plan.lgP, w = j * plan.step[st];
#pragma unroll
  for (int q = 0; q < R; ++q) at[q * stride] = q == 0 ? x[0] : cmul(x[q], tw[q * w]);
}

// A stage within shared memory.
template <int NT, int R>
__device__ __forceinline__ void inner_stage(const FftPlan& plan, int st, const float2* tw,
                                            float2* buf) {
  const int items = (plan.n / R) << plan.lgP, sq = threadIdx.x & ((1 << plan.lgP) - 1);
  const int stride = plan.sub[st] << plan.lgP;
  for (int e = threadIdx.x; e < items; e += NT) {
    int j;
    float2* at = buf + (butterfly(plan, st, e >> plan.lgP, j) << plan.lgP) + sq;
    float2 x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = at[r * stride];
    dft<R>(x);
    put_stage<R>(plan, st, tw, at, j, x);
  }
}

template <class F>
__device__ __forceinline__ void with_radix(int R, F&& f) {
  switch (R) {
#define TP_FFT_CASE(r) \
  case r:              \
    f(std::integral_constant<int, r>());  \
    break;
    TP_FFT_CASE(2)
    TP_FFT_CASE(3)
    TP_FFT_CASE(4)
    TP_FFT_CASE(5)
    TP_FFT_CASE(6)
    TP_FFT_CASE(7)
    TP_FFT_CASE(8)
    TP_FFT_CASE(9)
    TP_FFT_CASE(10)
    TP_FFT_CASE(11)
    TP_FFT_CASE(12)
    TP_FFT_CASE(13)
    TP_FFT_CASE(14)
    TP_FFT_CASE(15)
    TP_FFT_CASE(16)
#undef TP_FFT_CASE
  }
}

// Stages from st on up to (not including) the one that ends at `last`.
template <int NT>
__device__ __forceinline__ void inner_stages(const FftPlan& plan, int st, int last,
                                             const float2* tw, float2* buf) {
  for (; st < last; ++st) {
    with_radix(plan.radix[st], [&](auto R) { inner_stage<NT, R.value>(plan, st, tw, buf); });
    __syncthreads();
  }
}

int64_t fft_points(int64_t n3) { return n3 % 2 == 0 ? n3 / 2 : n3; }
size_t fft_smem(int64_t n3, int lgP) {
  const size_t m = size_t(fft_points(n3));
  return (size_t(n3) + (m << lgP)) * sizeof(float2) + m * sizeof(uint16_t);
}

// Forward: the tubes of a gather to their half spectra.
template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT)
    fft_fwd_kernel(const __grid_constant__ DftGather g, const __grid_constant__ FftPlan plan) {
  extern __shared__ __align__(16) float2 fsm[];
  const int N = plan.n3, M = plan.n, lgP = plan.lgP, P = 1 << lgP;
  const bool even = M != N;
  float2* tw = fsm;
  float2* buf = fsm + N;
  uint16_t* place = reinterpret_cast<uint16_t*>(buf + (size_t(M) << lgP));
  build_tables<NT>(plan, tw, place, false);
  __syncthreads();
  const Extent ex = extent_of(g);
  const int sq = threadIdx.x & (P - 1);
  // tube s of a group: linear over the tensor, rows fastest, or (transposed) in
  // tiles of trows x tcols
  const int tcols = g.out_transposed ? min(FFT_TCOLS, P) : 1, trows = P / tcols;
  const int64_t total = ex.rows_pad * ex.cols_pad;
  const int64_t rtiles = (ex.rows_pad + trows - 1) / trows;
  const int64_t groups = g.out_transposed ? rtiles * ((ex.cols_pad + tcols - 1) / tcols)
                                          : (total + P - 1) / P;
  // the thread's tube when it stores: transposed, consecutive threads take
  // consecutive columns
  const int so = g.out_transposed ? (sq % tcols) * trows + sq / tcols : sq;
  auto tube = [&](int64_t grp, int s, int64_t& r, int64_t& c) {
    if (g.out_transposed) {
      const int64_t tc = grp / rtiles;
      r = (grp - tc * rtiles) * trows + s % trows;
      c = tc * tcols + s / trows;
      return r < ex.rows_pad && c < ex.cols_pad;
    }
    const int64_t e = grp * P + s;
    c = e / ex.rows_pad;
    r = e - c * ex.rows_pad;
    return e < total;
  };
  for (int64_t grp = blockIdx.x; grp < groups; grp += gridDim.x) {
    int64_t r, c;
    {
      const float* src = nullptr;
      float scale = 0.f;
      if (tube(grp, sq, r, c)) src = tube_ptr(g, ex, r, c, scale);
      const int64_t ss = g.slice_stride;
      with_radix(plan.radix[0], [&](auto Rc) {
        constexpr int R = Rc.value;
        const int L = plan.sub[0], items = L << lgP;
        const int64_t step = (even ? 2 * L : L) * ss;
        for (int e = threadIdx.x; e < items; e += NT) {
          const int j = e >> lgP;
          float2 x[R];
          const float* from = src + (even ? 2 * j : j) * ss;
#pragma unroll
          for (int q = 0; q < R; ++q, from += step) {
            x[q].x = src ? __ldg(from) : 0.f;
            x[q].y = src && even ? __ldg(from + ss) : 0.f;
          }
          if (g.scale) {
#pragma unroll
            for (int q = 0; q < R; ++q) x[q] = make_float2(scale * x[q].x, scale * x[q].y);
          }
          dft<R>(x);
          put_stage<R>(plan, 0, tw, buf + (j << lgP) + sq, j, x);
        }
      });
      __syncthreads();
    }
    inner_stages<NT>(plan, 1, plan.s, tw, buf);
    if (tube(grp, so, r, c)) {
      const int64_t o = g.out_transposed ? c + g.out_ld * r : r + g.out_ld * c;
      auto put = [&](int k, float re, float im) {
        const int64_t at = int64_t(k) * g.out_slice + o;
        if (g.out_re_lo) {
          put_split(g.out_re, g.out_re_lo, g.out_bf16 != 0, at, re);
          put_split(g.out_im, g.out_im_lo, g.out_bf16 != 0, at, im);
        } else {
          g.out_re[at] = re;
          g.out_im[at] = im;
        }
      };
      const int last = M / 2;   // even N: k and M - k; odd N: the half spectrum
      for (int e = threadIdx.x; e < (last + 1) << lgP; e += NT) {
        const int k = e >> lgP;
        const float2 z = buf[(int(place[k]) << lgP) + so];
        if (!even) {
          put(k, z.x, k == 0 ? 0.f : z.y);
        } else if (k == 0) {
          put(0, z.x + z.y, 0.f);
          put(M, z.x - z.y, 0.f);
        } else {
          const float2 w = buf[(int(place[M - k]) << lgP) + so], t = tw[k];
          // E = (Z_k + conj Z_{M-k}) / 2, O = -i (Z_k - conj Z_{M-k}) / 2
          const float ex_ = 0.5f * (z.x + w.x), ey = 0.5f * (z.y - w.y);
          const float2 od = cmul(t, make_float2(0.5f * (z.y + w.y), -0.5f * (z.x - w.x)));
          put(k, ex_ + od.x, ey + od.y);                    // E + w^k O
          if (2 * k != M) put(M - k, ex_ - od.x, od.y - ey);   // conj(E - w^k O)
        }
      }
    }
    __syncthreads();
  }
}

// Inverse: half spectra in{re,im}[k*in_slice + r] to real tubes
// out[r + rows*t] (imaginary parts of the k = 0 and k = n3/2 slices ignored).
template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT)
    fft_inv_kernel(const float* __restrict__ ire, const float* __restrict__ iim, int64_t rows,
                   int64_t in_slice, const __grid_constant__ FftPlan plan,
                   float* __restrict__ out) {
  extern __shared__ __align__(16) float2 fsm[];
  const int N = plan.n3, M = plan.n, lgP = plan.lgP, P = 1 << lgP;
  const bool even = M != N;
  float2* tw = fsm;
  float2* buf = fsm + N;
  uint16_t* freq = reinterpret_cast<uint16_t*>(buf + (size_t(M) << lgP));
  build_tables<NT>(plan, tw, freq, true);
  __syncthreads();
  const int sq = threadIdx.x & (P - 1);
  const float inv = 1.0f / float(M);
  for (int64_t r0 = int64_t(blockIdx.x) * P; r0 < rows; r0 += int64_t(gridDim.x) * P) {
    const int64_t r = r0 + sq;
    const bool in = r < rows;
    // conj(Z) from the half spectrum; even N: Z_k = E + i O, E = (X_k +
    // conj X_{M-k}) / 2, O = w_N^{-k} (X_k - conj X_{M-k}) / 2
    auto get = [&](int k) {
      const int64_t o = int64_t(k) * in_slice + r;
      return make_float2(in ? __ldg(ire + o) : 0.f,
                         in && k != 0 && 2 * k != N ? __ldg(iim + o) : 0.f);
    };
#pragma unroll 4
    for (int e = threadIdx.x; e < (M / 2 + 1) << lgP; e += NT) {
      const int k = e >> lgP;
      const float2 x = get(k);
      float2* lo = buf + (k << lgP) + sq;
      float2* hi = buf + ((M - k) << lgP) + sq;
      if (!even) {
        *lo = make_float2(x.x, -x.y);
        if (k > 0) *hi = x;
      } else {
        const float2 y = get(M - k);
        if (k == 0) {
          *lo = make_float2(0.5f * (x.x + y.x), -0.5f * (x.x - y.x));
        } else {
          const float ex = 0.5f * (x.x + y.x), ey = 0.5f * (x.y - y.y);
          const float2 t = tw[k];
          const float2 od = cmul(make_float2(t.x, -t.y),
                                 make_float2(0.5f * (x.x - y.x), 0.5f * (x.y + y.y)));
          *lo = make_float2(ex - od.y, -(ey + od.x));
          if (2 * k != M) *hi = make_float2(ex + od.y, ey - od.x);
        }
      }
    }
    __syncthreads();
    inner_stages<NT>(plan, 0, plan.s - 1, tw, buf);
    // z = conj(FFT(conj Z)) / M
    with_radix(plan.radix[plan.s - 1], [&](auto Rc) {
      constexpr int R = Rc.value;
      const int items = (M / R) << lgP;
      const int64_t step = (M / R) * (even ? 2 * rows : rows);
      for (int e = threadIdx.x; e < items; e += NT) {
        const int b = e >> lgP;
        const float2* at = buf + ((b * R) << lgP) + sq;
        float2 x[R];
#pragma unroll
        for (int q = 0; q < R; ++q) x[q] = at[q << lgP];
        dft<R>(x);
        if (!in) continue;
        float* to = out + r + rows * (even ? 2 * int(freq[b * R]) : int(freq[b * R]));
#pragma unroll
        for (int q = 0; q < R; ++q, to += step) {
          to[0] = x[q].x * inv;
          if (even) to[rows] = -x[q].y * inv;
        }
      }
    });
    __syncthreads();
  }
}

// The factorisation of m into radices up to `top` in non-increasing order with
// the fewest stages; false if there is none.
bool fewest(int m, int top, int depth, const int* cur, FftPlan* best, int* best_s) {
  if (m == 1) {
    // fewer stages, then the smaller largest radix
    if (*best_s == 0 || depth < *best_s || (depth == *best_s && cur[0] < best->radix[0])) {
      for (int i = 0; i < depth; ++i) best->radix[i] = cur[i];
      *best_s = depth;
    }
    return true;
  }
  if (depth == FFT_STAGES || (*best_s && depth + 1 > *best_s)) return false;
  int next[FFT_STAGES];
  for (int i = 0; i < depth; ++i) next[i] = cur[i];
  bool any = false;
  for (int r = top; r >= 2; --r) {
    if (m % r) continue;
    next[depth] = r;
    any |= fewest(m / r, r, depth + 1, next, best, best_s);
  }
  return any;
}

// Lengths beyond this were never taken: three arrays of N complex values
// within 200 KB.
constexpr int64_t FFT_N_MAX = 200 * 1024 / (3 * sizeof(float2));

int fft_threads(int64_t m) { return m > FFT_M_LONG ? FFT_NT_LONG : FFT_NT; }

bool make_plan(int64_t n3, int64_t tubes, FftPlan* p) {
  if (n3 < 2 || n3 > FFT_N_MAX) return false;
  p->n3 = int(n3);
  p->n = int(fft_points(n3));
  p->s = 0;
  const int none[1] = {0};
  if (!fewest(p->n, FFT_RMAX, 0, none, p, &p->s) || p->s == 0) return false;
  // an odd radix last: its sub-transforms start in different banks
  for (int i = p->s - 1; i >= 0; --i) {
    if (p->radix[i] % 2 == 0) continue;
    const int odd = p->radix[i];
    for (int u = i; u + 1 < p->s; ++u) p->radix[u] = p->radix[u + 1];
    p->radix[p->s - 1] = odd;
    break;
  }
  int m = p->n;
  for (int i = 0; i < p->s; ++i) {
    p->step[i] = p->n3 / m;
    m /= p->radix[i];
    p->sub[i] = m;
    p->magic[i] = unsigned((uint64_t(1) << 32) / unsigned(m)) + 1;
  }
  // tubes per block; fewer (eight at least: whole sectors) where the blocks
  // would not fill the chip
  int lg = FFT_LGP_MAX;
  while (lg > 0 && (int64_t(p->n) << lg) > FFT_PER_THREAD * fft_threads(p->n)) --lg;
  while (lg > 3 && (tubes >> lg) < 2 * int64_t(sm_count())) --lg;
  p->lgP = lg;
  return true;
}

unsigned fft_grid(int64_t groups, size_t smem, int threads) {
  const int64_t per_sm = std::min<int64_t>(1024 / threads, 227 * 1024 / int64_t(smem + 1024));
  const int64_t cap = int64_t(sm_count()) * std::max<int64_t>(1, per_sm);
  return unsigned(std::max<int64_t>(1, std::min(groups, cap)));
}

int bad_length(int64_t n3) {
  set_error("fft: n3 = %lld is not a product of radices 2,3,5,7,11,13 that fits in shared memory",
            (long long)n3);
  return TP_EUNSUPPORTED;
}

}  // namespace

bool fft_supported(int64_t n3) {
  if (n3 < 2 || n3 > FFT_N_MAX) return false;
  for (int r : {2, 3, 5, 7, 11, 13})
    while (n3 % r == 0) n3 /= r;
  return n3 == 1;
}

int launch_fft_fwd(const DftGather& g, cudaStream_t st) {
  FftPlan plan;
  if (!make_plan(g.n3, g.rows * g.cols, &plan)) return bad_length(g.n3);
  if (g.rows == 0 || g.cols == 0) return TP_OK;
  const size_t smem = fft_smem(g.n3, plan.lgP);
  const int64_t P = int64_t(1) << plan.lgP;
  const int64_t tcols = std::min<int64_t>(FFT_TCOLS, P), trows = P / tcols;
  const int64_t groups = g.out_transposed
                             ? ((g.rows + trows - 1) / trows) * ((g.cols + tcols - 1) / tcols)
                             : (g.rows * g.cols + P - 1) / P;
  const int nt = fft_threads(plan.n);
  auto kernel = nt == FFT_NT ? fft_fwd_kernel<FFT_NT> : fft_fwd_kernel<FFT_NT_LONG>;
  TP_SET_SMEM(kernel, smem);
  {
    KernelScope ks("fft_fwd", st);
    kernel<<<fft_grid(groups, smem, nt), nt, smem, st>>>(g, plan);
  }
  return launch_status("fft_fwd_kernel");
}

int launch_fft_inv(const float* ire, const float* iim, int64_t rows, int64_t in_slice, int64_t n3,
                   float* out, cudaStream_t st) {
  FftPlan plan;
  if (!make_plan(n3, rows, &plan)) return bad_length(n3);
  if (rows == 0) return TP_OK;
  const size_t smem = fft_smem(n3, plan.lgP);
  const int64_t P = int64_t(1) << plan.lgP;
  const int nt = fft_threads(plan.n);
  auto kernel = nt == FFT_NT ? fft_inv_kernel<FFT_NT> : fft_inv_kernel<FFT_NT_LONG>;
  TP_SET_SMEM(kernel, smem);
  {
    KernelScope ks("fft_inv", st);
    kernel<<<fft_grid((rows + P - 1) / P, smem, nt), nt, smem, st>>>(ire, iim, rows, in_slice, plan,
                                                                     out);
  }
  return launch_status("fft_inv_kernel");
}

}  // namespace tp
