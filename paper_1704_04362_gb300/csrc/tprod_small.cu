// A small FP32 t-product (Algorithm 1) of short tubes in one launch: the
// transforms of both operands, the facewise products and the inverse.
//
// A block of 256 threads owns 8 x 8 tubes of C.  K is walked in chunks of 16:
// threads 0 .. 127 load and transform the chunk's 8 x 16 tubes of A, the others
// its 16 x 8 tubes of B (registers, rfft_tube.cuh), the half spectra meet in
// shared memory (two buffers, the next chunk's samples already on their way),
// and every thread adds the chunk to up to three frequencies of one tube.  The
// sums go back through shared memory to the threads that invert them.
//
// Bound by latency: the four launches of the general path (two transforms,
// product, inverse) are 16 us on the device and 18 us of host work where the
// arithmetic is less than one.  Operand tubes are loaded and transformed once
// per 8 rows or columns of C, which only a few blocks can afford.
// 64 x 48 x 32 x 16: 13.1 -> 5.8 us on the device, 17.9 -> 4.0 us of host work a
// call.
#include "rfft_tube.cuh"

namespace tp {
namespace {

constexpr int ST = 8;       // rows and columns of a block's tile
constexpr int SK = 16;      // K chunk
constexpr int SBP = SK + 2; // pitch of B's chunk (16-byte rows, banks apart)
constexpr int STHR = 256;
static_assert(2 * ST * SK == STHR, "one operand tube a thread");

template <int N>
__global__ void __launch_bounds__(STHR)
    tprod_small_kernel(const float* __restrict__ A, const float* __restrict__ B,
                       float* __restrict__ C, int n1, int n2, int n4) {
  constexpr int H = N / 2 + 1, G = STHR / (ST * ST), HT = (H + G - 1) / G;
  __shared__ __align__(16) float2 As[2][H][SK][ST];
  __shared__ __align__(16) float2 Bs[2][H][ST][SBP];
  const int tid = threadIdx.x, half = tid / (ST * SK), u = tid % (ST * SK);
  const int i0 = int(blockIdx.x) * ST, j0 = int(blockIdx.y) * ST;
  // operand tube: A(i0 + li, k0 + lk) or B(k0 + lk, j0 + li)
  const int li = half ? u / SK : u % ST, lk = half ? u % SK : u / ST;
  const bool live = half ? j0 + li < n4 : i0 + li < n1;
  const float* from = half ? B + int64_t(n2) * (j0 + li) + lk : A + int64_t(n1) * lk + i0 + li;
  const int64_t step = half ? SK : int64_t(n1) * SK, ss = half ? int64_t(n2) * n4 : int64_t(n1) * n2;
  Tube<N> tube;
  auto fetch = [&](int k0) {
    const bool in = live && k0 + lk < n2;
    const float* p = from + (k0 / SK) * step;
#pragma unroll
    for (int t = 0; t < N; ++t) tube.set(t, in ? __ldg(p + t * ss) : 0.f);
  };
  const int i = tid % ST, j = tid / ST % ST, g = tid / (ST * ST);
  float2 acc[HT];
#pragma unroll
  for (int x = 0; x < HT; ++x) acc[x] = make_float2(0.f, 0.f);
  fetch(0);
  int buf = 0;
  for (int k0 = 0; k0 < n2; k0 += SK, buf ^= 1) {
    if (half)
      forward_any<N>(tube, [&](int f, float re, float im) { Bs[buf][f][li][lk] = make_float2(re, im); });
    else
      forward_any<N>(tube, [&](int f, float re, float im) { As[buf][f][lk][li] = make_float2(re, im); });
    __syncthreads();   // also: every thread is done with the other buffer
    if (k0 + SK < n2) fetch(k0 + SK);
#pragma unroll
    for (int x = 0; x < HT; ++x) {
      const int f = g + G * x;
      if (f >= H) continue;
#pragma unroll
      for (int k = 0; k < SK; k += 2) {   // zero tubes past K
        const float4 b = *reinterpret_cast<const float4*>(&Bs[buf][f][j][k]);
        const float2 a0 = As[buf][f][k][i], a1 = As[buf][f][k + 1][i];
        acc[x].x = fmaf(-a0.y, b.y, fmaf(a0.x, b.x, acc[x].x));
        acc[x].y = fmaf(a0.y, b.x, fmaf(a0.x, b.y, acc[x].y));
        acc[x].x = fmaf(-a1.y, b.w, fmaf(a1.x, b.z, acc[x].x));
        acc[x].y = fmaf(a1.y, b.z, fmaf(a1.x, b.w, acc[x].y));
      }
    }
  }
  // buffer `buf` was last read before the latest barrier
  float2* Cs = &As[buf][0][0][0];
#pragma unroll
  for (int x = 0; x < HT; ++x)
    if (g + G * x < H) Cs[(g + G * x) * ST * ST + tid % (ST * ST)] = acc[x];
  __syncthreads();
  if (tid < ST * ST && i0 + i < n1 && j0 + j < n4) {
    float2 X[H];
#pragma unroll
    for (int f = 0; f < H; ++f) X[f] = Cs[f * ST * ST + tid];
    inverse_any<N>(X, tube);
    float* to = C + int64_t(n1) * (j0 + j) + i0 + i;
#pragma unroll
    for (int t = 0; t < N; ++t) to[int64_t(n1) * n4 * t] = tube.get(t);
  }
}

template <int N>
int launch_small(const float* A, const float* B, float* C, int n1, int n2, int n4,
                 cudaStream_t st) {
  const dim3 grid(unsigned((n1 + ST - 1) / ST), unsigned((n4 + ST - 1) / ST));
  {
    KernelScope ks("tprod_small", st);
    tprod_small_kernel<N><<<grid, STHR, 0, st>>>(A, B, C, n1, n2, n4);
  }
  return launch_status("tprod_small_kernel");
}

}  // namespace

// The rule: tubes that a thread's registers transform, and tiles that the SMs
// take in one or two rounds; beyond, the repeated transforms cost more than
// three launches.  General path against this, n3 = 16, in us: 64 tiles, K = 128
// 20.1 / 12.3, K = 512 65.6 / 43.9; 256 tiles, K = 128 21.3 / 16.8, K = 512
// 66.6 / 60.3; 625 tiles, K = 128 27.8 / 37.9.  Beyond K = 4096 the few blocks'
// chain of chunks is not measured.
bool tprod_small_applies(int64_t n1, int64_t n2, int64_t n4, int64_t n3) {
  return n3 <= 16 && n2 <= 4096 && n1 <= 4096 && n4 <= 4096 &&
         ((n1 + ST - 1) / ST) * ((n4 + ST - 1) / ST) <= 256;
}

int launch_tprod_small(const float* A, const float* B, float* C, int64_t n1, int64_t n2,
                       int64_t n4, int64_t n3, cudaStream_t st) {
  const int a = int(n1), k = int(n2), b = int(n4);
  switch (n3) {
    case 1: return launch_small<1>(A, B, C, a, k, b, st);
    case 2: return launch_small<2>(A, B, C, a, k, b, st);
    case 3: return launch_small<3>(A, B, C, a, k, b, st);
    case 4: return launch_small<4>(A, B, C, a, k, b, st);
    case 5: return launch_small<5>(A, B, C, a, k, b, st);
    case 6: return launch_small<6>(A, B, C, a, k, b, st);
    case 7: return launch_small<7>(A, B, C, a, k, b, st);
    case 8: return launch_small<8>(A, B, C, a, k, b, st);
    case 9: return launch_small<9>(A, B, C, a, k, b, st);
    case 10: return launch_small<10>(A, B, C, a, k, b, st);
    case 11: return launch_small<11>(A, B, C, a, k, b, st);
    case 12: return launch_small<12>(A, B, C, a, k, b, st);
    case 13: return launch_small<13>(A, B, C, a, k, b, st);
    case 14: return launch_small<14>(A, B, C, a, k, b, st);
    case 15: return launch_small<15>(A, B, C, a, k, b, st);
    default: return launch_small<16>(A, B, C, a, k, b, st);
  }
}

}  // namespace tp
