// One tube's transforms in a thread's registers: lengths 1 .. 16 and the powers
// of two up to 128 (the formulas stand in rfft_reg.cu).
#pragma once

#include "tp_internal.cuh"

namespace tp {
namespace {

constexpr int kTw = 128;

constexpr double series_sin(double x) {   // |x| <= pi/4
  double term = x, sum = x;
  for (int n = 1; n <= 12; ++n) {
    term *= -(x * x) / double((2 * n) * (2 * n + 1));
    sum += term;
  }
  return sum;
}
constexpr double series_cos(double x) {   // |x| <= pi/4
  double term = 1.0, sum = 1.0;
  for (int n = 1; n <= 12; ++n) {
    term *= -(x * x) / double((2 * n - 1) * (2 * n));
    sum += term;
  }
  return sum;
}

struct TwTable {
  float c[kTw];   // cos(2 pi m / 128)
  float s[kTw];   // sin(2 pi m / 128)
};

// Angle 2 pi m / 128 = q (pi/2) + b with quadrant q and b = (pi/2) r / 128;
// b above pi/4 is taken as the complement so that the series stay on [0, pi/4].
constexpr TwTable make_twiddles() {
  TwTable t{};
  const double half_pi = 1.57079632679489661923;
  for (int m = 0; m < kTw; ++m) {
    const int q = (4 * m) / kTw;
    const int r = 4 * m - q * kTw;
    double cb = 0.0, sb = 0.0;
    if (2 * r <= kTw) {
      const double b = half_pi * double(r) / double(kTw);
      cb = series_cos(b);
      sb = series_sin(b);
    } else {
      const double b = half_pi * double(kTw - r) / double(kTw);
      cb = series_sin(b);
      sb = series_cos(b);
    }
    double c = cb, s = sb;
    if (q == 1) {
      c = -sb;
      s = cb;
    } else if (q == 2) {
      c = -cb;
      s = -sb;
    } else if (q == 3) {
      c = sb;
      s = -cb;
    }
    t.c[m] = float(c);
    t.s[m] = float(s);
  }
  return t;
}

__constant__ TwTable kTwd = make_twiddles();

template <int N>
struct Pow2 {
  static constexpr bool v = N > 1 && (N & (N - 1)) == 0;
};

// (cos, sin)(2 pi m / N) for m < N, evaluated by the compiler in double on
// [0, pi/4] as above and rounded once.
template <int N>
struct SmallTable {
  float c[N], s[N];
};
template <int N>
constexpr SmallTable<N> make_small() {
  SmallTable<N> t{};
  const double two_pi = 6.28318530717958647692;
  for (int m = 0; m < N; ++m) {
    // octant of m / N: 8 m = q N + r, angle = q pi / 4 + (pi / 4) r / N
    const int q = (8 * m) / N, r = 8 * m - q * N;
    const double b = two_pi / 8.0 * (q & 1 ? double(N - r) : double(r)) / double(N);
    const double cb = series_cos(b), sb = series_sin(b);
    // odd octants measure b back from their upper end
    double c = 0.0, s = 0.0;
    switch (q) {
      case 0: c = cb; s = sb; break;
      case 1: c = sb; s = cb; break;
      case 2: c = -sb; s = cb; break;
      case 3: c = -cb; s = sb; break;
      case 4: c = -cb; s = -sb; break;
      case 5: c = -sb; s = -cb; break;
      case 6: c = sb; s = -cb; break;
      default: c = cb; s = -sb; break;
    }
    t.c[m] = float(c);
    t.s[m] = float(s);
  }
  return t;
}

template <int N>
__constant__ SmallTable<N> kSmall = make_small<N>();

__host__ __device__ constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n / 2); }

__device__ __forceinline__ constexpr int bitrev(int k, int bits) {
  int r = 0;
  for (int b = 0; b < bits; ++b) r |= ((k >> b) & 1) << (bits - 1 - b);
  return r;
}

// In-place M-point FFT (exp(-2 pi i nk / M)), natural order in, bit-reversed out.
template <int M>
__device__ __forceinline__ void fft_dif(float2 (&a)[M]) {
  constexpr int S = ilog2(M);
#pragma unroll
  for (int st = 0; st < S; ++st) {
    const int L = M >> (st + 1);   // butterfly half-span
#pragma unroll
    for (int b = 0; b < M; b += 2 * L) {
#pragma unroll
      for (int j = 0; j < L; ++j) {
        const float2 u = a[b + j], v = a[b + j + L];
        a[b + j] = make_float2(u.x + v.x, u.y + v.y);
        const float dx = u.x - v.x, dy = u.y - v.y;
        if (j == 0) {
          a[b + j + L] = make_float2(dx, dy);
        } else if (2 * j == L) {   // times exp(-i pi / 2) = -i
          a[b + j + L] = make_float2(dy, -dx);
        } else {                   // times exp(-2 pi i j / (2L)) = c - i s
          const int m = j * (kTw / (2 * L));
          const float c = kTwd.c[m], s = kTwd.s[m];
          a[b + j + L] = make_float2(fmaf(dx, c, dy * s), fmaf(dy, c, -(dx * s)));
        }
      }
    }
  }
}

// Half spectrum X_0 .. X_M of the packed tube z (destroyed); put(k, re, im).
template <int N, class Put>
__device__ __forceinline__ void forward_tube(float2 (&z)[N / 2], Put&& put) {
  constexpr int M = N / 2, B = ilog2(N / 2);
  fft_dif<M>(z);
  const float2 z0 = z[0];
  put(0, z0.x + z0.y, 0.f);
  put(M, z0.x - z0.y, 0.f);
#pragma unroll
  for (int k = 1; 2 * k <= M; ++k) {
    const float2 A = z[bitrev(k, B)], Bv = z[bitrev(M - k, B)];
    const float ex = 0.5f * (A.x + Bv.x), ey = 0.5f * (A.y - Bv.y);
    const float ox = 0.5f * (A.y + Bv.y), oy = -0.5f * (A.x - Bv.x);   // (Z_k - conj Z_{M-k}) / 2i
    const int m = k * (kTw / N);
    const float c = kTwd.c[m], s = kTwd.s[m];                            // w^k = c - i s
    const float tx = fmaf(ox, c, oy * s), ty = fmaf(oy, c, -(ox * s));
    put(k, ex + tx, ey + ty);
    if (2 * k != M) put(M - k, ex - tx, ty - ey);
  }
}

// Samples of a tube as the transforms hold them: pairs (x_{2n}, x_{2n+1}) for
// powers of two, else one by one.
template <int N, bool P2 = Pow2<N>::v>
struct Tube {
  float2 z[N / 2];
  __device__ __forceinline__ void set(int t, float v) {
    if (t & 1) z[t >> 1].y = v;
    else z[t >> 1].x = v;
  }
  __device__ __forceinline__ float get(int t) const { return (t & 1) ? z[t >> 1].y : z[t >> 1].x; }
};
template <int N>
struct Tube<N, false> {
  float x[N];
  __device__ __forceinline__ void set(int t, float v) { x[t] = v; }
  __device__ __forceinline__ float get(int t) const { return x[t]; }
};

// Half spectrum of a tube of any supported length; put(k, re, im).
template <int N, class Put>
__device__ __forceinline__ void forward_any(Tube<N>& tube, Put&& put) {
  if constexpr (Pow2<N>::v) {
    forward_tube<N>(tube.z, put);
  } else {
    constexpr int NH = (N - 1) / 2;   // folded pairs; an even N has x_{N/2} besides
    float e[NH + 1], o[NH + 1];
#pragma unroll
    for (int t = 1; t <= NH; ++t) {
      e[t] = tube.x[t] + tube.x[N - t];
      o[t] = tube.x[t] - tube.x[N - t];
    }
#pragma unroll
    for (int k = 0; k <= N / 2; ++k) {
      float re = tube.x[0], im = 0.f;
      if (N % 2 == 0) re += (k & 1) ? -tube.x[N / 2] : tube.x[N / 2];
#pragma unroll
      for (int t = 1; t <= NH; ++t) {
        const int m = k * t % N;
        re = m == 0 ? re + e[t] : fmaf(e[t], kSmall<N>.c[m], re);
        if (k != 0 && 2 * k != N) im = fmaf(-o[t], kSmall<N>.s[m], im);
      }
      put(k, re, im);
    }
  }
}

// Samples of one tube from its half spectrum X[0 .. M]: x_{2n} = z[n].x,
// x_{2n+1} = z[n].y on return (z in natural order).
template <int N>
__device__ __forceinline__ void inverse_tube(const float2 (&X)[N / 2 + 1], float2 (&z)[N / 2]) {
  constexpr int M = N / 2, B = ilog2(N / 2);
  float2 a[M];
  a[0] = make_float2(0.5f * (X[0].x + X[M].x), -0.5f * (X[0].x - X[M].x));   // conj Z_0
#pragma unroll
  for (int k = 1; 2 * k <= M; ++k) {
    const float2 P = X[k], Q = X[M - k];
    const float ex = 0.5f * (P.x + Q.x), ey = 0.5f * (P.y - Q.y);
    const float dx = P.x - Q.x, dy = P.y + Q.y;                        // X_k - conj X_{M-k}
    const int m = k * (kTw / N);
    const float c = kTwd.c[m], s = kTwd.s[m];                          // conj(w^k) = c + i s
    const float ox = 0.5f * fmaf(dx, c, -(dy * s)), oy = 0.5f * fmaf(dx, s, dy * c);
    a[k] = make_float2(ex - oy, -(ey + ox));                           // conj(E + i O)
    if (2 * k != M) a[M - k] = make_float2(ex + oy, ey - ox);          // conj(conj E + i conj O)
  }
  fft_dif<M>(a);
  constexpr float inv = 1.0f / float(M);
#pragma unroll
  for (int n = 0; n < M; ++n) {
    const float2 v = a[bitrev(n, B)];
    z[n] = make_float2(v.x * inv, -v.y * inv);
  }
}

// Samples of a tube of any supported length from its half spectrum; the
// imaginary parts of the real slices are not read.
template <int N>
__device__ __forceinline__ void inverse_any(const float2 (&X)[N / 2 + 1], Tube<N>& tube) {
  if constexpr (Pow2<N>::v) {
    inverse_tube<N>(X, tube.z);
  } else {
    constexpr int NH = (N - 1) / 2;
    constexpr float w1 = 1.0f / float(N), w2 = 2.0f / float(N);
#pragma unroll
    for (int t = 0; t <= N / 2; ++t) {
      float p = X[0].x, s = 0.f;   // x_t = w1 p + w2 s, and the odd part below
      if (N % 2 == 0) p += (t & 1) ? -X[N / 2].x : X[N / 2].x;
      float q = 0.f;
#pragma unroll
      for (int k = 1; k <= NH; ++k) {
        const int m = k * t % N;
        s = m == 0 ? s + X[k].x : fmaf(X[k].x, kSmall<N>.c[m], s);
        if (t != 0 && 2 * t != N) q = fmaf(X[k].y, kSmall<N>.s[m], q);
      }
      const float even = fmaf(w2, s, w1 * p), odd = w2 * q;
      tube.set(t, even - odd);
      if (t > 0 && 2 * t != N) tube.set(N - t, even + odd);
    }
  }
}

}  // namespace
}  // namespace tp
