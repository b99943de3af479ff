// Singular-value thresholding of slices with few singular values above the
// threshold, which is what the nuclear-norm ADMM meets in nearly all of its
// iterations (the rank of the data above tau = 1/mu, everything else well
// below: 10 of 144 in the 144 x 256 x 80 completion).  The shrunk slice
// needs only the singular triplets above tau, so instead of all q right
// singular vectors (one-sided Jacobi, q^2 / 2 rotations a sweep) each slice
// keeps a block of 32 vectors from iteration to iteration and advances it by
// subspace iteration on its Gram matrix G = W^H W:
//   Y = T_2(G) Q;  Q <- Y R^{-1},  Y^H Y = R^H R  (a quadratic Chebyshev
//   filter below the kept vectors, Zhou and Saad 2007; Cholesky QR, 32 x 32)
// and, after two of these, Rayleigh-Ritz: Y = G Q, the eigenvectors of Q^H Y
// (32 x 32 Jacobi) rotate Q and Y, lambda_j = q_j^H y_j, r_j = ||y_j - lambda_j
// q_j||, until every vector above the threshold is resolved.  What is left is
// certified, not assumed: with the vectors T above the threshold,
//   A = tau^2 I - G + sum_T lambda_j q_j q_j^H
// has a Cholesky factor only if it is positive definite, and then (Weyl) G has
// at most |T| eigenvalues above tau^2, so nothing above the threshold was
// missed.  The error of the shrunk slice that r_j leaves is at most about
// (s_j - tau) r_j / (lambda_j - tau^2) = r_j / (s_j + tau), whatever the gap.
// A slice with more than 26 values above tau, a factor that breaks down or a
// residual that stays above its bound is flagged and takes the Jacobi instead
// (svt.cu), from the V it last left there.
//
// One CTA per slice: Q and Y in shared memory, G read from L2 (packed
// two-lane FMAs, a row x 8 columns a thread), the Cholesky in place in G
// by panels of 32 columns.
// Bound by one block's share of an SM: of a slice's 1.35 M cycles the products
// with G take a third (bound by their loads, 3 from shared and 2 from global
// memory per 16 packed FMAs of a row's 8 columns), the certificate's panels a
// fifth, the 32 x 32 Jacobi a sixth, small products, sums and factors the rest.
// 41 slices of 144 x 256 (the 144 x 256 x 80 completion), one iteration: 3.5 ms
// by the warm-started Jacobi and its GEMMs -> 0.53 ms here and 0.14 ms of GEMMs.
// From 48 columns on (below, the Jacobi's slices are small and many fit an
// SM) up to 384, where Q and Y (2 x 2 x 48 KB) still fit the shared memory.
#include <algorithm>

#include "svt_top.cuh"

namespace tp {
namespace {

constexpr int L = SVT_TOP_L;          // vectors kept per slice
constexpr int LS = L + 1;             // row stride of the L x L matrices
constexpr int MAX_WARPS = 20;        // 96 registers a thread: eight loads of A in flight
constexpr int MAX_ABOVE = L - 6;      // a buffer of vectors below the threshold
constexpr int MAX_ROUNDS = 8;         // Rayleigh-Ritz rounds
// Iterations left to the Jacobi after a failed attempt (too many values above,
// a residual above its bound, a factor that breaks down): RETRY, doubled with
// every further failure in a row up to RETRY_MAX, so that a slice that the
// attempts no longer fit costs a few of them per run, not one per iteration.
// Noise-free 144 x 256 x 80, rank 10, iterations 100 to 120 (tau near the
// residuals' floor), ms an iteration: 3.9 with an attempt in each, 3.3 by the
// Jacobi alone, 3.2 with this.
constexpr int RETRY = 4, RETRY_MAX = 64;
constexpr float TOL = 3e-7f;          // r_j / (s_j + tau), relative to s_1
constexpr float TOL_MAX = 1.5e-6f;    //   accepted once it no longer falls
constexpr float ORTH_TOL = 5e-6f;     // |x_i^H x_j - delta_ij| of the vectors above
constexpr float NULL_PIVOT = 3e-6f;   // pivot of a dependent column, relative to its square

struct Tile {   // one row, eight columns
  float2 re[4], im[4];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int u = 0; u < 4; ++u) re[u] = im[u] = make_float2(0.f, 0.f);
  }
};

// t += x B[c0 .. c0+7], a row of B in shared memory
__device__ __forceinline__ void accumulate_one(Tile& t, float xr, float xi, const float* br,
                                               const float* bi) {
  const float2 pr = make_float2(xr, xr), pi = make_float2(xi, xi), ni = make_float2(-xi, -xi);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float4 b = reinterpret_cast<const float4*>(br)[h];
    const float4 d = reinterpret_cast<const float4*>(bi)[h];
    const float2 b0 = make_float2(b.x, b.y), b1 = make_float2(b.z, b.w);
    const float2 d0 = make_float2(d.x, d.y), d1 = make_float2(d.z, d.w);
    t.re[2 * h] = __ffma2_rn(pr, b0, t.re[2 * h]);
    t.re[2 * h + 1] = __ffma2_rn(pr, b1, t.re[2 * h + 1]);
    t.im[2 * h] = __ffma2_rn(pr, d0, t.im[2 * h]);
    t.im[2 * h + 1] = __ffma2_rn(pr, d1, t.im[2 * h + 1]);
    t.re[2 * h] = __ffma2_rn(ni, d0, t.re[2 * h]);
    t.re[2 * h + 1] = __ffma2_rn(ni, d1, t.re[2 * h + 1]);
    t.im[2 * h] = __ffma2_rn(pi, b0, t.im[2 * h]);
    t.im[2 * h + 1] = __ffma2_rn(pi, b1, t.im[2 * h + 1]);
  }
}

// t += sum_k A(row, k) B[k][c0 .. c0+7]: A in global memory (column-major,
// leading dimension lda), B in shared memory (row stride L).  The next eight
// values of A are loaded before the current ones are used; whole blocks of
// eight take no bounds checks and fixed offsets (with two rows of `inner` a
// warp and the Jacobi's refined reciprocal roots 0.608 -> 0.529 ms a launch for
// 41 slices of 144 columns).  (Two rows a
// thread halve the loads of B but leave too few warps: 70 against 50 thousand
// cycles for q = 144.)
__device__ __forceinline__ void accumulate(Tile& t, const float* ar, const float* ai, int lda,
                                           int K, const float* Br, const float* Bi, int c0) {
  constexpr int U = 8;
  const int blocks = K / U;
  const float *br = Br + c0, *bi = Bi + c0;
  float nr[U], ni[U];
  auto fetch = [&]() {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      nr[u] = *ar;
      ni[u] = *ai;
      ar += lda;
      ai += lda;
    }
  };
  if (blocks > 0) fetch();
  for (int b = 0; b < blocks; ++b, br += U * L, bi += U * L) {
    float xr[U], xi[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      xr[u] = nr[u];
      xi[u] = ni[u];
    }
    if (b + 1 < blocks) fetch();
#pragma unroll
    for (int u = 0; u < U; ++u) accumulate_one(t, xr[u], xi[u], br + u * L, bi + u * L);
  }
  for (int k = blocks * U; k < K; ++k, ar += lda, ai += lda, br += L, bi += L)
    accumulate_one(t, *ar, *ai, br, bi);
}

__device__ __forceinline__ float column(const float2 (&v)[4], int u) {
  return (u & 1) ? v[u >> 1].y : v[u >> 1].x;
}

struct Shared {
  float *Qr, *Qi, *Yr, *Yi;            // q x L, row-major
  float *Sr, *Si, *Zr, *Zi;            // L x L
  float *red;                          // MAX_WARPS x L
  float *lam, *scale;                  // L
  int *order;                          // L
};

// S = A^H B (L x L) of two of Q and Y: lane = column of B, a warp per column
// of A.
__device__ void inner(const Shared& s, const float* ar, const float* ai, const float* br,
                      const float* bi, int q, int warp, int lane, int nw) {
  // two rows of the result a warp, so that b is read once for both (16 warps;
  // at least that many run)
  constexpr int H = L / 2;
  if (warp >= H) return;
  float2 sr = make_float2(0.f, 0.f), si = sr;
#pragma unroll 4
  for (int k = 0; k < q; ++k) {
    const float2 xr = make_float2(ar[k * L + warp], ar[k * L + warp + H]);
    const float2 xi = make_float2(ai[k * L + warp], ai[k * L + warp + H]);
    const float yr = br[k * L + lane], yi = bi[k * L + lane];
    const float2 pr = make_float2(yr, yr), pi = make_float2(yi, yi), nr = make_float2(-yr, -yr);
    sr = __ffma2_rn(xr, pr, __ffma2_rn(xi, pi, sr));
    si = __ffma2_rn(xr, pi, __ffma2_rn(xi, nr, si));
  }
  s.Sr[warp * LS + lane] = sr.x;
  s.Si[warp * LS + lane] = si.x;
  s.Sr[(warp + H) * LS + lane] = sr.y;
  s.Si[(warp + H) * LS + lane] = si.y;
}

// dst = src M (q x L, L x L), M(b, c) at mr[b * LS + col], col = order[c] or c.
// dst may be src (a warp owns its rows).
__device__ void times_small(float* dr, float* di, const float* sr, const float* si,
                            const float* mr, const float* mi, const int* order, int q, int warp,
                            int lane, int nw) {
  const int col = order ? order[lane] : lane;
  for (int k0 = warp * 4; k0 < q; k0 += nw * 4) {
    float ar[4] = {0.f, 0.f, 0.f, 0.f}, ai[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int b = 0; b < L; ++b) {
      const float zr = mr[b * LS + col], zi = mi[b * LS + col];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int k = min(k0 + u, q - 1);
        const float yr = sr[k * L + b], yi = si[k * L + b];
        ar[u] = fmaf(yr, zr, fmaf(-yi, zi, ar[u]));
        ai[u] = fmaf(yr, zi, fmaf(yi, zr, ai[u]));
      }
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (k0 + u < q) {
        dr[(k0 + u) * L + lane] = ar[u];
        di[(k0 + u) * L + lane] = ai[u];
      }
    __syncwarp();
  }
}

// S (Hermitian, lower triangle, n <= L) = L L^H without the square roots: on
// exit S(r, c), r > c, holds the columns before scaling, S(j, j) the pivots
// d_j, and Z the inverse of the unit lower factor (rows of L^{-1} times
// sqrt(d)).  Every thread updates its entries of the trailing block and of the
// inverse; one barrier a column.  A pivot not above floor * S(j, j) is
// recorded as 0 and its column left out; returns whether there was none
// (floor 0: positive definite).
__device__ bool factor(const Shared& s, int n, float floor, int tid, int nt) {
  for (int e = tid; e < L * L; e += nt) {
    s.Zr[(e / L) * LS + e % L] = e / L == e % L ? 1.f : 0.f;
    s.Zi[(e / L) * LS + e % L] = 0.f;
  }
  if (tid < n) s.scale[tid] = s.Sr[tid * LS + tid];
  const int warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
  __syncthreads();
  bool full = true;
  for (int j = 0; j < n; ++j) {
    const float d = s.Sr[j * LS + j];
    const bool good = d > 0.f && d > floor * s.scale[j];   // the same for every thread
    if (good) {
      const float inv = 1.f / d;
      // row r > j of the trailing block (columns c > j: a(r, c) -= a(r, j)
      // conj(a(c, j)) / d) and of the inverse (c <= j: row r -= (a(r, j) / d)
      // row j): a warp per row, lane = c
      const bool trail = lane > j;
      float* const vr = trail ? s.Sr : s.Zr;
      float* const vi = trail ? s.Si : s.Zi;
      const int yo = trail ? lane * LS + j : j * LS + lane;
      const float yr = vr[yo], yi = trail ? -vi[yo] : vi[yo];
      for (int r = j + 1 + warp; r < n; r += nw) {
        if (lane > r) continue;
        const float xr = s.Sr[r * LS + j] * inv, xi = s.Si[r * LS + j] * inv;
        vr[r * LS + lane] -= xr * yr - xi * yi;
        vi[r * LS + lane] -= xr * yi + xi * yr;
      }
    } else {
      full = false;
      if (floor == 0.f) break;
    }
    __syncthreads();
    if (!good && tid == 0) s.Sr[j * LS + j] = 0.f;   // read again only after the loop
  }
  __syncthreads();
  return full;
}

// Pairs of the round-robin steps: step i pairs column a(i, j) with b(i, j),
// j < L / 2, a < b.
__device__ void fill_pairs(uchar2* pairs, int tid, int nt) {
  for (int e = tid; e < (L - 1) * (L / 2); e += nt) {
    const int step = e / (L / 2), i = e % (L / 2);
    int a = i == 0 ? L - 1 : (step + i) % (L - 1);
    int b = i == 0 ? step : (step - i + L - 1) % (L - 1);
    if (a > b) {
      const int t = a;
      a = b;
      b = t;
    }
    pairs[e] = make_uchar2((unsigned char)a, (unsigned char)b);
  }
}

// 1 / sqrt(x), the hardware's value after one Newton-Raphson step
__device__ __forceinline__ float rsqrt_refined(float x) {
  const float y = rsqrtf(x);
  return y * fmaf(-0.5f * x, y * y, 1.5f);
}

// Two-sided Jacobi of the Hermitian S: S <- Z^H S Z, Z accumulated, with its
// entries off the diagonal below 5e-8 of the largest diagonal one wherever a
// pair could hold an eigenvalue above t2 (the vectors below the threshold need
// not be resolved among themselves).  Round-robin steps of L / 2 disjoint
// pairs: one thread per pair forms the rotation; a step without one costs a
// barrier only.  Else one thread per two pairs (p <= q) applies both to their
// 2 x 2 block and its mirror, the others rotate Z, two rows a thread.
__device__ void small_jacobi(const Shared& s, float t2, int tid, int nt, const uchar2* pairs,
                             float4* rot) {
  for (int e = tid; e < L * L; e += nt) {
    s.Zr[(e / L) * LS + e % L] = e / L == e % L ? 1.f : 0.f;
    s.Zi[(e / L) * LS + e % L] = 0.f;
  }
  constexpr int H = L / 2, BLOCKS = H * (H + 1) / 2;
  __syncthreads();
  float top = 0.f;
  if (tid < H)
    for (int j = 0; j < L; ++j) top = fmaxf(top, s.Sr[j * LS + j]);
  const float small = 2.5e-15f * top * top;
  for (int sweep = 0; sweep < 12; ++sweep) {
    bool any = false;
    for (int step = 0; step < L - 1; ++step) {
      const uchar2* ps = pairs + step * H;
      bool turn = false;
      if (tid < H) {
        const int a = ps[tid].x, b = ps[tid].y;
        const float al = s.Sr[a * LS + a], be = s.Sr[b * LS + b];
        const float gr = s.Sr[a * LS + b], gi = s.Si[a * LS + b];
        const float g2 = fmaf(gr, gr, gi * gi);
        // rotation by (c, s e^{i phi}) with gamma = |gamma| e^{i phi}
        float c = 1.f, sr = 0.f, si = 0.f;
        if (g2 > small && al + be > 0.98f * t2) {
          // refined reciprocal square roots: the step's chain is half as long as
          // with the rounded roots and divisions (c and e^{i phi} are unit to
          // rounding whatever the error of t)
          const float ig = rsqrt_refined(g2), z = 0.5f * (be - al) * ig;
          const float w = fmaf(z, z, 1.f);
          const float t = __fdividef(copysignf(1.f, z), fabsf(z) + w * rsqrt_refined(w));
          c = rsqrt_refined(fmaf(t, t, 1.f));
          sr = c * t * (gr * ig);
          si = c * t * (gi * ig);
          turn = true;
        }
        rot[tid] = make_float4(c, sr, si, 0.f);
      }
      if (!__syncthreads_or(turn)) continue;
      any = true;
      for (int e = tid; e < BLOCKS + L * H / 2; e += nt) {
        if (e < BLOCKS) {
          // e -> (ip, iq), ip <= iq, rows of the triangle folded in pairs
          int ip = e / (H + 1), iq = e - ip * (H + 1);
          if (iq <= ip) {
            iq = H - 1 - iq;
            ip = H - 1 - ip;
            if (ip > iq) {
              const int t = ip;
              ip = iq;
              iq = t;
            }
          } else {
            iq -= 1;
          }
          const int a = ps[ip].x, b = ps[ip].y, c2 = ps[iq].x, d = ps[iq].y;
          const float4 R = rot[ip], T = rot[iq];
          // columns c2, d: x' = c x - conj(s) y, y' = s x + c y
          float2 m[2][2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int row = u ? b : a;
            const float2 x = make_float2(s.Sr[row * LS + c2], s.Si[row * LS + c2]);
            const float2 y = make_float2(s.Sr[row * LS + d], s.Si[row * LS + d]);
            m[u][0] = make_float2(T.x * x.x - (T.y * y.x + T.z * y.y),
                                  T.x * x.y - (T.y * y.y - T.z * y.x));
            m[u][1] = make_float2(T.x * y.x + (T.y * x.x - T.z * x.y),
                                  T.x * y.y + (T.y * x.y + T.z * x.x));
          }
          // rows a, b: the conjugate; the mirror block is the conjugate transpose
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            const int col = v ? d : c2;
            const float2 x = m[0][v], y = m[1][v];
            const float2 p = make_float2(R.x * x.x - (R.y * y.x - R.z * y.y),
                                         R.x * x.y - (R.y * y.y + R.z * y.x));
            const float2 w = make_float2(R.x * y.x + (R.y * x.x + R.z * x.y),
                                         R.x * y.y + (R.y * x.y - R.z * x.x));
            s.Sr[a * LS + col] = p.x;
            s.Si[a * LS + col] = p.y;
            s.Sr[b * LS + col] = w.x;
            s.Si[b * LS + col] = w.y;
            if (ip != iq) {
              s.Sr[col * LS + a] = p.x;
              s.Si[col * LS + a] = -p.y;
              s.Sr[col * LS + b] = w.x;
              s.Si[col * LS + b] = -w.y;
            }
          }
        } else {
          const int w = e - BLOCKS, row0 = w / H, iq = w % H;
          const int c2 = ps[iq].x, d = ps[iq].y;
          const float4 T = rot[iq];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int row = row0 + u * (L / 2);
            const float2 x = make_float2(s.Zr[row * LS + c2], s.Zi[row * LS + c2]);
            const float2 y = make_float2(s.Zr[row * LS + d], s.Zi[row * LS + d]);
            s.Zr[row * LS + c2] = T.x * x.x - (T.y * y.x + T.z * y.y);
            s.Zi[row * LS + c2] = T.x * x.y - (T.y * y.y - T.z * y.x);
            s.Zr[row * LS + d] = T.x * y.x + (T.y * x.x - T.z * x.y);
            s.Zi[row * LS + d] = T.x * y.y + (T.y * x.y + T.z * x.x);
          }
        }
      }
      __syncthreads();
    }
    if (!any) break;
  }
}

// Cholesky of A = t2 I - unit G + X X^H in place in G's lower triangle (X: q x L,
// column-major in global memory), panels of L columns; false when A is not
// positive definite.
__device__ bool certify(const Shared& s, float* gr, float* gi, int q, float unit, float t2,
                        const float* xr, const float* xi, int tid, int nt) {
  const int warp = tid >> 5, lane = tid & 31, nrw = nt >> 6;
  const int lr = lane & 15, c0 = (warp & 1) * 16 + (lane >> 4) * 8;
  for (int j0 = 0; j0 < q; j0 += L) {
    const int nb = min(L, q - j0);
    // B operands of the panel: -conj(L(j0 + c, k)) and conj(X(j0 + c, j))
    for (int e = tid; e < j0 * L; e += nt) {
      const int c = e % L, k = e / L;
      const bool in = c < nb;
      s.Yr[e] = in ? -gr[j0 + c + int64_t(q) * k] : 0.f;
      s.Yi[e] = in ? gi[j0 + c + int64_t(q) * k] : 0.f;
    }
    for (int e = tid; e < L * L; e += nt) {
      const int c = e % L, j = e / L;
      const bool in = c < nb;
      s.Zr[e] = in ? xr[j0 + c + int64_t(q) * j] : 0.f;
      s.Zi[e] = in ? -xi[j0 + c + int64_t(q) * j] : 0.f;
    }
    __syncthreads();
    for (int i0 = j0 + (warp >> 1) * 16; i0 < q; i0 += nrw * 16) {
      const int i = i0 + lr, ic = min(i, q - 1);
      Tile t;
      t.clear();
      accumulate(t, gr + ic, gi + ic, q, j0, s.Yr, s.Yi, c0);
      accumulate(t, xr + ic, xi + ic, q, L, s.Zr, s.Zi, c0);
      if (i >= q) continue;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int c = c0 + u;
        if (c >= nb) continue;
        const int64_t o = i + int64_t(q) * (j0 + c);
        gr[o] = (i == j0 + c ? t2 : 0.f) - unit * gr[o] + column(t.re, u);
        gi[o] = -unit * gi[o] + column(t.im, u);
      }
    }
    __syncthreads();
    for (int e = tid; e < L * L; e += nt) {
      const int c = e / L, r = e % L;
      const bool in = r < nb && c <= r;
      s.Sr[r * LS + c] = in ? gr[j0 + r + int64_t(q) * (j0 + c)] : 0.f;
      s.Si[r * LS + c] = in ? gi[j0 + r + int64_t(q) * (j0 + c)] : 0.f;
    }
    __syncthreads();
    if (!factor(s, nb, 0.f, tid, nt)) return false;
    // L = (unscaled columns) D^{-1/2}, inverse = D^{-1/2} (unit inverse)
    for (int e = tid; e < L * L; e += nt) {
      const int r = e / L, c = e % L;
      const float dr = r < nb ? rsqrtf(s.Sr[r * LS + r]) : 0.f;
      const float dc = c < nb ? rsqrtf(s.Sr[c * LS + c]) : 0.f;
      if (r < nb && c <= r) {
        gr[j0 + r + int64_t(q) * (j0 + c)] = s.Sr[r * LS + c] * dc;
        gi[j0 + r + int64_t(q) * (j0 + c)] = s.Si[r * LS + c] * dc;
      }
      // B operand of the solve below, conj(inverse(c, k)) at [k][c]: X L^H = P
      // gives X = P inverse^H
      s.Yr[c * L + r] = c <= r ? s.Zr[r * LS + c] * dr : 0.f;
      s.Yi[c * L + r] = c <= r ? -s.Zi[r * LS + c] * dr : 0.f;
    }
    __syncthreads();
    if (j0 + L < q) {   // rows below the block (nb == L here)
      const int lo = j0 + L;
      for (int i0 = lo + (warp >> 1) * 16; i0 < q; i0 += nrw * 16) {
        const int i = i0 + lr, ic = min(i, q - 1);
        Tile t;
        t.clear();
        accumulate(t, gr + ic + int64_t(q) * j0, gi + ic + int64_t(q) * j0, q, L, s.Yr, s.Yi, c0);
        // both warps of the pair (the column halves) have read these rows
        asm volatile("bar.sync %0, 64;" ::"r"(1 + (warp >> 1)) : "memory");
        if (i >= q) continue;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int64_t o = i + int64_t(q) * (j0 + c0 + u);
          gr[o] = column(t.re, u);
          gi[o] = column(t.im, u);
        }
      }
    }
    __syncthreads();
  }
  return true;
}

// A starting entry: the sign of a hash of its position.
__device__ __forceinline__ float start_entry(int k, int c, float scale) {
  uint32_t x = uint32_t(k) * 0x9E3779B1u + uint32_t(c) * 0x85EBCA77u + 0x165667B1u;
  x ^= x >> 15;
  x *= 0x2C1B3C6Du;
  x ^= x >> 13;
  return (x & 0x8000u) ? -scale : scale;
}

__global__ void __launch_bounds__(32 * MAX_WARPS) svt_top_kernel(SvtTopArgs g) {
  extern __shared__ __align__(16) float top_sm[];
  const int f = blockIdx.x, q = g.q;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  __shared__ float4 rot[L / 2];
  __shared__ uchar2 pairs[(L - 1) * (L / 2)];
  __shared__ int verdict, above_s;
  __shared__ float err_prev, unit_s, edge_s;
  const int attempt = g.attempt[f];
  __syncthreads();
  if (!attempt) {
    if (tid == 0) {
      const int w = g.wait[f] - 1;   // the failures in a row stay
      g.wait[f] = w;
      g.attempt[f] = (w & 0xffff) == 0;
      g.fast[f] = 0;
    }
    return;
  }
  Shared s;
  s.Qr = top_sm;
  s.Qi = s.Qr + q * L;
  s.Yr = s.Qi + q * L;
  s.Yi = s.Yr + q * L;
  s.Sr = s.Yi + q * L;
  s.Si = s.Sr + L * LS;
  s.Zr = s.Si + L * LS;
  s.Zi = s.Zr + L * LS;
  s.red = s.Zi + L * LS;
  s.lam = s.red + MAX_WARPS * L;
  s.scale = s.lam + L;
  s.order = reinterpret_cast<int*>(s.scale + L);
  float* gr = g.gr + f * g.sG;
  float* gi = g.gi + f * g.sG;
  float* xr = g.xr + int64_t(f) * q * L;   // conj(Q), row-major
  float* xi = g.xi + int64_t(f) * q * L;

  // sum over the rows of a per-entry value, lane = column: every lane of warp
  // 0 gets its column's sum
  auto column_sums = [&](auto&& value) {
    float a = 0.f;
    for (int k = warp; k < q; k += nw) a += value(k * L + lane);
    s.red[warp * L + lane] = a;
    __syncthreads();
    float t = 0.f;
    if (warp == 0)
      for (int w = 0; w < nw; ++w) t += s.red[w * L + lane];
    return t;
  };

  if (warp == 0) {   // a power of two that brings G's largest entry near 1
    float m = 0.f;
    for (int k = lane; k < q; k += 32) m = fmaxf(m, gr[k + int64_t(q) * k]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    int ex = 0;
    if (m > 0.f && isfinite(m)) frexpf(m, &ex);
    if (lane == 0) unit_s = ldexpf(1.f, max(-126, min(126, -ex)));
  }
  for (int e = tid; e < q * L; e += nt) {
    s.Qr[e] = xr[e];
    s.Qi[e] = -xi[e];
  }
  fill_pairs(pairs, tid, nt);
  __syncthreads();
  const float unit = unit_s;   // everything below is of unit G
  const float tau2 = float(fmin(double(unit) / (*g.mu * *g.mu), 1e30)), tau = sqrtf(tau2);
  bool cold;
  {   // columns lost to the null space (or never started) get a fresh start
    const float t = column_sums([&](int e) { return s.Qr[e] * s.Qr[e] + s.Qi[e] * s.Qi[e]; });
    if (warp == 0) s.scale[lane] = t;
    __syncthreads();
    const bool lost = !(s.scale[lane] > 0.f);
    if (lost)
      for (int k = warp; k < q; k += nw) {
        s.Qr[k * L + lane] = start_entry(k, lane, rsqrtf(float(q)));
        s.Qi[k * L + lane] = 0.f;
      }
    cold = __syncthreads_or(lost);
  }
  const int lr = lane & 15, c0 = (warp & 1) * 16 + (lane >> 4) * 8;
  // out = f(unit G a), a warp pair (the column halves) per 16 rows; f gets the
  // entry's index and its value
  auto times_g = [&](const float* ar, const float* ai, float* outr, float* outi, auto&& f) {
    for (int i0 = (warp >> 1) * 16; i0 < q; i0 += (nw >> 1) * 16) {
      const int i = i0 + lr, ic = min(i, q - 1);
      Tile t;
      t.clear();
      accumulate(t, gr + ic, gi + ic, q, q, ar, ai, c0);
      if (i >= q) continue;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int o = i * L + c0 + 4 * h;
        float vr[4], vi[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          vr[u] = unit * column(t.re, 4 * h + u);
          vi[u] = unit * column(t.im, 4 * h + u);
          f(o + u, vr[u], vi[u]);
        }
        *reinterpret_cast<float4*>(outr + o) = make_float4(vr[0], vr[1], vr[2], vr[3]);
        *reinterpret_cast<float4*>(outi + o) = make_float4(vi[0], vi[1], vi[2], vi[3]);
      }
    }
    __syncthreads();
  };
  const auto plain = [](int, float&, float&) {};
  // Y = unit G Q  ->  Q = orth(Y) or, with edge > 0, orth(T_2(A) Q), A mapping
  // [0, edge] to [-1, 1]: the quadratic Chebyshev polynomial grows the vectors
  // above the edge by (2 (2 x - 1)^2 - 1), x = lambda / edge, against x^2 for
  // two plain products
  auto orthonormalise = [&](float edge) {
    if (edge > 0.f) {
      const float w = 2.f / edge;
      for (int e = tid; e < q * L; e += nt) {   // A Q
        s.Yr[e] = w * s.Yr[e] - s.Qr[e];
        s.Yi[e] = w * s.Yi[e] - s.Qi[e];
      }
      __syncthreads();
      const float *yr = s.Yr, *yi = s.Yi, *qr = s.Qr, *qi = s.Qi;
      times_g(s.Yr, s.Yi, s.Qr, s.Qi, [=](int o, float& vr, float& vi) {
        vr = 2.f * (w * vr - yr[o]) - qr[o];   // 2 A (A Q) - Q
        vi = 2.f * (w * vi - yi[o]) - qi[o];
      });
      float* t = s.Qr;
      s.Qr = s.Yr;
      s.Yr = t;
      t = s.Qi;
      s.Qi = s.Yi;
      s.Yi = t;
    }
    inner(s, s.Yr, s.Yi, s.Yr, s.Yi, q, warp, lane, nw);
    __syncthreads();
    factor(s, L, NULL_PIVOT, tid, nt);
    // Q = Y L^{-H}: the matrix conj(inverse(c, b)) at (b, c), in S's place; a
    // dependent column becomes zero
    if (tid < L) {
      const float d = s.Sr[tid * LS + tid];
      s.scale[tid] = d > 0.f ? rsqrtf(d) : 0.f;
    }
    __syncthreads();
    for (int e = tid; e < L * L; e += nt) {
      const int b = e / L, c = e % L;
      const float w = b <= c ? s.scale[c] : 0.f;
      s.Sr[b * LS + c] = b <= c ? w * s.Zr[c * LS + b] : 0.f;
      s.Si[b * LS + c] = b <= c ? -w * s.Zi[c * LS + b] : 0.f;
    }
    __syncthreads();
    times_small(s.Qr, s.Qi, s.Yr, s.Yi, s.Sr, s.Si, nullptr, q, warp, lane, nw);
    __syncthreads();
  };
  // a fresh start takes single products (its columns are nearly dependent
  // after two), and so does a block whose smallest vectors would drown in the
  // rounding of the largest; the polynomial's edge is the smallest kept value
  if (tid == 0) edge_s = cold ? 0.f : g.edge[f] * unit;
  __syncthreads();
  const float edge0 = edge_s;
  for (int r = 0; r < (edge0 > 0.f ? 2 : 4); ++r) {
    times_g(s.Qr, s.Qi, s.Yr, s.Yi, plain);
    orthonormalise(edge0);
  }
  for (int round = 0;; ++round) {
    times_g(s.Qr, s.Qi, s.Yr, s.Yi, plain);
    inner(s, s.Qr, s.Qi, s.Yr, s.Yi, q, warp, lane, nw);
    __syncthreads();
    small_jacobi(s, tau2, tid, nt, pairs, rot);
    __syncthreads();
    if (warp == 0) {   // descending order
      const float t = s.Sr[lane * LS + lane];
      int rank = 0;
      for (int m = 0; m < L; ++m) {
        const float u = s.Sr[m * LS + m];
        rank += (u > t) || (u == t && m < lane);
      }
      s.order[lane] = lane;   // for values that are not numbers
      __syncwarp();
      s.order[rank & (L - 1)] = lane;
    }
    __syncthreads();
    times_small(s.Qr, s.Qi, s.Qr, s.Qi, s.Zr, s.Zi, s.order, q, warp, lane, nw);
    times_small(s.Yr, s.Yi, s.Yr, s.Yi, s.Zr, s.Zi, s.order, q, warp, lane, nw);
    __syncthreads();
    const float lsum = column_sums([&](int e) { return s.Qr[e] * s.Yr[e] + s.Qi[e] * s.Yi[e]; });
    if (warp == 0) s.lam[lane] = lsum;
    __syncthreads();
    const float lc = s.lam[lane];
    const float rsum = column_sums([&](int e) {
      const float a = s.Yr[e] - lc * s.Qr[e], b = s.Yi[e] - lc * s.Qi[e];
      return a * a + b * b;
    });
    if (warp == 0) {
      const bool up = lc > tau2;
      float err = up ? sqrtf(rsum) / (sqrtf(lc) + tau) : 0.f;
      float top = fmaxf(lc, 0.f), low = lc;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        err = fmaxf(err, __shfl_xor_sync(0xffffffffu, err, o));
        top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
        low = fminf(low, __shfl_xor_sync(0xffffffffu, low, o));
      }
      // a value that is not a number must not pass (fmaxf drops it)
      const bool sane = __all_sync(0xffffffffu, isfinite(lc) && isfinite(rsum));
      const unsigned who = __ballot_sync(0xffffffffu, up);
      const int n = __popc(who);
      const float s1 = sqrtf(top);
      if (lane == 0) {
        above_s = n;
        g.above[f] = who;
        int v = 0;   // 1 resolved, -1 give up
        if (!sane || n > MAX_ABOVE) v = -1;
        else if (err <= TOL * s1) v = 1;
        else if (round >= 1 && err <= TOL_MAX * s1 && err > 0.6f * err_prev) v = 1;
        else if (round >= MAX_ROUNDS) v = -1;
        verdict = v;
        err_prev = err;
        edge_s = low > 4e-3f * top ? low : 0.f;
        g.edge[f] = edge_s / unit;
      }
    }
    __syncthreads();
    if (verdict != 0) break;
    orthonormalise(edge_s);
  }
  for (int e = tid; e < q * L; e += nt) {   // kept whatever the verdict
    xr[e] = s.Qr[e];
    xi[e] = -s.Qi[e];
  }
  bool done = verdict > 0;
  if (done && above_s > 0) {
    // the vectors above the threshold must be orthonormal (a vector lost to
    // rounding could repeat another one)
    inner(s, s.Qr, s.Qi, s.Qr, s.Qi, q, warp, lane, nw);
    __syncthreads();
    bool off = false;
    for (int a = warp; a < L; a += nw) {
      const float re = s.Sr[a * LS + lane] - (a == lane ? 1.f : 0.f), im = s.Si[a * LS + lane];
      off |= s.lam[a] > tau2 && s.lam[lane] > tau2 && !(re * re + im * im <= ORTH_TOL * ORTH_TOL);
    }
    done = !__syncthreads_or(off);
  }
  if (done) {
    float* hr = g.hr + f * g.sG;   // scratch: sqrt(lambda_j) q_j of the vectors above
    float* hi = g.hi + f * g.sG;
    for (int e = tid; e < q * L; e += nt) {
      const int k = e % q, j = e / q;
      const float w = s.lam[j] > tau2 ? sqrtf(s.lam[j]) : 0.f;
      hr[e] = w * s.Qr[k * L + j];
      hi[e] = w * s.Qi[k * L + j];
    }
    __syncthreads();
    done = certify(s, gr, gi, q, unit, tau2 * (1.f + 1e-6f), hr, hi, tid, nt);
  }
  if (tid == 0) {
    const int failed = done ? 0 : min((g.wait[f] >> 16) + 1, 16);
    g.fast[f] = done ? 1 : 0;
    g.wait[f] = done ? 0 : failed << 16 | min(RETRY << (failed - 1), RETRY_MAX);
    g.attempt[f] = done ? 1 : 0;
  }
}

// Shrink factors c_j = max(s_j - tau, 0) / (s_j n_j^2), s_j = ||h_j|| / n_j,
// n_j = ||x_j||, of the vectors above the threshold, and the rebuild's small operand: D X^H
// (element (j, b) at j + L b) or, transposed, X D (element (b, j) at b + q j).
__global__ void __launch_bounds__(32 * L) svt_top_coef_kernel(SvtTopArgs g, const float* hr,
                                                              const float* hi, int p,
                                                              int transpose) {
  __shared__ float coef[L];
  __shared__ double nv_s[L], nh_s[L];
  const int f = blockIdx.x, q = g.q, lane = threadIdx.x & 31, j = threadIdx.x >> 5;
  if (!g.fast[f]) return;
  const float* Hr = hr + f * g.sG;
  const float* Hi = hi + f * g.sG;
  const float* xr = g.xr + int64_t(f) * q * L;
  const float* xi = g.xi + int64_t(f) * q * L;
  // sums of squares as float pairs (Dekker's two-sum with the exact FMA
  // square residual): float64 runs at 1/64 of the float32 rate
  auto add_sq = [](float2& a, float x) {
    const float p = x * x, e = fmaf(x, x, -p), t = a.x + p, bp = t - a.x;
    a.y += (a.x - (t - bp)) + (p - bp) + e;
    a.x = t;
  };
  float2 sv = make_float2(0.f, 0.f), sh = sv;
  for (int b = lane; b < q; b += 32) {
    add_sq(sv, xr[b * L + j]);
    add_sq(sv, xi[b * L + j]);
  }
  for (int a = lane; a < p; a += 32) {
    add_sq(sh, Hr[a + int64_t(p) * j]);
    add_sq(sh, Hi[a + int64_t(p) * j]);
  }
  double nv = double(sv.x) + double(sv.y), nh = double(sh.x) + double(sh.y);
  for (int o = 16; o > 0; o >>= 1) {
    nv += __shfl_xor_sync(0xffffffffu, nv, o);
    nh += __shfl_xor_sync(0xffffffffu, nh, o);
  }
  if (lane == 0) {
    nv_s[j] = nv;
    nh_s[j] = nh;
  }
  __syncthreads();
  if (threadIdx.x < L) {   // one warp's float64 divisions, not every warp's
    nv = nv_s[lane];
    nh = nh_s[lane];
    const double tau = 1.0 / *g.mu, sj = nv > 0.0 ? sqrt(nh / nv) : 0.0;
    const bool up = (g.above[f] >> lane) & 1u;
    coef[lane] = up && sj > tau ? float((sj - tau) / (sj * nv)) : 0.f;
  }
  __syncthreads();
  float* Or = g.gr + f * g.sG;
  float* Oi = g.gi + f * g.sG;
  for (int e = threadIdx.x; e < q * L; e += blockDim.x) {
    if (!transpose) {
      const float c = coef[e % L];
      Or[e] = c * xr[e];
      Oi[e] = c * xi[e];
    } else {
      const int b = e % q, k = e / q;
      const float c = coef[k];
      Or[e] = c * xr[b * L + k];
      Oi[e] = -c * xi[b * L + k];
    }
  }
}

__global__ void svt_top_init_kernel(SvtTopArgs g, int64_t h, float* vr, float* vi) {
  const int64_t n = h * g.q * L, qq = int64_t(g.q) * g.q;
  const int64_t step = int64_t(gridDim.x) * blockDim.x;
  const int64_t t0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  for (int64_t e = t0; e < n; e += step) g.xr[e] = g.xi[e] = 0.f;   // started by the kernel
  for (int64_t e = t0; e < h * qq; e += step) {
    const int64_t r = e % qq;
    vr[e] = r % (g.q + 1) == 0 ? 1.f : 0.f;
    vi[e] = 0.f;
  }
  for (int64_t e = t0; e < h; e += step) {
    g.attempt[e] = 1;
    g.fast[e] = 0;
    g.wait[e] = 0;
    g.edge[e] = 0.f;
    g.above[e] = 0;
  }
}

size_t top_smem(int q) {
  return (size_t(4) * q * L + 4 * L * LS + MAX_WARPS * L + 4 * L) * sizeof(float);
}

}  // namespace

// q from 48 (below, 32 vectors are most of the slice and the Jacobi is quick)
// to 384 (Q and Y in shared memory).
bool svt_top_applies(int64_t q) { return q >= 48 && q <= 384; }

// Grows with q also past the sizes that are taken: callers size a workspace
// for a larger tensor than they pass (the picked slices of CUR t-NN).
size_t svt_top_ws(int64_t q, size_t h) {
  if (q < 48) return 0;
  const size_t qm = size_t(q < 384 ? q : 384);
  return 2 * ws_bytes(qm * L * h, 4) + 5 * ws_bytes(h, 4);
}

int svt_top_init(const SvtTopArgs& g, int64_t h, float* vr, float* vi, cudaStream_t st) {
  int64_t blocks = (h * g.q * g.q + 255) / 256;
  if (blocks > int64_t(sm_count()) * 8) blocks = int64_t(sm_count()) * 8;
  {
    KernelScope ks("svt_top_init", st);
    svt_top_init_kernel<<<unsigned(blocks), 256, 0, st>>>(g, h, vr, vi);
  }
  return launch_status("svt_top_init");
}

int svt_top_launch(const SvtTopArgs& g, int64_t h, cudaStream_t st) {
  const size_t smem = top_smem(g.q);
  // two warps (the column halves) per 16 rows in as few passes as MAX_WARPS
  // allow, at least 16 for the small steps
  const int nrb = (g.q + 15) / 16, passes = (nrb + MAX_WARPS / 2 - 1) / (MAX_WARPS / 2);
  const int warps = std::max(2 * ((nrb + passes - 1) / passes), 16);
  TP_SET_SMEM(svt_top_kernel, smem);
  {
    KernelScope ks("svt_top", st);
    svt_top_kernel<<<unsigned(h), 32 * warps, smem, st>>>(g);
  }
  return launch_status("svt_top_kernel");
}

int svt_top_coef(const SvtTopArgs& g, int64_t h, const float* hr, const float* hi, int64_t p,
                 bool transpose, cudaStream_t st) {
  {
    KernelScope ks("svt_top_coef", st);
    svt_top_coef_kernel<<<unsigned(h), 32 * L, 0, st>>>(g, hr, hi, int(p), transpose ? 1 : 0);
  }
  return launch_status("svt_top_coef_kernel");
}

}  // namespace tp
