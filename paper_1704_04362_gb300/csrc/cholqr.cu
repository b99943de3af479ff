// orth() in float64, for tall slices and the picked slices of t-CX: CholeskyQR2 of a batch of slices (p x l,
// l <= 96, planar float32, column-major) with float64 Gram matrices, Cholesky
// factors and solves; only Y itself is rounded to float32, once a pass.
//
//   G = Y^H Y,  G = R^H R,  Y <- Y R^{-1},   twice
// (Fukaya, Nakatsukasa, Yanagisawa and Yamamoto 2014); a Cholesky breakdown is
// retried once with the diagonal shifted by 11 (p l + l (l + 1)) u ||Y||_F^2,
// followed by two plain passes (shifted CholeskyQR3).
//
// The last orthonormalisation of the randomized t-SVD decides how far Q is from
// orthonormal, and every singular value is off by as much, so it ends in float64;
// the ones before it only carry a subspace to the next product and stay with the
// float32 tree (householder.cu).  After two power iterations the last one is the
// tree too, with one pass of this on its nearly orthonormal Q ("polish"); with
// fewer every one is two passes of this (rsvd.cu).  Singular values of slices of
// 400 to 1000 rows after one power iteration: 5e-8 .. 9e-8 off with two passes, 6e-8
// .. 9e-8 with the tree and one, 8e-8 .. 1.2e-7 with the tree alone.
//
// Bound by the float64 pipe (two lanes a cycle and SM): a Gram entry is six
// operations a row, a solve six per entry of R and row.  So the Gram entries are
// spread over blocks by pairs of columns and the solves by rows, and every
// operand is converted to float64 once per block instead of once per use.  Every
// entry's sum runs over the rows (the solve's over the columns) in order, so
// the split changes no result.  33 slices of 1024 x 50: one block per slice
// 14.5 ms -> 3.2 ms.  17 slices of 256 x 64 (t-CX), one pass: 0.20 ms of solves
// (a warp per 32 rows 0.50), 0.18 of factors (a root and its divisions in every
// warp, rows of the trailing triangle by warps 0.28), 0.28 for two Gram matrices.
#include "householder.cuh"

namespace tp {
namespace {

constexpr int GRAM_THREADS = 128;   // column pairs a block
constexpr int GRAM_ROWS = 32;       // rows staged at once
constexpr int FACTOR_THREADS = 256;

// State of a slice between the launches of a pass.
struct Progress {
  int passes;    // passes left
  int shifted;   // the next pass adds the shift
  int solve;     // this pass has a factor
};

struct CholArgs {
  float *yr, *yi;          // element (r, c) of slice f at f*sY + r + p*c
  int64_t sY;
  int p, lfull;
  const int32_t* lcols;    // per-slice column counts or null
  double2* G;              // [slice][l][l], row-major: the Gram matrix, then R
  Progress* state;
  int32_t* status;
  int* weak;               // see householder.cuh
  int first;               // pass 0: every slice takes part
  int passes;              // plain passes wanted
};

// a / b from y = 1 / b rounded to nearest: two corrections by the exact remainder
// give the quotient rounded to nearest (Markstein 1990).  Five operations where
// every division by the same b took some thirty.
__device__ __forceinline__ double quotient(double a, double b, double y) {
  double q = a * y;
  q = fma(fma(-b, q, a), y, q);
  return fma(fma(-b, q, a), y, q);
}

__device__ __forceinline__ int columns_of(const CholArgs& g, int f) {
  return g.lcols ? min(max(int(g.lcols[f]), 1), g.lfull) : g.lfull;
}

// Upper triangle of G, one pair of columns a thread; the block's rows arrive in
// chunks of GRAM_ROWS as float64 in shared memory (row pitch odd, so that
// neither the writes along a column nor the reads along a row conflict).
__global__ void __launch_bounds__(GRAM_THREADS) cholqr_gram_kernel(const CholArgs g) {
  extern __shared__ __align__(16) double2 chol_sm[];
  const int f = blockIdx.y, l = columns_of(g, f), p = g.p, pitch = l | 1;
  if (!g.first && g.state[f].passes <= 0) return;
  const int npairs = l * (l + 1) / 2, e0 = int(blockIdx.x) * GRAM_THREADS;
  if (e0 >= npairs) return;
  const float* yr = g.yr + int64_t(f) * g.sY;
  const float* yi = g.yi + int64_t(f) * g.sY;
  // e -> (a, b), a <= b, row-major upper triangle
  int a = 0, rem = min(e0 + int(threadIdx.x), npairs - 1);
  while (rem >= l - a) rem -= l - a, ++a;
  const int b = a + rem;
  double sr = 0.0, si = 0.0;
  for (int r0 = 0; r0 < p; r0 += GRAM_ROWS) {
    const int nr = min(GRAM_ROWS, p - r0);
    __syncthreads();
    for (int e = threadIdx.x; e < GRAM_ROWS * l; e += GRAM_THREADS) {
      const int r = e % GRAM_ROWS, c = e / GRAM_ROWS;
      if (r >= nr) continue;
      const int64_t o = r0 + r + int64_t(p) * c;
      chol_sm[r * pitch + c] = make_double2(double(yr[o]), double(yi[o]));
    }
    __syncthreads();
    for (int r = 0; r < nr; ++r) {
      const double2 x = chol_sm[r * pitch + a], y = chol_sm[r * pitch + b];
      const double ar = x.x, ai = x.y, br = y.x, bi = y.y;
      sr += ar * br + ai * bi;   // products of float32 values: exact
      si += ar * bi - ai * br;
    }
  }
  if (e0 + int(threadIdx.x) < npairs)
    g.G[(int64_t(f) * g.lfull + a) * g.lfull + b] = make_double2(sr, si);
}

// R of every slice whose Gram matrix was formed (upper triangle of G in place),
// one block a slice; sets what the slice does next.
__global__ void __launch_bounds__(FACTOR_THREADS) cholqr_factor_kernel(const CholArgs g) {
  extern __shared__ __align__(16) double2 chol_sm[];   // l x l, row-major; then the triangle
  __shared__ int bad;
  const int f = blockIdx.x, l = columns_of(g, f), tid = threadIdx.x;
  Progress s = g.first ? Progress{g.passes, 0, 0} : g.state[f];
  if (s.passes <= 0) {
    if (tid == 0) g.state[f].solve = 0;
    return;
  }
  double2* Gf = g.G + int64_t(f) * g.lfull * g.lfull;
  for (int e = tid; e < l * l; e += FACTOR_THREADS) {
    const int a = e / l, b = e - a * l;
    if (a <= b) chol_sm[e] = Gf[a * g.lfull + b];
  }
  // entry e of the trailing triangle, counted from its last corner: (l-1-b, l-1-a),
  // e = b (b + 1) / 2 + a, a <= b, whatever its size
  uchar2* tri = reinterpret_cast<uchar2*>(chol_sm + l * l);
  for (int b = tid; b < l; b += FACTOR_THREADS)
    for (int a = 0; a <= b; ++a)
      tri[b * (b + 1) / 2 + a] = make_uchar2((unsigned char)(l - 1 - b), (unsigned char)(l - 1 - a));
  if (tid == 0) bad = 0;
  __syncthreads();
  if (s.shifted) {
    if (tid == 0) {
      double tr = 0.0;
      for (int j = 0; j < l; ++j) tr += chol_sm[j * l + j].x;
      const double sh = 11.0 * (double(g.p) * l + double(l) * (l + 1)) * 1.1102230246251565e-16 * tr;
      for (int j = 0; j < l; ++j) chol_sm[j * l + j].x += sh;
    }
    __syncthreads();
  }
  // row i of R, then its share of every entry right of and below it.  One
  // thread takes the root and its reciprocal: in every warp they would fill the
  // float64 pipe.
  __shared__ double dii, yii;
  for (int i = 0; i < l; ++i) {
    if (tid == 0) {
      const double d = chol_sm[i * l + i].x;
      if (!(d > 0.0) || !isfinite(d)) bad = 1;
      dii = sqrt(d);
      yii = 1.0 / dii;
    }
    __syncthreads();
    if (bad) break;   // the same for every thread
    for (int k = i + tid; k < l; k += FACTOR_THREADS) {
      const double2 v = chol_sm[i * l + k];
      chol_sm[i * l + k] = k == i ? make_double2(dii, 0.0)
                                  : make_double2(quotient(v.x, dii, yii), quotient(v.y, dii, yii));
    }
    __syncthreads();
    const int m = l - 1 - i;
    for (int e = tid; e < m * (m + 1) / 2; e += FACTOR_THREADS) {   // subtract conj(R_ij) R_ik
      const int j = tri[e].x, k = tri[e].y;
      const double2 x = chol_sm[i * l + j], y = chol_sm[i * l + k], v = chol_sm[j * l + k];
      const double ar = x.x, ai = x.y, br = y.x, bi = y.y;
      double sr = v.x, si = v.y;
      sr -= ar * br + ai * bi;
      si -= ar * bi - ai * br;
      chol_sm[j * l + k] = make_double2(sr, si);
    }
    __syncthreads();
  }
  __syncthreads();
  const bool ok = bad == 0;
  if (ok)
    for (int e = tid; e < l * l; e += FACTOR_THREADS) {
      const int a = e / l, b = e - a * l;
      if (a <= b) Gf[a * g.lfull + b] = chol_sm[e];
    }
  if (tid != 0) return;
  if (g.weak) {
    double lo = INFINITY, hi = 0.0;
    for (int j = 0; j < l && ok; ++j) {
      lo = fmin(lo, chol_sm[j * l + j].x);
      hi = fmax(hi, chol_sm[j * l + j].x);
    }
    if (!ok || !(lo > double(CHOLQR_WEAK) * hi)) atomicOr(g.weak, 1);
  }
  s.solve = ok;
  if (ok) {
    s.shifted = 0;
    --s.passes;
  } else if (s.shifted) {   // left as it is
    s.passes = 0;
    if (g.status) atomicOr(g.status, TP_DEV_BREAKDOWN);
  } else {
    s.shifted = 1;   // this pass again with a shift, then two plain ones
    s.passes = 3;
  }
  g.state[f] = s;
}

// Y <- Y R^{-1}: x R = y by forward substitution, x_i and then its share of
// every column right of it, so that a row's updates are independent of one
// another.  A block has RT rows, its warps' groups of RT threads take the
// columns in turn: four groups of a warp each where the rows are few (a quarter
// of the float64 pipe serves one warp).  In pass 0 the columns past the slice's
// count are set to zero.
__global__ void cholqr_solve_kernel(const CholArgs g, int RT) {
  extern __shared__ __align__(16) double2 chol_sm[];
  const int f = blockIdx.y, l = columns_of(g, f), p = g.p, T = blockDim.x, tid = threadIdx.x;
  const int row = tid % RT, group = tid / RT, groups = T / RT;
  const int r = int(blockIdx.x) * RT + row;
  float* yr = g.yr + int64_t(f) * g.sY + r;
  float* yi = g.yi + int64_t(f) * g.sY + r;
  if (g.first && r < p)
    for (int c = l + group; c < g.lfull; c += groups) yr[int64_t(p) * c] = yi[int64_t(p) * c] = 0.f;
  if (!g.state[f].solve) return;
  double2* R = chol_sm;             // l x l, row-major; on the diagonal (d, 1 / d)
  double2* x = chol_sm + l * l;     // x[i * RT + row]
  const double2* Gf = g.G + int64_t(f) * g.lfull * g.lfull;
  for (int e = tid; e < l * l; e += T) {
    const int a = e / l, b = e - a * l;
    if (a > b) continue;
    double2 v = Gf[a * g.lfull + b];
    if (a == b) v.y = 1.0 / v.x;
    R[e] = v;
  }
  for (int j = group; j < l; j += groups)
    x[j * RT + row] = r < p ? make_double2(double(yr[int64_t(p) * j]), double(yi[int64_t(p) * j]))
                            : make_double2(0.0, 0.0);
  __syncthreads();
  for (int i = 0; i < l; ++i) {
    const int turn = i % groups;
    if (group == turn) {
      const double2 s = x[i * RT + row], d = R[i * l + i];
      const float qr = float(quotient(s.x, d.x, d.y)), qi = float(quotient(s.y, d.x, d.y));
      if (r < p) {
        yr[int64_t(p) * i] = qr;
        yi[int64_t(p) * i] = qi;
      }
      x[i * RT + row] = make_double2(double(qr), double(qi));
    }
    if (groups > 1) __syncthreads();
    const double2 q = x[i * RT + row];
    const double xr = q.x, xi = q.y;
    // this group's columns right of i
#pragma unroll 4
    for (int j = i + 1 + (group - turn - 1 + groups) % groups; j < l; j += groups) {
      const double2 w = R[i * l + j], v = x[j * RT + row];
      const double ar = w.x, ai = w.y;
      double sr = v.x, si = v.y;
      sr -= xr * ar - xi * ai;
      si -= xr * ai + xi * ar;
      x[j * RT + row] = make_double2(sr, si);
    }
  }
}

size_t solve_smem(int l, int T) { return (size_t(l) * l + size_t(l) * T) * sizeof(double2); }

}  // namespace

size_t cholqr_scratch(int64_t l, int64_t batch) {
  return ws_bytes(size_t(l) * l * batch, sizeof(double2)) + ws_bytes(size_t(batch), sizeof(Progress));
}

int cholqr_launch(float* yr, float* yi, int64_t rows, int l, const int32_t* lcols, int64_t batch,
                  void* scratch, int32_t* status, cudaStream_t st, int* weak, bool polish) {
  if (l < 1 || l > HQR_MAX_L || rows < l || rows > 0x7fffffff || batch > 65535) {
    set_error("cholqr: needs l <= rows, l <= %d and at most 65535 slices", HQR_MAX_L);
    return TP_EUNSUPPORTED;
  }
  if (batch <= 0) return TP_OK;
  Arena ws;
  ws.base = static_cast<char*>(scratch);
  CholArgs g{yr, yi, rows * l, int(rows), l, lcols, nullptr, nullptr, status, weak, 1, polish ? 1 : 2};
  g.G = ws.take<double2>(size_t(l) * l * batch);
  g.state = ws.take<Progress>(size_t(batch));
  const size_t gram_smem = size_t(GRAM_ROWS) * (l | 1) * sizeof(double2);
  const size_t factor_smem = size_t(l) * l * sizeof(double2) + size_t(l) * (l + 1) / 2 * sizeof(uchar2);
  // rows a block: two blocks an SM where they fit; few rows in blocks of 32 with
  // four warps each
  int T = 128;
  while (T > 32 && (solve_smem(l, T) > size_t(100) * 1024 ||
                    (rows + T - 1) / T * batch < 2 * int64_t(sm_count())))
    T /= 2;
  const int threads = T == 32 ? 128 : T;
  TP_SET_SMEM(cholqr_gram_kernel, gram_smem);
  TP_SET_SMEM(cholqr_factor_kernel, factor_smem);
  TP_SET_SMEM(cholqr_solve_kernel, solve_smem(l, T));
  const unsigned pairs = unsigned((l * (l + 1) / 2 + GRAM_THREADS - 1) / GRAM_THREADS);
  const unsigned blocks = unsigned((rows + T - 1) / T), slices = unsigned(batch);
  // four passes at most: the breakdown, its shifted repeat and two plain ones
  for (int it = 0; it < (polish ? 1 : 4); ++it) {
    g.first = it == 0;
    {
      KernelScope ks("cholqr_gram", st);
      cholqr_gram_kernel<<<dim3(pairs, slices), GRAM_THREADS, gram_smem, st>>>(g);
    }
    {
      KernelScope ks("cholqr_factor", st);
      cholqr_factor_kernel<<<slices, FACTOR_THREADS, factor_smem, st>>>(g);
    }
    {
      KernelScope ks("cholqr_solve", st);
      cholqr_solve_kernel<<<dim3(blocks, slices), threads, solve_smem(l, T), st>>>(g, T);
    }
  }
  return launch_status("cholqr");
}

}  // namespace tp
