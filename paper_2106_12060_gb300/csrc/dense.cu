// Small dense FP64 linear algebra for the preconditioner (Sec. 3): the Gram of
// the sketch, its Cholesky factor R (R^T R = (S Z)^T (S Z) + lambda I, the R
// of the QR of [S Z; sqrt(lambda) I]), R^{-1}, and products of d x d factors
// with d x c blocks (the M^{-1} = R^{-1} R^{-T} applications of Table 1).
//
// GB300 executes FP64 at ~1/60 of its FP32 rate, so these kernels spread the
// O(s d^2) and O(d^3) work over many CTAs (split-K Gram, blocked right-looking
// Cholesky, one warp per column of R^{-1}).
#include <mutex>
#include <string>

#include "plan.h"
#include "small_dense.cuh"

namespace gbcca {

// ------------------------------------------------------------------- Gram
// C (d1 x d2) = A^T B (+ diag_add on the diagonal), A: m x d1, B: m x d2,
// row-major, FP64.  64 x 64 output tiles, split over K into `ks` partials that
// a second kernel adds in fixed order.
constexpr int kGT = 64, kGK = 16;

__global__ void __launch_bounds__(256)
gram_tn_kernel(const double* __restrict__ A, int64_t lda, const double* __restrict__ B, int64_t ldb,
               int64_t m, int d1, int d2, int64_t kchunk, double* __restrict__ part) {
  __shared__ double As[kGK][kGT];
  __shared__ double Bs[kGK][kGT];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int i0 = blockIdx.y * kGT, j0 = blockIdx.x * kGT;
  const int64_t k0 = blockIdx.z * kchunk, k1 = min(m, k0 + kchunk);
  double acc[4][4] = {};
  for (int64_t kk = k0; kk < k1; kk += kGK) {
    for (int e = tid; e < kGK * kGT; e += 256) {
      int r = e / kGT, c = e % kGT;
      int64_t row = kk + r;
      As[r][c] = (row < k1 && i0 + c < d1) ? A[row * lda + i0 + c] : 0.0;
      Bs[r][c] = (row < k1 && j0 + c < d2) ? B[row * ldb + j0 + c] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kGK; ++r) {
      double a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = As[r][ty + 16 * u];
#pragma unroll
      for (int u = 0; u < 4; ++u) b[u] = Bs[r][tx + 16 * u];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int w = 0; w < 4; ++w) acc[u][w] += a[u] * b[w];
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      int i = i0 + ty + 16 * u, j = j0 + tx + 16 * w;
      if (i < d1 && j < d2) part[((int64_t)blockIdx.z * d1 + i) * d2 + j] = acc[u][w];
    }
}

// The same partials on 16 x 16 tiles, one entry per thread (the same chain of
// terms), for matrices whose 64 x 64 tiles would leave SMs idle: a tile's 64 rows
// are 70 us of FP64 issue on one SM, three times in a solve with 50 columns.
__global__ void __launch_bounds__(256)
gram_tn_small_kernel(const double* __restrict__ A, int64_t lda, const double* __restrict__ B, int64_t ldb,
                     int64_t m, int d1, int d2, int64_t kchunk, double* __restrict__ part) {
  constexpr int kR = 64;  // rows per step
  __shared__ double As[kR][17], Bs[kR][17];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int i0 = blockIdx.y * 16, j0 = blockIdx.x * 16;
  const int64_t k0 = blockIdx.z * kchunk, k1 = min(m, k0 + kchunk);
  double acc = 0.0;
  for (int64_t kk = k0; kk < k1; kk += kR) {
#pragma unroll
    for (int u = 0; u < kR / 16; ++u) {
      const int r = ty + 16 * u;
      const int64_t row = kk + r;
      As[r][tx] = row < k1 && i0 + tx < d1 ? A[row * lda + i0 + tx] : 0.0;
      Bs[r][tx] = row < k1 && j0 + tx < d2 ? B[row * ldb + j0 + tx] : 0.0;
    }
    __syncthreads();
    const int nr = (int)min((int64_t)kR, k1 - kk);
#pragma unroll 8
    for (int r = 0; r < nr; ++r) acc += As[r][ty] * Bs[r][tx];
    __syncthreads();
  }
  if (i0 + ty < d1 && j0 + tx < d2) part[((int64_t)blockIdx.z * d1 + i0 + ty) * d2 + j0 + tx] = acc;
}

static void launch_gram_tn(const double* A, int64_t lda, const double* B, int64_t ldb, int64_t m, int d1, int d2, int ks,
                           int64_t kchunk, double* part, cudaStream_t st) {
  if (ceil_div(d1, kGT) * ceil_div(d2, kGT) * ks < 152)
    gram_tn_small_kernel<<<dim3(ceil_div(d2, 16), ceil_div(d1, 16), ks), 256, 0, st>>>(A, lda, B, ldb, m, d1, d2, kchunk,
                                                                                     part);
  else
    gram_tn_kernel<<<dim3(ceil_div(d2, kGT), ceil_div(d1, kGT), ks), 256, 0, st>>>(A, lda, B, ldb, m, d1, d2, kchunk, part);
}

// C (d x d) from the split-K partials of a symmetric Gram whose tiles were
// formed on and below the diagonal only: the upper tiles mirror the lower.
__global__ void sum_parts_sym_kernel(const double* __restrict__ part, int nparts, int d, double diag_add,
                                     double* __restrict__ C) {
  const int64_t len = (int64_t)d * d;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < len; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / d), j = (int)(e % d);
    const int64_t src = (i / kGT >= j / kGT) ? e : (int64_t)j * d + i;
    double s = 0;
    for (int p = 0; p < nparts; ++p) s += part[(int64_t)p * len + src];
    if (i == j) s += diag_add;
    C[e] = s;
  }
}

__global__ void sum_parts_kernel(const double* __restrict__ part, int nparts, int64_t len, int d1, int d2,
                                 double diag_add, double* __restrict__ C) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < len; e += (int64_t)gridDim.x * blockDim.x) {
    double s = 0;
    for (int p = 0; p < nparts; ++p) s += part[(int64_t)p * len + e];
    int i = (int)(e / d2), j = (int)(e % d2);
    if (i == j) s += diag_add;
    C[e] = s;
  }
}

// Double-float multiply-add (inputs split into FP32 pairs hi + lo; products
// hi*hi formed exactly as an FP32 pair with fma, the cross terms hi*lo +
// lo*hi added to the compensation; sums kept as FP32 pairs with TwoSum).  About 2^-44 relative accuracy per term at FP32 instruction rates:
// GB300 executes FP64 at ~1/60 of its FP32 rate.
__device__ __forceinline__ void df_acc(float& S, float& Cc, float ah, float al, float bh, float bl) {
  const float p = ah * bh;
  const float e = fmaf(ah, bh, -p);
  const float t = S + p;
  const float bp = t - S;
  const float err = (S - (t - bp)) + (p - bp);
  S = t;
  Cc += err + e + fmaf(ah, bl, al * bh);
}

// The same double-float Gram from inputs already split into float pairs
// (A = Ah + Al, B = Bh + Bl, row-major with leading dimensions lda, ldb):
// the tile loads are plain float loads, batched, with no FP64 conversions.
// tri: A and B lower triangular (A[q][i] = 0 for i > q), so rows
// q < max(i0, j0) contribute nothing to a tile.
__global__ void __launch_bounds__(256)
gram_dfs_kernel(const float* __restrict__ Ahg, const float* __restrict__ Alg, int64_t lda, const float* __restrict__ Bhg,
                const float* __restrict__ Blg, int64_t ldb, int64_t m, int d1, int d2, int64_t kchunk,
                double* __restrict__ part, int tri, int sym) {
  __shared__ float Ah[kGK][kGT], Al[kGK][kGT], Bh[kGK][kGT], Bl[kGK][kGT];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  int i0, j0;
  if (sym) {
    // A == B: only the tiles on and below the diagonal, blockIdx.x = ti (ti + 1) / 2 + tj
    const int t = blockIdx.x;
    int ti = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
    while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
    while (ti * (ti + 1) / 2 > t) --ti;
    i0 = ti * kGT;
    j0 = (t - ti * (ti + 1) / 2) * kGT;
  } else {
    i0 = blockIdx.y * kGT;
    j0 = blockIdx.x * kGT;
  }
  const int64_t k1 = min(m, (int64_t)blockIdx.z * kchunk + kchunk);
  const int64_t k0 = tri ? max((int64_t)blockIdx.z * kchunk, (int64_t)max(i0, j0)) : (int64_t)blockIdx.z * kchunk;
  float S[4][4] = {}, Cc[4][4] = {};
  for (int64_t kk = k0; kk < k1; kk += kGK) {
    float v[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + 256 * u, r = e / kGT, c = e % kGT;
      const int64_t row = kk + r;
      const bool ia = row < k1 && i0 + c < d1, ib = row < k1 && j0 + c < d2;
      v[u][0] = ia ? Ahg[row * lda + i0 + c] : 0.f;
      v[u][1] = ia ? Alg[row * lda + i0 + c] : 0.f;
      v[u][2] = ib ? Bhg[row * ldb + j0 + c] : 0.f;
      v[u][3] = ib ? Blg[row * ldb + j0 + c] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + 256 * u, r = e / kGT, c = e % kGT;
      Ah[r][c] = v[u][0];
      Al[r][c] = v[u][1];
      Bh[r][c] = v[u][2];
      Bl[r][c] = v[u][3];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kGK; ++r) {
      float ah[4], al[4], bh[4], bl[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        ah[u] = Ah[r][ty + 16 * u];
        al[u] = Al[r][ty + 16 * u];
        bh[u] = Bh[r][tx + 16 * u];
        bl[u] = Bl[r][tx + 16 * u];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int w = 0; w < 4; ++w) df_acc(S[u][w], Cc[u][w], ah[u], al[u], bh[w], bl[w]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int i = i0 + ty + 16 * u, j = j0 + tx + 16 * w;
      if (i < d1 && j < d2) part[((int64_t)blockIdx.z * d1 + i) * d2 + j] = (double)S[u][w] + (double)Cc[u][w];
    }
}

// Ranges of rows over which a Gram of `tiles` tiles and `len` entries is summed
// in FP32, as many as fill the GPU and the workspace holds.
static int df_splits(int tiles, int64_t len, int64_t m, bool tri, int64_t ws_len) {
  int ks = std::max(1, std::min<int>(ceil_div(tri ? 2 * 304 : 304, tiles), ceil_div(m, 64)));
  while (ks > 1 && (int64_t)ks * len > ws_len) --ks;
  return ks;
}
int64_t gram_df_chunk(int64_t m, int d, int64_t ws_len) {
  const int td = ceil_div(d, kGT), ks = df_splits(td * (td + 1) / 2, (int64_t)d * d, m, false, ws_len);
  return (m + ks - 1) / ks;
}

int gram_df_split(const float* Ah, const float* Al, int64_t lda, const float* Bh, const float* Bl, int64_t ldb,
                  int64_t m, int d1, int d2, double* C, double diag_add, double* ws, int64_t ws_len, cudaStream_t st,
                  bool tri) {
  // the same operand on both sides: a symmetric result, formed from the
  // tiles on and below the diagonal only
  const bool sym = Ah == Bh && Al == Bl && lda == ldb && d1 == d2;
  const int td = ceil_div(d1, kGT);
  const int tiles = sym ? td * (td + 1) / 2 : ceil_div(d1, kGT) * ceil_div(d2, kGT);
  const int64_t len = (int64_t)d1 * d2;
  const int ks = df_splits(tiles, len, m, tri, ws_len);
  if ((int64_t)ks * len > ws_len) {
    set_last_error("gram_df_split: workspace too small");
    return GBCCA_ERR_INVALID_ARG;
  }
  const int64_t kchunk = (m + ks - 1) / ks;
  dim3 grid = sym ? dim3(tiles, 1, ks) : dim3(ceil_div(d2, kGT), ceil_div(d1, kGT), ks);
  gram_dfs_kernel<<<grid, 256, 0, st>>>(Ah, Al, lda, Bh, Bl, ldb, m, d1, d2, kchunk, ws, tri ? 1 : 0, sym ? 1 : 0);
  GB_CHECK_LAUNCH();
  if (sym)
    sum_parts_sym_kernel<<<ceil_div(len, 256), 256, 0, st>>>(ws, ks, d1, diag_add, C);
  else
    sum_parts_kernel<<<ceil_div(len, 256), 256, 0, st>>>(ws, ks, len, d1, d2, diag_add, C);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

int gram_tn(const double* A, int64_t lda, const double* B, int64_t ldb, int64_t m, int d1, int d2, double* C,
            double diag_add, double* ws, int64_t ws_len, cudaStream_t st) {
  int tiles = ceil_div(d1, kGT) * ceil_div(d2, kGT);
  int ks = std::max(1, std::min<int>(ceil_div(304, tiles), ceil_div(m, 64)));
  int64_t len = (int64_t)d1 * d2;
  while (ks > 1 && (int64_t)ks * len > ws_len) --ks;
  if ((int64_t)ks * len > ws_len) {
    set_last_error("gram_tn: workspace too small");
    return GBCCA_ERR_INVALID_ARG;
  }
  int64_t kchunk = (m + ks - 1) / ks;
  launch_gram_tn(A, lda, B, ldb, m, d1, d2, ks, kchunk, ws, st);
  GB_CHECK_LAUNCH();
  sum_parts_kernel<<<ceil_div(len, 256), 256, 0, st>>>(ws, ks, len, d1, d2, diag_add, C);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// ------------------------------------------- M^{-1} in double-float form
// For FP32/BF16 plans the solver applies M^{-1} = R^{-1} R^{-T} (Table 1's
// preconditioned gradient) through an explicit symmetric matrix held as a
// float pair hi + lo (~2^-44 relative), formed once per preconditioner, and
// multiplied with double-float arithmetic.  One launch covers both views and
// replaces two dependent triangular products per view; its rounding error is
// ~2^-44 sqrt(d) kappa(M), below that of FP32 triangular products
// (~2^-24 kappa(R) each).
__global__ void split_df_kernel(const double* __restrict__ A, int64_t len, float* __restrict__ hi,
                                float* __restrict__ lo) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= len) return;
  const double x = A[e];
  const float h = (float)x;
  hi[e] = h;
  lo[e] = (float)(x - (double)h);
}

int minv_df_build(const double* Rinv, int d, float* hi, float* lo, double* ws, int64_t ws_len, cudaStream_t st) {
  const int64_t dd = (int64_t)d * d;
  if (ws_len < 5 * dd) {
    set_last_error("minv_df_build: workspace too small");
    return GBCCA_ERR_INVALID_ARG;
  }
  // T = R^{-T} (lower triangular) as a float pair, then C = T^T T = R^{-1} R^{-T}
  float* Th = reinterpret_cast<float*>(ws);
  float* Tl = Th + dd;
  double* C = ws + dd;
  GB_TRY(split_df(Rinv, d, d, true, Th, Tl, st));
  GB_TRY(gram_df_split(Th, Tl, d, Th, Tl, d, d, d, d, C, 0.0, ws + 2 * dd, ws_len - 2 * dd, st, true));
  split_df_kernel<<<ceil_div(dd, 256), 256, 0, st>>>(C, dd, hi, lo);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

__device__ __forceinline__ void df_add(float& S, float& Cc, float s2, float c2) {
  const float t = S + s2;
  const float bp = t - S;
  const float err = (S - (t - bp)) + (s2 - bp);
  S = t;
  Cc += err + c2;
}

constexpr int kMvThreads = 256;
constexpr int kMvStageBytes = 212992;  // shared memory of one staged K chunk (A rows + X rows) at most

// n floats (4, 2 or 1) from global to shared memory, asynchronously
__device__ __forceinline__ void cp_async_f(float* smem, const float* gmem, int n) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem);
  if (n == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem) : "memory");
  else if (n == 2) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(gmem) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gmem) : "memory");
}
// the widest of those that keeps every row start of two matrices aligned
static int copy_width(const float* a, const float* b, int cols, int ld) {
  const uintptr_t at = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b);
  if ((cols | ld) % 4 == 0 && at % 16 == 0) return 4;
  return (cols | ld) % 2 == 0 && at % 8 == 0 ? 2 : 1;
}
__host__ __device__ __forceinline__ int mv_cols(int c) { return (c + 3) / 4 * 4; }

// Y_b (m x c) = A_b X_b for problem b = blockIdx.y, A_b (m x K, row-major)
// and X_b (K x c, row stride ldx) as double-float pairs hi + lo; optionally
// Y_b as a pair too (Yh, Yl, row stride c).  A CTA owns kMvRows rows of Y, as
// few (2, 4, 6 or 8) as put one CTA on every SM: a CTA stages all of X, so more
// CTAs than SMs only stage it again.  The
// K range is walked in chunks staged in shared memory by the widest
// asynchronous copies the alignment allows, in two halves, so that the first
// is worked on while the second arrives.  A thread owns 2 rows x 4 columns of
// an interleaved slice of K (KS slices): eight double-float multiply-adds (12
// FP32 instructions each) for six shared-memory loads.  The KS partial pairs
// of an output are added in fixed order through shared memory at the end: no
// scratch in global memory, no atomics, and the result does not depend on
// scheduling.  Bound by FP32 issue (512 x 512 x 20, two views: 3 us of
// arithmetic); one output per thread behind 4-byte copies of all of X per
// four rows took 13 to 19 us a launch.
template <int kMvRows>
__global__ void __launch_bounds__(kMvThreads) dfmv_kernel(DfmvArgs a) {
  if (a.done != nullptr && *a.done) return;
  // the problem's fields by selection (a dynamic index into the parameter
  // array would copy it to local memory)
  const bool b1 = blockIdx.y != 0;
#define GB_SEL(f) (b1 ? a.p[1].f : a.p[0].f)
  struct {
    const float *hi, *lo, *Xh, *Xl;
    double* Y;
    int m, K, ldx, ldy;
    float *Yh, *Yl;
    int wa, wx;
  } P{GB_SEL(hi), GB_SEL(lo), GB_SEL(Xh), GB_SEL(Xl), GB_SEL(Y), GB_SEL(m), GB_SEL(K), GB_SEL(ldx), GB_SEL(ldy),
      GB_SEL(Yh), GB_SEL(Yl), GB_SEL(wa), GB_SEL(wx)};
#undef GB_SEL
  const int r0 = blockIdx.x * kMvRows;
  if (r0 >= P.m) return;  // uniform over the CTA
  extern __shared__ __align__(16) float mvs[];
  const int c = a.c, cp = mv_cols(c), Kc = a.kc, lda = Kc + 4;
  float* Ah = mvs;                 // [kMvRows][lda]
  float* Al = Ah + kMvRows * lda;
  float* Xh = Al + kMvRows * lda;  // [Kc][cp]
  float* Xl = Xh + Kc * cp;
  const int t = threadIdx.x;
  const int CG = cp / 4, per = kMvRows / 2 * CG;  // threads of a slice: row pairs x CG column groups
  const int KS = kMvThreads / per;
  const int ks = t / per, w = t - ks * per, rg = w / CG, cg = w - rg * CG;
  const bool active = ks < KS;
  const int wa = P.wa, wx = P.wx;
  // pad columns of X hold zeros (they are never copied)
  if (cp != c)
    for (int i = t; i < Kc * (cp - c); i += kMvThreads) {
      const int q = i / (cp - c), cc = c + i - q * (cp - c);
      Xh[q * cp + cc] = 0.f;
      Xl[q * cp + cc] = 0.f;
    }
  float S[2][4] = {}, Cc[2][4] = {};
  for (int k0 = 0; k0 < P.K; k0 += Kc) {
    const int kn = min(Kc, P.K - k0), half = min(kn, (kn + 7) / 8 * 4);
    __syncthreads();  // the previous chunk has been consumed
    for (int h = 0; h < 2; ++h) {
      const int q0 = h == 0 ? 0 : half, qn = (h == 0 ? half : kn) - q0;
      const int na = qn / wa;  // (half and K are multiples of wa)
      for (int i = t; i < kMvRows * na; i += kMvThreads) {
        const int r = i / na, q = q0 + (i - r * na) * wa;
        const int64_t o = (int64_t)min(r0 + r, P.m - 1) * P.K + k0 + q;
        cp_async_f(Ah + r * lda + q, P.hi + o, wa);
        cp_async_f(Al + r * lda + q, P.lo + o, wa);
      }
      const int nx = c / wx;
      for (int i = t; i < qn * nx; i += kMvThreads) {
        const int q = q0 + i / nx, cc = (i % nx) * wx;
        const int64_t o = (int64_t)(k0 + q) * P.ldx + cc;
        cp_async_f(Xh + q * cp + cc, P.Xh + o, wx);
        cp_async_f(Xl + q * cp + cc, P.Xl + o, wx);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int h = 0; h < 2; ++h) {
      if (h == 0) asm volatile("cp.async.wait_group 1;" ::: "memory");
      else asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      if (active) {
        const float *ah = Ah + 2 * rg * lda, *al = Al + 2 * rg * lda;
        const int q1 = h == 0 ? half : kn;
#pragma unroll 2
        for (int q = (h == 0 ? 0 : half) + ks; q < q1; q += KS) {
          const float4 xh = *reinterpret_cast<const float4*>(Xh + q * cp + 4 * cg);
          const float4 xl = *reinterpret_cast<const float4*>(Xl + q * cp + 4 * cg);
          const float xhv[4] = {xh.x, xh.y, xh.z, xh.w}, xlv[4] = {xl.x, xl.y, xl.z, xl.w};
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const float vh = ah[u * lda + q], vl = al[u * lda + q];
#pragma unroll
            for (int j = 0; j < 4; ++j) df_acc(S[u][j], Cc[u][j], vh, vl, xhv[j], xlv[j]);
          }
        }
      }
    }
  }
  __syncthreads();
  float2* red = reinterpret_cast<float2*>(mvs);  // [KS][kMvRows][cp]
  const int nout = kMvRows * cp;
  if (active) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int j = 0; j < 4; ++j) red[ks * nout + (2 * rg + u) * cp + 4 * cg + j] = make_float2(S[u][j], Cc[u][j]);
  }
  __syncthreads();
  for (int e = t; e < kMvRows * c; e += kMvThreads) {
    const int r = e / c, col = e - r * c;
    if (r0 + r >= P.m) continue;
    float sum = 0.f, cc = 0.f;
    for (int q = 0; q < KS; ++q) {
      const float2 v = red[q * nout + r * cp + col];
      df_add(sum, cc, v.x, v.y);
    }
    const double y = (double)sum + (double)cc;
    P.Y[(int64_t)(r0 + r) * P.ldy + col] = y;
    if (P.Yh != nullptr) {
      const float h = (float)y;
      P.Yh[(int64_t)(r0 + r) * c + col] = h;
      P.Yl[(int64_t)(r0 + r) * c + col] = (float)(y - (double)h);
    }
  }
}

int dfmv(const DfmvArgs& a, int nprob, int sm_count, cudaStream_t st) {
  if (a.c < 1 || a.c > 64 || nprob < 1 || nprob > 2) {
    set_last_error("dfmv: unsupported column count");
    return GBCCA_ERR_INVALID_ARG;
  }
  int mmax = 0, kmax = 0;
  for (int b = 0; b < nprob; ++b) {
    if (a.p[b].ldx < a.c) {
      set_last_error("dfmv: X rows must hold c columns");
      return GBCCA_ERR_INVALID_ARG;
    }
    mmax = std::max(mmax, a.p[b].m);
    kmax = std::max(kmax, a.p[b].K);
  }
  // K chunk: as few equal chunks (multiples of 32) as the staged rows of A
  // and X allow; the final reduction (at most 16 KB) reuses the space
  DfmvArgs g = a;
  for (int b = 0; b < nprob; ++b) {
    g.p[b].wa = copy_width(a.p[b].hi, a.p[b].lo, a.p[b].K, 0);
    g.p[b].wx = copy_width(a.p[b].Xh, a.p[b].Xl, a.c, a.p[b].ldx);
  }
  int64_t rows_all = 0;
  for (int b = 0; b < nprob; ++b) rows_all += a.p[b].m;
  const int rows = 2 * (int)std::max<int64_t>(1, std::min<int64_t>(4, ceil_div(rows_all, 2 * sm_count)));
  const int per_q = 8 * (rows + mv_cols(a.c));
  const int chunks = ceil_div((int64_t)kmax * per_q, kMvStageBytes);
  g.kc = (ceil_div(kmax, chunks) + 31) / 32 * 32;
  const size_t smem = std::max<size_t>((size_t)per_q * g.kc + 8 * rows * 4, 8 * 8 * (size_t)kMvThreads);
  auto kern = rows == 2 ? dfmv_kernel<2> : rows == 4 ? dfmv_kernel<4> : rows == 6 ? dfmv_kernel<6> : dfmv_kernel<8>;
  GB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  kern<<<dim3(ceil_div(mmax, rows), nprob), kMvThreads, smem, st>>>(g);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// hi/lo split of the first c columns of X (rows x ldx doubles) into two
// rows x c float arrays
__global__ void split_rows_kernel(const double* __restrict__ X, int rows, int c, int ldx, float* __restrict__ hi,
                                  float* __restrict__ lo) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= rows * c) return;
  const int i = e / c, j = e - i * c;
  const double x = X[(int64_t)i * ldx + j];
  const float h = (float)x;
  hi[e] = h;
  lo[e] = (float)(x - (double)h);
}

int split_rows(const double* X, int rows, int c, int ldx, float* hi, float* lo, cudaStream_t st) {
  split_rows_kernel<<<ceil_div(rows * c, 256), 256, 0, st>>>(X, rows, c, ldx, hi, lo);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// hi/lo split of A (r x c) or of A^T
__global__ void split_df_t_kernel(const double* __restrict__ A, int r, int c, int trans, float* __restrict__ hi,
                                  float* __restrict__ lo) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)r * c) return;
  const int i = (int)(e / c), j = (int)(e % c);
  const double x = A[e];
  const float h = (float)x;
  const int64_t o = trans ? (int64_t)j * r + i : e;
  hi[o] = h;
  lo[o] = (float)(x - (double)h);
}

int split_df(const double* A, int r, int c, bool trans, float* hi, float* lo, cudaStream_t st) {
  split_df_t_kernel<<<ceil_div((int64_t)r * c, 256), 256, 0, st>>>(A, r, c, trans ? 1 : 0, hi, lo);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// ------------------------------------------------- allocation-free Gram
// The same split-K Gram as gram_tn (FP64 gram_tn_kernel + sum_parts_kernel),
// with its partial slabs in a fixed static device array instead of plan
// memory.  It serves callers that may not allocate device memory at all: a
// process that has reserved HBM up front in its own pool and budgets every
// byte, or one that cannot accept the device-wide synchronization that
// cudaMalloc / cudaFree may impose on all of its streams.
//
// Limit: the scratch holds kNoAllocScratch doubles (8 MiB).  A call needs at
// least one d x d partial slab, so d <= 1024; larger d is rejected with
// GBCCA_ERR_INVALID_ARG before any device work.  The number of split-K slabs
// is as many as fit (up to one per 64 rows and enough CTAs for the GPU).  Nothing in the scratch has
// to start at zero: every element of a slab that the second kernel reads is
// written by the first.  The scratch is one buffer per device shared by all
// callers, so two calls whose kernels may overlap in time (different streams,
// or threads without ordering) race on it; callers order them.
constexpr int64_t kNoAllocScratch = int64_t(1) << 20;
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocScratch];

namespace {
constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
double* g_noalloc_ptr[kNoAllocMaxDevices] = {};

// Device address of the scratch for the current device, looked up once per
// device.  The first call on a device resolves the symbol (which can load the
// module), so a caller that records work into a stream capture makes one
// call on that device before capturing.
int noalloc_scratch(double** out) {
  int dev = -1;
  GB_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kNoAllocMaxDevices) {
    set_last_error("allocation-free Gram: device ordinal out of range");
    return GBCCA_ERR_INVALID_ARG;
  }
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (g_noalloc_ptr[dev] == nullptr) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || p == nullptr) {
      set_last_error(std::string("cudaGetSymbolAddress(scratch): ") + cudaGetErrorString(e));
      return GBCCA_ERR_CUDA;
    }
    g_noalloc_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return GBCCA_OK;
}
}  // namespace

int noalloc_max_d() {
  int d = 1;
  while ((int64_t)(d + 1) * (d + 1) <= kNoAllocScratch) ++d;
  return d;
}

int gram_noalloc(const double* A, int64_t lda, int64_t m, int d, double lambda, double* C, cudaStream_t st) {
  const int64_t len = (int64_t)d * d;
  if (len > kNoAllocScratch) {
    set_last_error("allocation-free Gram: d = " + std::to_string(d) + " exceeds the " +
                   std::to_string(noalloc_max_d()) + " columns its 8 MiB static scratch holds");
    return GBCCA_ERR_INVALID_ARG;
  }
  double* ws = nullptr;
  GB_TRY(noalloc_scratch(&ws));
  const int tiles = ceil_div(d, kGT) * ceil_div(d, kGT);
  int ks = std::max(1, std::min<int>(ceil_div(304, tiles), ceil_div(m, 64)));
  while (ks > 1 && (int64_t)ks * len > kNoAllocScratch) --ks;
  const int64_t kchunk = (m + ks - 1) / ks;
  launch_gram_tn(A, lda, A, lda, m, d, d, ks, kchunk, ws, st);
  GB_CHECK_LAUNCH();
  sum_parts_kernel<<<ceil_div(len, 256), 256, 0, st>>>(ws, ks, len, d, d, lambda, C);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// --------------------------------------------------------------- Cholesky
// Right-looking blocked Cholesky of a symmetric positive definite d x d
// matrix (only its lower triangle is read): A = L L^T with 32 x 32 blocks.
// At the end R = L^T is written to the upper triangle and the strict lower
// triangle is zeroed, so A holds R with R^T R = A.  A non-positive pivot sets
// *flag = 1 (the caller reports GBCCA_ERR_NOT_SPD).
constexpr int kNB = 32;

__global__ void __launch_bounds__(128) chol_diag_kernel(double* A, int d, int p, int* flag) {
  // The 32 x 32 diagonal block in shared memory, factored by 4 warps: GB300
  // issues FP64 at a small fraction of its FP32 rate on each of the SM's four
  // schedulers, so the trailing updates of every step are spread over all four.
  __shared__ double L[kNB][kNB + 1];
  __shared__ double s_r;
  __shared__ int s_bad;
  const int tid = threadIdx.x;
  const int o = p * kNB, nb = min(kNB, d - o);
  for (int e = tid; e < kNB * kNB; e += blockDim.x) {
    const int r = e / kNB, c = e % kNB;
    L[r][c] = (r < nb && c <= r) ? A[(int64_t)(o + r) * d + o + c] : 0.0;
  }
  if (tid == 0) s_bad = 0;
  __syncthreads();
  for (int j = 0; j < nb; ++j) {
    if (tid == 0) {
      double piv = L[j][j];
      if (!(piv > 0.0)) {
        s_bad = 1;
        piv = 1.0;  // keep going with a harmless value; the result is discarded
      }
      const double rj = rsqrt_nr(piv);
      L[j][j] = piv * rj;
      s_r = rj;
    }
    __syncthreads();
    for (int i = j + 1 + tid; i < nb; i += blockDim.x) L[i][j] *= s_r;
    __syncthreads();
    // trailing lower triangle (i, c), j < c <= i < nb, enumerated row by row
    const int m = nb - j - 1, cnt = m * (m + 1) / 2;
    for (int e = tid; e < cnt; e += blockDim.x) {
      int i1 = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
      while ((i1 + 1) * (i1 + 2) / 2 <= e) ++i1;
      while (i1 * (i1 + 1) / 2 > e) --i1;
      const int i = j + 1 + i1, c = j + 1 + (e - i1 * (i1 + 1) / 2);
      L[i][c] -= L[i][j] * L[c][j];
    }
    __syncthreads();
  }
  if (tid == 0 && s_bad) raise_flag(flag, kFlagNotSpd);
  for (int e = tid; e < nb * nb; e += blockDim.x) {
    const int r = e / nb, c = e % nb;
    if (c <= r) A[(int64_t)(o + r) * d + o + c] = L[r][c];
  }
}

// A[i-block, p] <- A[i-block, p] L_pp^{-T}: one warp per row, lane c holding
// x_c; forward substitution in column order, each solved x_c broadcast by a
// shuffle to the lanes that still subtract it (the same multiply-adds, in the
// same order, as a serial substitution of the row).
constexpr int kTrsmRows = 8;  // rows (warps) per CTA
__global__ void __launch_bounds__(32 * kTrsmRows) chol_trsm_kernel(double* A, int d, int p) {
  __shared__ double L[kNB][kNB + 1];
  __shared__ double rinv[kNB];
  const int o = p * kNB, nb = min(kNB, d - o);
  for (int e = threadIdx.x; e < kNB * kNB; e += blockDim.x) {
    int r = e / kNB, c = e % kNB;
    L[r][c] = (r < nb && c <= r) ? A[(int64_t)(o + r) * d + o + c] : 0.0;
  }
  __syncthreads();
  if (threadIdx.x < kNB) rinv[threadIdx.x] = threadIdx.x < nb ? 1.0 / L[threadIdx.x][threadIdx.x] : 1.0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int row = o + nb + blockIdx.x * kTrsmRows + (threadIdx.x >> 5);
  if (row >= d) return;  // uniform over the warp
  double acc = lane < nb ? A[(int64_t)row * d + o + lane] : 0.0;
  double x = 0.0;
  for (int c = 0; c < nb; ++c) {
    if (lane == c) x = acc * rinv[c];
    const double xc = __shfl_sync(0xffffffffu, x, c);
    if (lane > c) acc -= L[lane][c] * xc;
  }
  if (lane < nb) A[(int64_t)row * d + o + lane] = x;
}

// Tile t of the trailing matrix's lower triangle in 16 x 16 tiles (row-major
// order: t = ti (ti + 1) / 2 + tj), A[I, J] -= A[I, p] A[J, p]^T with p the panel
// of 32 columns at `o`: one entry per thread, its 32 terms in order.  (On 32 x
// 32 tiles a step had few CTAs with 10 us of FP64 each.)
constexpr int kUT = 16;
__device__ __forceinline__ void chol_update_tile(double* A, int d, int o, int t, double (*a)[kNB + 1],
                                                 double (*b)[kNB + 1]) {
  int ti = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
  while (ti * (ti + 1) / 2 > t) --ti;
  const int tj = t - ti * (ti + 1) / 2;
  const int i0 = o + kNB + kUT * ti, j0 = o + kNB + kUT * tj;
  for (int e = threadIdx.x; e < kUT * kNB; e += blockDim.x) {
    const int r = e / kNB, c = e % kNB;
    a[r][c] = i0 + r < d ? A[(int64_t)(i0 + r) * d + o + c] : 0.0;
    b[r][c] = j0 + r < d ? A[(int64_t)(j0 + r) * d + o + c] : 0.0;
  }
  __syncthreads();
  const int r = threadIdx.x / kUT, c = threadIdx.x % kUT;
  const int i = i0 + r, j = j0 + c;
  if (i >= d || j > i) return;
  double s = 0;
#pragma unroll 8
  for (int q = 0; q < kNB; ++q) s += a[r][q] * b[c][q];
  A[(int64_t)i * d + j] -= s;
}
inline int update_tiles(int rows) {
  const int T = ceil_div(rows, kUT);
  return T * (T + 1) / 2;
}

// trailing update behind panel p (FP64 plans)
__global__ void __launch_bounds__(256) chol_syrk_kernel(double* A, int d, int p) {
  __shared__ double a[kUT][kNB + 1], b[kUT][kNB + 1];
  chol_update_tile(A, d, p * kNB, blockIdx.x, a, b);
}

// FP32/BF16 plans: the trailing update behind panel p with the next diagonal
// block factored in the same launch (CTA 0: its own update, then L and
// L^{-1} by group_chol_inverse, 32 dependent steps; L^{-T} goes to the
// diagonal block of Rinv).  p = -1: the first diagonal block only.
__global__ void __launch_bounds__(256) chol_next_kernel(double* A, double* Rinv, int d, int p, int* flag) {
  __shared__ double sa[kNB][kNB + 1], sb[kNB][kNB + 1], rs[kNB];
  if (blockIdx.x > 0) {  // tiles 0 .. 2 are the diagonal block
    chol_update_tile(A, d, p * kNB, (int)blockIdx.x + 2, sa, sb);
    return;
  }
  const int o = (p + 1) * kNB, nb = min(kNB, d - o), tid = threadIdx.x;
  if (p >= 0) {
    for (int e = tid; e < kNB * kNB; e += 256) {
      const int r = e / kNB, c = e % kNB;
      sb[r][c] = r < nb ? A[(int64_t)(o + r) * d + o - kNB + c] : 0.0;
    }
    __syncthreads();
  }
  for (int e = tid; e < nb * (nb + 1) / 2; e += 256) {
    int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= e) ++i;
    while (i * (i + 1) / 2 > e) --i;
    const int c = e - i * (i + 1) / 2;
    double s = 0;
    if (p >= 0) {
#pragma unroll 8
      for (int q = 0; q < kNB; ++q) s += sb[i][q] * sb[c][q];
    }
    sa[i][c] = A[(int64_t)(o + i) * d + o + c] - s;
  }
  __syncthreads();
  const bool ok = group_chol_inverse<256>(&sa[0][0], &sb[0][0], rs, nb, tid, 0, kNB + 1);
  if (!ok && tid == 0) raise_flag(flag, kFlagNotSpd);
  for (int e = tid; e < nb * nb; e += 256) {
    const int r = e / nb, c = e % nb;
    if (c <= r) {
      A[(int64_t)(o + r) * d + o + c] = sa[r][c] * rs[c];      // L_cc = L_cc^2 / L_cc on the diagonal
      Rinv[(int64_t)(o + c) * d + o + r] = sb[r][c];
    }
  }
}

// A[rows below, p] <- A[rows below, p] L_pp^{-T}: a warp per row, lane c the
// column, the 32 terms of a product with the inverse block (no substitution
// chain).
__global__ void __launch_bounds__(256) chol_panel_kernel(double* A, const double* __restrict__ Rinv, int d, int p) {
  __shared__ double Ls[kNB][kNB];  // L^{-T}: row q, column c >= q
  const int o = p * kNB, lane = threadIdx.x & 31;
  for (int e = threadIdx.x; e < kNB * kNB; e += 256)
    Ls[e / kNB][e % kNB] = Rinv[(int64_t)(o + e / kNB) * d + o + e % kNB];
  __syncthreads();
  const int row = o + kNB + blockIdx.x * 8 + (threadIdx.x >> 5);
  if (row >= d) return;  // uniform over the warp
  const double v = A[(int64_t)row * d + o + lane];
  double x = 0.0;
#pragma unroll 8
  for (int q = 0; q < kNB; ++q) x += __shfl_sync(0xffffffffu, v, q) * Ls[q][lane];
  A[(int64_t)row * d + o + lane] = x;
}

__global__ void lower_to_upper_kernel(double* A, int d) {
  int i = blockIdx.y * 32 + threadIdx.y, j = blockIdx.x * 32 + threadIdx.x;
  if (i >= d || j >= d || j < i) return;
  double l = A[(int64_t)j * d + i];  // L[j][i], j >= i
  A[(int64_t)i * d + j] = l;          // R[i][j]
  if (j > i) A[(int64_t)j * d + i] = 0.0;
}

// FP64 plans: their iterations amplify a change of rounding in R, so every
// entry keeps the order of its sums (pivots by 1 / sqrt, substitution).
int cholesky_upper(double* A, int d, int* flag, cudaStream_t st) {
  int nbk = ceil_div(d, kNB);
  for (int p = 0; p < nbk; ++p) {
    chol_diag_kernel<<<1, 128, 0, st>>>(A, d, p, flag);
    GB_CHECK_LAUNCH();
    int below = d - (p + 1) * kNB;
    if (below > 0) {
      chol_trsm_kernel<<<ceil_div(below, kTrsmRows), 32 * kTrsmRows, 0, st>>>(A, d, p);
      GB_CHECK_LAUNCH();
      chol_syrk_kernel<<<update_tiles(below), 256, 0, st>>>(A, d, p);
      GB_CHECK_LAUNCH();
    }
  }
  lower_to_upper_kernel<<<dim3(ceil_div(d, 32), ceil_div(d, 32)), dim3(32, 32), 0, st>>>(A, d);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// FP32/BF16 plans: the same factor, two launches per 32 columns; also writes the
// diagonal blocks of Rinv = R^{-1} (which must be zero elsewhere in them).  A
// step took a 32 us factorization of the diagonal block by four warps, an 8 us
// substitution and a 15 us update (0.9 ms for d = 512), one after another.
int cholesky_upper_blocks(double* A, double* Rinv, int d, int* flag, cudaStream_t st) {
  const int nbk = ceil_div(d, kNB);
  chol_next_kernel<<<1, 256, 0, st>>>(A, Rinv, d, -1, flag);
  GB_CHECK_LAUNCH();
  for (int p = 0; p + 1 < nbk; ++p) {
    const int below = d - (p + 1) * kNB;
    chol_panel_kernel<<<ceil_div(below, 8), 256, 0, st>>>(A, Rinv, d, p);
    GB_CHECK_LAUNCH();
    chol_next_kernel<<<1 + std::max(0, update_tiles(below) - 3), 256, 0, st>>>(A, Rinv, d, p, flag);
    GB_CHECK_LAUNCH();
  }
  lower_to_upper_kernel<<<dim3(ceil_div(d, 32), ceil_div(d, 32)), dim3(32, 32), 0, st>>>(A, d);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// ------------------------------------------------------- triangular inverse
// Rinv = R^{-1} for upper-triangular R by recursive doubling over aligned
// diagonal blocks: the 32 x 32 diagonal blocks are inverted by back
// substitution, then at each level h = 32, 64, ... the inverted neighbours
// A = [r0, r0+h) and C = [c0, c1) (c0 = r0 + h) are joined through
//   Rinv[A, C] = -Rinv[A, A] (R[A, C] Rinv[C, C]),
// two FP64 products per level.  Every level is one parallel launch pair, so
// the d^3/3 multiply-adds spread over all SMs.
constexpr int kTB = 32;

__global__ void tri_diag_inv_kernel(const double* __restrict__ R, double* __restrict__ Rinv, int d) {
  __shared__ double L[kTB][kTB + 1];
  __shared__ double X[kTB][kTB + 1];
  __shared__ double rinv[kTB];
  const int o = blockIdx.x * kTB, nb = min(kTB, d - o), j = threadIdx.x;
  for (int r = 0; r < kTB; ++r) L[r][j] = (r < nb && j < nb && j >= r) ? R[(int64_t)(o + r) * d + o + j] : 0.0;
  __syncthreads();
  rinv[j] = j < nb ? 1.0 / L[j][j] : 0.0;
  __syncthreads();
  for (int i = kTB - 1; i >= 0; --i) {
    double x = 0.0;
    if (i <= j && j < nb) {
      double s = 0.0;
      for (int q = i + 1; q <= j; ++q) s += L[i][q] * X[q][j];
      x = ((i == j) ? 1.0 : 0.0) - s;
      x *= rinv[i];
    }
    X[i][j] = x;  // each thread owns column j: no barrier needed
  }
  for (int r = 0; r < nb; ++r)
    if (j < nb) Rinv[(int64_t)(o + r) * d + o + j] = X[r][j];
}

// stage 0: T_p = R[A, C] Rinv[C, C]  (h x w, row stride h)
// stage 1: Rinv[A, C] = -Rinv[A, A] T_p
// Grid (ceil(h/16), ceil(h/16), pairs); each CTA one 16 x 16 output tile, an
// entry per thread with its terms in order, K in chunks of 32 restricted to
// where the triangular factor is non-zero.  Bound by the FP64 rate: 32 x 32
// tiles left most SMs without work on all levels but the last (41 us a launch
// on average at d = 512).
constexpr int kTT = 16;
template <int kStage>
__global__ void __launch_bounds__(256) tri_level_kernel(const double* __restrict__ R, double* __restrict__ Rinv,
                                                        double* __restrict__ T, int d, int h) {
  __shared__ double As[kTT][kTB + 1], Bs[kTB][kTT + 1];
  const int p = blockIdx.z;
  const int r0 = 2 * p * h, c0 = r0 + h;
  if (c0 >= d) return;
  const int w = min(d, c0 + h) - c0;
  const int i0 = blockIdx.y * kTT, j0 = blockIdx.x * kTT;
  if (i0 >= h || j0 >= w) return;
  double* Tp = T + (int64_t)p * h * h;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  // K range: stage 0 runs q in [0, w) with Rinv[C,C][q][j] = 0 for q > j;
  // stage 1 runs q in [0, h) with Rinv[A,A][i][q] = 0 for q < i
  const int klo = kStage == 0 ? 0 : i0;
  const int khi = kStage == 0 ? min(w, j0 + kTT) : h;
  double acc = 0.0;
  for (int k0 = klo; k0 < khi; k0 += kTB) {
    for (int e = threadIdx.x; e < kTT * kTB; e += 256) {
      const int r = e / kTB, c = e % kTB;       // A tile element (i, q)
      const int ia = i0 + r, qa = k0 + c;
      const int qr = e / kTT, jc = e % kTT;     // B tile element (q, j)
      const int qb = k0 + qr, jb = j0 + jc;
      double av = 0.0, bv = 0.0;
      if (kStage == 0) {
        if (ia < h && qa < khi) av = R[(int64_t)(r0 + ia) * d + c0 + qa];
        if (qb < khi && jb < w) bv = Rinv[(int64_t)(c0 + qb) * d + c0 + jb];
      } else {
        if (ia < h && qa < khi) av = Rinv[(int64_t)(r0 + ia) * d + r0 + qa];
        if (qb < khi && jb < w) bv = Tp[(int64_t)qb * h + jb];
      }
      As[r][c] = av;
      Bs[qr][jc] = bv;
    }
    __syncthreads();
    const int kn = min(kTB, khi - k0);
#pragma unroll 8
    for (int q = 0; q < kn; ++q) acc += As[ty][q] * Bs[q][tx];
    __syncthreads();
  }
  const int i = i0 + ty, j = j0 + tx;
  if (i < h && j < w) {
    if (kStage == 0)
      Tp[(int64_t)i * h + j] = acc;
    else
      Rinv[(int64_t)(r0 + i) * d + c0 + j] = -acc;
  }
}

// have_diag: the diagonal blocks of Rinv are in place (and it is zero elsewhere)
int tri_inverse_upper(const double* R, double* Rinv, int d, double* ws, int64_t ws_len, cudaStream_t st, bool have_diag) {
  if (ws_len < (int64_t)d * d) {
    set_last_error("tri_inverse_upper: workspace too small");
    return GBCCA_ERR_INVALID_ARG;
  }
  if (!have_diag) {
    GB_CUDA(cudaMemsetAsync(Rinv, 0, sizeof(double) * d * d, st));
    tri_diag_inv_kernel<<<ceil_div(d, kTB), kTB, 0, st>>>(R, Rinv, d);
    GB_CHECK_LAUNCH();
  }
  for (int h = kTB; h < d; h *= 2) {
    const int pairs = ceil_div(d - h, 2 * h);
    dim3 grid(ceil_div(h, kTT), ceil_div(h, kTT), pairs);
    tri_level_kernel<0><<<grid, 256, 0, st>>>(R, Rinv, ws, d, h);
    GB_CHECK_LAUNCH();
    tri_level_kernel<1><<<grid, 256, 0, st>>>(R, Rinv, ws, d, h);
    GB_CHECK_LAUNCH();
  }
  return GBCCA_OK;
}

// ------------------------------------------------- triangular factor x block
// C (m x n) = T^T B (T upper triangular m x m, B m x n) or, with kRight, B T (B
// m x n, T upper triangular n x n), FP64: the two halves of the warm start's
// R_x^{-T} C_xy R_y^{-1}.  Each CTA one 16 x 16 tile, an entry per thread with its
// terms in order, the inner range cut to where T is non-zero, the longest
// ranges first.  Bound by the FP64 rate: with 512 columns in both views a
// preconditioner takes 130 us longer than with double-float products (3.16 to
// 3.29 ms), whose rounding, amplified by the factors, left singular pairs 9
// to 29 times further off than FP64 products do (condition 1e4).
template <bool kRight>
__global__ void __launch_bounds__(256) tri_mul_kernel(const double* __restrict__ T, const double* __restrict__ B, int m,
                                                      int n, double* __restrict__ C) {
  __shared__ double As[kTT][kTB + 1], Bs[kTB][kTT + 1];
  const int i0 = ((int)gridDim.y - 1 - (int)blockIdx.y) * kTT, j0 = ((int)gridDim.x - 1 - (int)blockIdx.x) * kTT;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int khi = kRight ? min(n, j0 + kTT) : min(m, i0 + kTT);
  double acc = 0.0;
  for (int k0 = 0; k0 < khi; k0 += kTB) {
    for (int e = threadIdx.x; e < kTT * kTB; e += 256) {
      const int i = i0 + (kRight ? e / kTB : e % kTT), qa = k0 + (kRight ? e % kTB : e / kTT);  // A(i, q): B or T^T
      const int j = j0 + e % kTT, qb = k0 + e / kTT;                                            // B(q, j): T or B
      const bool ia = i < m && qa < khi, ib = j < n && qb < khi;
      As[i - i0][qa - k0] = ia ? (kRight ? B[(int64_t)i * n + qa] : T[(int64_t)qa * m + i]) : 0.0;
      Bs[qb - k0][j - j0] = ib ? (kRight ? T[(int64_t)qb * n + j] : B[(int64_t)qb * n + j]) : 0.0;
    }
    __syncthreads();
    const int kn = min(kTB, khi - k0);
#pragma unroll 8
    for (int q = 0; q < kn; ++q) acc += As[ty][q] * Bs[q][tx];
    __syncthreads();
  }
  if (i0 + ty < m && j0 + tx < n) C[(int64_t)(i0 + ty) * n + j0 + tx] = acc;
}

int tri_mul(bool right, const double* T, const double* B, int m, int n, double* C, cudaStream_t st) {
  auto kern = right ? tri_mul_kernel<true> : tri_mul_kernel<false>;
  kern<<<dim3(ceil_div(n, kTT), ceil_div(m, kTT)), 256, 0, st>>>(T, B, m, n, C);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// ------------------------------------------------------ factor x thin block
// C (m x c) = op(A) B for up to two problems in one launch, FP64: A ra x ca
// row-major (op = identity or transpose), B and C with row strides ldb, ldc.
// With tri set, A is upper triangular and the inner range is cut to where
// op(A) is non-zero.  A CTA owns a few rows of C and at most 64 columns; its
// threads are outputs x 64-wide slices of the inner dimension, each slice one
// chain in the order of its terms, and the slices are added in order through
// shared memory (no scratch, no second launch).  Bound by the FP64 rate (a
// warp-wide multiply-add takes 64 cycles whatever its lanes hold, four warps
// saturate an SM), so lanes hold outputs only; a tile version that computed
// 40 columns whatever the shape took 23 + 3 us per product of a 50 x 50 factor
// with 10 columns, eight of them an iteration for two views.
constexpr int kSlice = 64;
constexpr size_t kThinStageBytes = 65536;  // staged operands (beyond it every CTA copying B costs more than it saves)

// (rows per CTA: as many as its 256 threads hold outputs x slices of, at most 8)
static int thin_rows(int c, int K) { return std::max(1, std::min(8, 256 / (c * ceil_div(K, kSlice)))); }

// kStage (operands that fit shared memory): the CTA's rows of op(A) and all of
// B are copied there at once, so that a product waits for memory once, not once
// per eight terms (50 x 50 times 5 columns: 6.6 us a launch with the loads in
// registers).
template <bool kStage>
__global__ void __launch_bounds__(256) mat_thin_kernel(ThinMul p0, ThinMul p1, int rows0, int rows1, int transA, int tri,
                                                       int c, int c0, const int* done) {
  extern __shared__ double red[];  // [slice][rows x c], then with kStage [rows][K + 1] of op(A) and [K][c] of B
  if (!kStage && done != nullptr && *done) return;
  const bool b1 = blockIdx.y != 0;
  const double* A = b1 ? p1.A : p0.A;
  const double* B = (b1 ? p1.B : p0.B) + c0;
  const int ra = b1 ? p1.ra : p0.ra, ca = b1 ? p1.ca : p0.ca, rows = b1 ? rows1 : rows0;
  const int64_t ldb = b1 ? p1.ldb : p0.ldb;
  const int m = transA ? ca : ra, K = transA ? ra : ca;
  const int i0 = blockIdx.x * rows;
  if (i0 >= m) return;  // uniform over the CTA
  const int nout = rows * c, ns = (K + kSlice - 1) / kSlice;
  double* As = red + nout * ns;
  double* Bs = As + rows * (K + 1);
  if constexpr (kStage) {
    auto copy = [](double* dst, const double* src) {
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                   : "memory");
    };
    const int nr = min(rows, m - i0);
    for (int f = threadIdx.x; f < rows * K; f += 256) {
      const int r = transA ? f % rows : f / K, l = transA ? f / rows : f - r * K;
      if (r < nr) copy(As + r * (K + 1) + l, transA ? A + (int64_t)l * ca + i0 + r : A + (int64_t)(i0 + r) * ca + l);
    }
    for (int f = threadIdx.x; f < K * c; f += 256) copy(Bs + f, B + (f / c) * ldb + f % c);
    const bool skip = done != nullptr && *done;  // read behind the copies' issue
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (skip) return;
  }
  for (int f = threadIdx.x; f < nout * ns; f += 256) {
    const int sl = f / nout, e = f - sl * nout, r = e / c, col = e - r * c, i = i0 + r;
    // op(A)[i][l] is non-zero for l >= i (A upper) or l <= i (its transpose)
    const int lo = max(sl * kSlice, tri && !transA ? i : 0);
    const int hi = min(min(K, (sl + 1) * kSlice), tri && transA ? i + 1 : K);
    double s = 0.0;
    if (kStage && i < m) {
      const double *Ar = As + r * (K + 1), *Bc = Bs + col;
#pragma unroll 8
      for (int l = lo; l < hi; ++l) s += Ar[l] * Bc[l * c];
    } else if (i < m) {
      const double* Ai = transA ? A + i : A + (int64_t)i * ca;
      const int64_t sa = transA ? ca : 1;
      // eight terms at a time, the next eight in flight under the arithmetic
      double x0[8], y0[8], x1[8], y1[8];
      auto load = [&](int l, double(&x)[8], double(&y)[8]) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int q = min(l + u, hi - 1);
          x[u] = Ai[q * sa];
          y[u] = B[q * ldb + col];
        }
      };
      auto add = [&](int l, const double(&x)[8], const double(&y)[8]) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (l + u < hi) s += x[u] * y[u];
      };
      if (lo < hi) load(lo, x0, y0);
      for (int l = lo; l < hi; l += 16) {
        load(l + 8, x1, y1);
        add(l, x0, y0);
        load(l + 16, x0, y0);
        add(l + 8, x1, y1);
      }
    }
    red[f] = s;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nout; e += 256) {
    const int r = e / c, col = e - r * c;
    if (i0 + r >= m) continue;
    double s = 0.0;
    for (int q = 0; q < ns; ++q) s += red[q * nout + e];
    (b1 ? p1.C : p0.C)[(int64_t)(i0 + r) * (b1 ? p1.ldc : p0.ldc) + c0 + col] = s;
  }
}

int mat_thin(const ThinMul* p, int nprob, bool transA, bool tri, int c, cudaStream_t st, const int* done) {
  for (int c0 = 0; c0 < c; c0 += 64) {
    const int cw = std::min(64, c - c0);
    int blocks = 1, rows[2] = {1, 1};
    size_t smem = 0, stage = 0;
    for (int b = 0; b < nprob; ++b) {
      const int m = transA ? p[b].ca : p[b].ra, K = transA ? p[b].ra : p[b].ca;
      rows[b] = thin_rows(cw, K);
      blocks = std::max(blocks, ceil_div(m, rows[b]));
      const size_t red = sizeof(double) * rows[b] * cw * ceil_div(K, kSlice);
      smem = std::max(smem, red);
      stage = std::max(stage, red + sizeof(double) * ((size_t)rows[b] * (K + 1) + (size_t)K * cw));
    }
    const bool staged = stage <= kThinStageBytes;
    if (staged) smem = stage;
    auto kern = staged ? mat_thin_kernel<true> : mat_thin_kernel<false>;
    GB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<dim3(blocks, nprob), 256, smem, st>>>(p[0], p[nprob > 1 ? 1 : 0], rows[0], rows[1], transA ? 1 : 0, tri ? 1 : 0,
                                                 cw, c0, done);
    GB_CHECK_LAUNCH();
  }
  return GBCCA_OK;
}

}  // namespace gbcca
