// Small dense factorizations inside one CTA (matrices of at most 40 columns in
// shared memory).  What bounds them on this GPU is the latency of dependent
// FP64 instructions and their issue rate (a warp-wide FP64 instruction holds
// its scheduler for tens of cycles), so every step uses as few dependent FP64
// instructions and barriers as possible, all four schedulers, and FP32 where
// the result is corrected afterwards.
#pragma once
#include "common.cuh"

namespace gbcca {

// 1 / x in FP64 by the Newton-Raphson iteration for 1 / y - x, y <- y + y (1 - x y),
// which doubles the correct bits: a single-precision quotient (about 22 bits),
// one step in FP32 with the mantissa of x split into a float and the rest, one
// step in FP64.  Only that last step is FP64 work (two dependent multiply-adds):
// the mantissa comes out of, and the reciprocal goes back into, a double as
// integers, since conversions run at the FP64 rate.  At most one unit in the
// last place from the quotient; 1 / x where x or the result is not normal.
__device__ __forceinline__ double rcp_nr(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int ex = (int)(hi >> 20 & 0x7ff);
  if ((unsigned)(ex - 2) > 2041u) return 1.0 / x;
  const float m = __uint_as_float(0x3f800000u | (hi & 0xfffffu) << 3 | lo >> 29);  // |x| = 2^(ex - 1023) (m + rest)
  const float rest = (float)(lo & 0x1fffffffu) * 2.220446049250313e-16f;          // 2^-52 a bit
  const float r = __fdividef(1.f, m);
  const float c = r * (fmaf(-m, r, 1.f) - rest * r);
  // r + c in units of 2^-52: r is a multiple of 2^-25, and 2^51 (one half)
  // starts the mantissa of exponent field 1022
  const long long y52 = ((long long)__float2int_rn(r * 33554432.f) << 27) + __float2int_rn(c * 4503599627370496.f);
  const long long bits = ((long long)(2045 - ex) << 52) + ((y52 - (1ll << 51)) << 1);
  const double y = __longlong_as_double(bits | (long long)(hi & 0x80000000u) << 32);
  return fma(y, fma(-x, y, 1.0), y);
}

// Barrier over the G threads of a group (id 0: the whole CTA).
template <int G>
__device__ __forceinline__ void group_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(G) : "memory");
}

// L^{-1} of the Cholesky factor A = L L^T of an n x n symmetric positive
// definite matrix (row-major, lower triangle read and destroyed) by G threads
// with barrier `id`; g is the thread's index in the group.  Li (n x n,
// row-major) receives L^{-1}, its upper triangle zero; rs is scratch of n and
// receives 1 / L_ii (column c of A is left as L_ic / rs_c, i > c, and the pivot
// L_cc^2).  ld: row stride of A and Li (0: n).
// Returns false, in every thread of the group, if a pivot is not positive
// (the result is then void).  n <= 20 with G = 128, n <= 40 with G = 256.
//
// LDL^T with the inverse carried along: at step j the entry (i, c) of row
// i > j, c in 0 .. i, is the trailing matrix for c > j and the unit inverse
// for c <= j, and both are updated by -a_ij y_c with y_c = (entry c of row j
// of L^T or L^{-1}) / d_j; the square roots follow at the end, all at once.
// The group's first warp runs one step ahead: it updates column j + 1 of the
// matrix and row j + 1 of the inverse (a lane per entry), and so has the next
// pivot, its reciprocal and the next y while the other warps update the rest,
// one multiply-add per entry.  A step is that warp's chain (a multiply-add,
// the reciprocal, a multiplication) and one barrier.  With the reciprocal and
// the products a_ij / d_j formed by every thread a 32 x 32 block took 36 us of
// FP64 issue; a Cholesky by one warp followed by the inverse, a column per
// lane, was a chain of several hundred FP64 instructions.
template <int G>
__device__ bool group_chol_inverse(double* A, double* Li, double* rs, int n, int g, int id, int ld = 0) {
  if (ld == 0) ld = n;
  __shared__ double s_y[3][2][40];  // one per barrier id (0, or 1 and 2)
  double(*ys)[40] = s_y[id];
  constexpr int kItems = G == 128 ? 3 : 4;       // entries (i, c), c <= i, per thread of the other warps
  constexpr int kT = G - 32;
  static_assert(kItems * (G - 32) >= (G == 128 ? 210 : 820), "entries per thread");
  int ri[kItems], ci[kItems];
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const int e = g < 32 ? 900 : g - 32 + kT * u;
    int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= e) ++i;
    while (i * (i + 1) / 2 > e) --i;
    ri[u] = i;
    ci[u] = e - i * (i + 1) / 2;
    if (i < n) {
      Li[i * ld + ci[u]] = i == ci[u] ? 1.0 : 0.0;
      if (i != ci[u]) Li[ci[u] * ld + i] = 0.0;
    }
  }
  group_sync<G>(id);
  bool ok = true;
  for (int j = -1; j < n - 1; ++j) {
    if (g < 32) {
      const int p = j + 1;  // the next pivot
      double val[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = g + 32 * h;
        val[h] = 0.0;
        if (c < n && h * 32 < n) {
          double* at = c >= p ? A + c * ld + p : Li + p * ld + c;
          val[h] = *at;
          if (j >= 0) {
            const double f = c >= p ? A[c * ld + j] : A[p * ld + j];
            val[h] -= f * ys[j & 1][c >= p ? p : c];
            *at = val[h];
          }
        }
      }
      double d = __shfl_sync(0xffffffffu, p < 32 ? val[0] : val[1], p & 31);
      if (!(d > 0.0)) {
        ok = false;
        d = 1.0;
      }
      const double r = rcp_nr(d);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = g + 32 * h;
        if (c < n && h * 32 < n) ys[p & 1][c] = c == p ? r : val[h] * r;
      }
    } else if (j >= 0) {
      const double* y = ys[j & 1];
#pragma unroll
      for (int u = 0; u < kItems; ++u) {
        const int i = ri[u], c = ci[u];
        if (i > j + 1 && i < n && c != j + 1) {
          double* at = (c > j ? A : Li) + i * ld + c;
          *at -= A[i * ld + j] * y[c];
        }
      }
    }
    group_sync<G>(id);
  }
  if (g < 32) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = g + 32 * h;
      if (c < n) {
        const double d = A[c * ld + c];
        rs[c] = d > 0.0 ? rsqrt_nr(d) : 1.0;
      }
    }
    __syncwarp();
    if (!ok && g == 0) rs[0] = -1.0;  // the verdict, for every thread
  }
  group_sync<G>(id);
  ok = __double2hiint(rs[0]) > 0;
#pragma unroll
  for (int u = 0; u < kItems; ++u)
    if (ri[u] < n) Li[ri[u] * ld + ci[u]] *= rs[ri[u]];
  group_sync<G>(id);
  return ok;
}

// Symmetric eigendecomposition in FP32 by parallel (round-robin ordered)
// two-sided Jacobi, n * n <= 256 kI, by all 256 threads of the CTA: on return the
// diagonal of *A holds the eigenvalues (unsorted) and the columns of *Q the
// eigenvectors.  A2 and Q2 are second buffers; the pointers come back swapped
// as the last round left them.  Every warp forms all rotations of a round in
// its own lanes, a thread updates one or two entries of A (four old entries,
// two rotations) and of Q from one buffer into the other, so a round costs
// one barrier.  A sweep in which no pair exceeded 1e-6 of its diagonal ends
// it.  (One warp updating rows, then columns, in place took 53 us for n = 10.)
__device__ __forceinline__ void jacobi_role(int i, int r, int m, int np, int& pair, int& partner) {
  auto mod = [&](int x) { return x >= m - 1 ? x - (m - 1) : x; };
  if (i == 0) {
    pair = 0;
    partner = 1 + mod(m - 2 + r);
    return;
  }
  int t = i - 1 - r;
  if (t < 0) t += m - 1;
  if (t <= np - 2) {
    pair = t + 1;
    partner = 1 + mod(m - 2 - pair + r);
  } else {
    pair = m - 2 - t;
    partner = pair == 0 ? 0 : 1 + mod(pair - 1 + r);
  }
}

template <int kI>
__device__ __forceinline__ void blk_jacobi_f32(float*& A, float*& A2, float*& Q, float*& Q2, int n) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int m = n + (n & 1), np = m / 2;
  int ei[kI], ej[kI];
#pragma unroll
  for (int u = 0; u < kI; ++u) {
    const int e = tid + 256 * u;
    ei[u] = e / n;
    ej[u] = e - ei[u] * n;
    if (ei[u] < n) Q[e] = ei[u] == ej[u] ? 1.f : 0.f;
  }
  __syncthreads();
  for (int sweep = 0; sweep < 12; ++sweep) {
    bool big = false;
    for (int r = 0; r < m - 1; ++r) {
      float c = 1.f, s = 0.f;
      if (lane < np) {
        const int x = lane - 1 + r, y = m - 2 - lane + r;
        const int a = lane == 0 ? 0 : 1 + (x >= m - 1 ? x - (m - 1) : x);
        const int b = 1 + (y >= m - 1 ? y - (m - 1) : y);
        const int p = min(a, b), q = max(a, b);
        if (q < n) {
          const float apq = A[p * n + q], app = A[p * n + p], aqq = A[q * n + q];
          const float w = fabsf(app * aqq);
          if (apq * apq > 1e-16f * w) {
            big = apq * apq > 1e-12f * w || big;
            const float tau = (aqq - app) / (2.f * apq);
            const float t = __fdividef(tau >= 0.f ? 1.f : -1.f, fabsf(tau) + sqrtf(1.f + tau * tau));
            c = rsqrtf(1.f + t * t);
            s = t * c;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kI; ++u) {
        const bool in = ei[u] < n;
        if (n * n <= 256 * u) break;  // uniform
        const int i = in ? ei[u] : 0, j = in ? ej[u] : 0;
        int pi, qi, pj, qj;
        jacobi_role(i, r, m, np, pi, qi);
        jacobi_role(j, r, m, np, pj, qj);
        const float c_i = __shfl_sync(0xffffffffu, c, pi), c_j = __shfl_sync(0xffffffffu, c, pj);
        float s_i = __shfl_sync(0xffffffffu, s, pi), s_j = __shfl_sync(0xffffffffu, s, pj);
        if (i < qi) s_i = -s_i;
        if (j < qj) s_j = -s_j;
        if (qi >= n) qi = i;  // a bye (its rotation is the identity)
        if (qj >= n) qj = j;
        if (in) {
          const float x0 = c_i * A[i * n + j] + s_i * A[qi * n + j];
          const float x1 = c_i * A[i * n + qj] + s_i * A[qi * n + qj];
          A2[i * n + j] = c_j * x0 + s_j * x1;
          Q2[i * n + j] = c_j * Q[i * n + j] + s_j * Q[i * n + qj];
        }
      }
      __syncthreads();
      float* t = A;
      A = A2;
      A2 = t;
      t = Q;
      Q = Q2;
      Q2 = t;
    }
    // every warp formed the same rotations: the verdict is uniform
    if (!__any_sync(0xffffffffu, big)) break;
  }
}

// Eigendecomposition of a symmetric FP64 matrix T (n x n, n <= 40, row-major
// in shared memory, unchanged) by all 256 threads: eigenvalues descending in
// lam, eigenvectors in the columns of Q.  W is scratch of 3 n^2 doubles.
//
// FP32 Jacobi gives vectors good to ~1e-6, which two steps of the refinement
// of Ogita and Aishima (Iterative refinement for symmetric eigenvalue
// decomposition, 2018; quadratically convergent, products of n x n matrices
// only) bring to FP64: with R = I - Q^T Q, S = Q^T T Q and lam_j = S_jj /
// (1 - R_jj), Q += Q E, E_ij = (S_ij + lam_j R_ij) / (lam_j - lam_i) for
// separated pairs and R_ij / 2 for the others.  The result is accepted when
// Q^T T Q is diagonal to 1e-13 of its diagonal; clusters that the refinement
// leaves coupled are finished by FP64 Jacobi sweeps on that nearly diagonal
// matrix.  (FP64 Jacobi from the start is bound by the FP64 rate of one SM,
// divisions and square roots above all: 390 us for n = 20.)
template <typename F>
__device__ void blk_eig(const double* T, double* Q, double* lam, int n, double* W, F jacobi64) {
  const int tid = threadIdx.x, nn = n * n;
  double* S = W;
  double* E = W + nn;
  double* Y = W + 2 * nn;
  __shared__ double s_red[2][8];
  __shared__ double s_lam[40];
  __shared__ int s_rank[40];
  {
    float* A = reinterpret_cast<float*>(W);
    float *A2 = A + nn, *Qf = A2 + nn, *Q2 = Qf + nn;
    // scaled by the largest diagonal entry into the FP32 range
    double mx = 0;
    for (int i = 0; i < n; ++i) mx = fmax(mx, fabs(T[i * n + i]));
    const double inv = mx > 0 ? 1.0 / mx : 1.0;
    for (int e = tid; e < nn; e += 256) A[e] = (float)(T[e] * inv);
    if (nn <= 512) blk_jacobi_f32<2>(A, A2, Qf, Q2, n);
    else blk_jacobi_f32<7>(A, A2, Qf, Q2, n);
    for (int e = tid; e < nn; e += 256) Q[e] = (double)Qf[e];
  }
  __syncthreads();
  auto form = [&]() {  // Y = T Q; S = Q^T Y
    for (int e = tid; e < nn; e += 256) {
      const int i = e / n, j = e - i * n;
      double s = 0;
#pragma unroll 4
      for (int q = 0; q < n; ++q) s += T[i * n + q] * Q[q * n + j];
      Y[e] = s;
    }
    __syncthreads();
    for (int e = tid; e < n * (n + 1) / 2; e += 256) {
      int j = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
      while ((j + 1) * (j + 2) / 2 <= e) ++j;
      while (j * (j + 1) / 2 > e) --j;
      const int i = e - j * (j + 1) / 2;
      double s = 0;
#pragma unroll 4
      for (int q = 0; q < n; ++q) s += Q[q * n + i] * Y[q * n + j];
      S[i * n + j] = s;
      S[j * n + i] = s;
    }
    __syncthreads();
  };
  // sums of squares of S off and on the diagonal
  auto norms = [&](double& off, double& dg) {
    double o = 0, d = 0;
    for (int e = tid; e < nn; e += 256) {
      const double v = S[e] * S[e];
      if (e / n == e % n) d += v;
      else o += v;
    }
    o = warp_sum(o);
    d = warp_sum(d);
    if ((tid & 31) == 0) {
      s_red[0][tid >> 5] = o;
      s_red[1][tid >> 5] = d;
    }
    __syncthreads();
    off = dg = 0;
    for (int q = 0; q < 8; ++q) {
      off += s_red[0][q];
      dg += s_red[1][q];
    }
    __syncthreads();
  };
  double off = 0, dg = 0;
  for (int step = 0; step < 2; ++step) {
    form();
    norms(off, dg);
    // R = I - Q^T Q in place of Y
    for (int e = tid; e < nn; e += 256) {
      const int i = e / n, j = e - i * n;
      double s = i == j ? 1.0 : 0.0;
#pragma unroll 4
      for (int q = 0; q < n; ++q) s -= Q[q * n + i] * Q[q * n + j];
      Y[e] = s;
    }
    __syncthreads();
    if (tid < n) s_lam[tid] = S[tid * n + tid] / (1.0 - Y[tid * n + tid]);
    __syncthreads();
    // pairs closer than the coupling are left to the orthogonalization
    const double delta = 2.0 * (sqrt(off) + 1e-15 * sqrt(dg));
    for (int e = tid; e < nn; e += 256) {
      const int i = e / n, j = e - i * n;
      const double gap = s_lam[j] - s_lam[i];
      E[e] = (i != j && fabs(gap) > delta) ? (S[e] + s_lam[j] * Y[e]) / gap : 0.5 * Y[e];
    }
    __syncthreads();
    for (int e = tid; e < nn; e += 256) {  // Y = Q + Q E
      const int i = e / n, j = e - i * n;
      double s = Q[e];
#pragma unroll 4
      for (int q = 0; q < n; ++q) s += Q[i * n + q] * E[q * n + j];
      Y[e] = s;
    }
    __syncthreads();
    for (int e = tid; e < nn; e += 256) Q[e] = Y[e];
    __syncthreads();
  }
  form();
  norms(off, dg);
  if (!(off <= 1e-26 * dg)) {
    // coupled clusters: S = J diag J^T by FP64 Jacobi, Q <- Q J
    jacobi64(S, E, s_lam, n);  // S destroyed, J in E
    __syncthreads();
    for (int e = tid; e < nn; e += 256) {
      const int i = e / n, j = e - i * n;
      double s = 0;
      for (int q = 0; q < n; ++q) s += Q[i * n + q] * E[q * n + j];
      Y[e] = s;
    }
  } else {
    if (tid < n) s_lam[tid] = S[tid * n + tid];
    for (int e = tid; e < nn; e += 256) Y[e] = Q[e];
  }
  __syncthreads();
  // descending order (ties keep the lower index first)
  if (tid < n) {
    const double l = s_lam[tid];
    int r = 0;
    for (int j = 0; j < n; ++j) {
      const double o = s_lam[j];
      if (o > l || (o == l && j < tid)) ++r;
    }
    s_rank[tid] = r;
    lam[r] = l;
  }
  __syncthreads();
  for (int e = tid; e < nn; e += 256) Q[(e / n) * n + s_rank[e % n]] = Y[e];
  __syncthreads();
}

}  // namespace gbcca
