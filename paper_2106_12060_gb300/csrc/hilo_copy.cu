// BF16 hi/lo copy of FP32 data for the tensor-core pass (Sec. 4.2 gradient
// and Sec. 5.1-5.2 for the products the pass forms; Cor. 4.6 and Cor. 5.6
// for their one read of the data per iteration).
//
// When FP32 data is bound to a plan, each view Z is stored once more as a
// row-interleaved BF16 matrix of 2n rows: row 2i = bf16(z_i), row 2i + 1 =
// bf16(z_i - bf16(z_i)).  The two rows of a data row sum to it within 2^-17
// relative per element (z in [2^e, 2^(e+1)): |z - hi| <= 2^(e-8), and
// rounding the remainder to 8 bits errs by at most 2^(e-17)), and they take
// the 4 bytes per element of the FP32 data.  For FDA the copy is made of the
// class-centred rows Xhat = X - M[y] (Sec. 5.1), so that the pass needs no
// class-mean correction: S_w Phi = Xhat^T (Xhat Phi).  Products of BF16
// operands are exact in FP32, so the pass (pass_tc.cu) computes the products
// of this fixed representation with FP32 accumulation; its epilogue adds the
// two product rows of each data row.
#include <cuda_bf16.h>

#include "common.cuh"
#include "plan.h"

namespace gbcca {

namespace {

// RN to bf16 of s + e (|e| at most half an ulp of s): e only matters when s
// lies halfway between two bf16 values.
__device__ __forceinline__ uint32_t bf16_bits(float s, float e) {
  const uint32_t u = __float_as_uint(s);
  if ((u & 0xffffu) == 0x8000u && e != 0.f) return (u >> 16) + ((e > 0.f) == (s > 0.f) ? 1u : 0u);
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(s));
}
__device__ __forceinline__ float bf16_value(uint32_t b) { return __uint_as_float(b << 16); }
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float t = s - a;
  e = (a - (s - t)) + (b - t);
}

// Row i of the data (FDA: minus its class mean) goes to rows 2i (hi) and
// 2i + 1 (lo) of the copy, leading dimension ldo (a multiple of 8).
//
// Memory bound: 4 bytes read and 4 written per element.  In FP64 (two
// conversions and two subtractions per element) it was bound by the FP64
// rate, about two operations per clock and SM: 1594 us for 300000 x (384 + 200),
// now about 210 us, near the copy rate of memory.
// Uncentred data need no FP64 at all: z - bf16(z) is exact in FP32.  The
// class means are float pairs (mh + ml = the FP64 mean to 2^-48), z - mh is
// taken with its rounding error, and both roundings to bf16 use the
// remainder on ties.  The centred value is within 2^-48 |m|, and never further
// than 2^-24 of itself, from FP64's; rounded to the copy's 17 bits, none of 4e6
// pairs differed from FP64 centring for means of up to ten deviations, one in
// 35000 at 1e4 and one in 700 at 1e6.
// A CTA takes `rows` whole rows as 4-column chunks, kChunks chunks of a thread
// in flight; kVec: 16-byte loads (row starts and stride 16-byte aligned), a
// ragged last chunk by element (nothing past a row's d columns is read).
constexpr int kChunks = 4;
template <bool kVec, bool kCentre>
__global__ void __launch_bounds__(256) hilo_copy_kernel(const float* __restrict__ Z, int64_t ld, int64_t n, int d,
                                                        int rows, const int32_t* __restrict__ y,
                                                        const float* __restrict__ mh, const float* __restrict__ ml,
                                                        int ldm, __nv_bfloat16* __restrict__ out, int64_t ldo) {
  const int nch = (d + 3) >> 2;
  const int64_t i0 = (int64_t)blockIdx.x * rows;
  const int nr = (int)min((int64_t)rows, n - i0);
  const int total = nr * nch;
  for (int base = threadIdx.x; base < total; base += 256 * kChunks) {
    float4 z[kChunks];
    int row[kChunks], col[kChunks];
#pragma unroll
    for (int u = 0; u < kChunks; ++u) {
      const int e = base + 256 * u;
      row[u] = e / nch;
      col[u] = 4 * (e - row[u] * nch);
      z[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (e < total) {
        const float* src = Z + (i0 + row[u]) * ld + col[u];
        if (kVec && col[u] + 4 <= d) {
          z[u] = __ldcs(reinterpret_cast<const float4*>(src));
        } else {
          z[u].x = src[0];
          if (col[u] + 1 < d) z[u].y = src[1];
          if (col[u] + 2 < d) z[u].z = src[2];
          if (col[u] + 3 < d) z[u].w = src[3];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kChunks; ++u) {
      if (base + 256 * u >= total) continue;
      const int64_t i = i0 + row[u];
      float v[4] = {z[u].x, z[u].y, z[u].z, z[u].w};
      float r[4] = {0.f, 0.f, 0.f, 0.f};
      if (kCentre) {
        const int64_t m = (int64_t)y[i] * ldm + col[u];
        const float4 a = *reinterpret_cast<const float4*>(mh + m), b = *reinterpret_cast<const float4*>(ml + m);
        const float h[4] = {a.x, a.y, a.z, a.w}, l[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float t, e;
          two_sum(v[q], -h[q], t, e);
          two_sum(t, e - l[q], v[q], r[q]);
        }
      }
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        hi[q] = bf16_bits(v[q], r[q]);
        float w = v[q] - bf16_value(hi[q]), we = 0.f;  // exact
        if (kCentre) two_sum(w, r[q], w, we);
        lo[q] = bf16_bits(w, we);
      }
      const uint2 H = make_uint2(hi[0] | (hi[1] << 16), hi[2] | (hi[3] << 16));
      const uint2 L = make_uint2(lo[0] | (lo[1] << 16), lo[2] | (lo[3] << 16));
      *reinterpret_cast<uint2*>(out + 2 * i * ldo + col[u]) = H;
      *reinterpret_cast<uint2*>(out + (2 * i + 1) * ldo + col[u]) = L;
    }
  }
}

// The class means as float pairs, rows padded to ldm (a multiple of 4) with zeros.
__global__ void split_means_kernel(const double* __restrict__ means, int l, int d, int ldm, float* __restrict__ mh,
                                   float* __restrict__ ml) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= l * ldm) return;
  const int c = e / ldm, j = e - c * ldm;
  const double m = j < d ? means[(int64_t)c * d + j] : 0.0;
  const float h = (float)m;
  mh[e] = h;
  ml[e] = (float)(m - (double)h);
}

int means_ld(const Plan& p) { return (p.v[0].d + 3) / 4 * 4; }

// Shapes the tensor-core pass streams through the copy: FP32 CCA of any
// shape the library accepts (d <= 1024, k <= 20); FP32 FDA with d <= 1024
bool hilo_shape_ok(const Plan& p) {
  if (p.dtype != GBCCA_FP32) return false;
  return p.kind == kCCA || p.v[0].d <= 1024;
}

}  // namespace

int hilo_alloc(Plan& p) {
  p.ts_ready = false;
  if (!p.opt.tensor_cores || !hilo_shape_ok(p)) return GBCCA_OK;
  for (int v = 0; v < p.nviews; ++v) {
    // rows padded to 16 bytes (the TMA row stride)
    const int64_t ldo = (p.v[v].d + 7) / 8 * 8;
    p.ts_ld[v] = ldo;
    void* t = nullptr;
    if (counted_malloc(&t, sizeof(__nv_bfloat16) * (size_t)2 * p.n * ldo) != cudaSuccess) {
      cudaGetLastError();
      set_last_error("allocation of the BF16 hi/lo copy of the data failed");
      return GBCCA_ERR_OOM;
    }
    p.ts_copy[v] = static_cast<__nv_bfloat16*>(t);
  }
  if (p.kind == kLDA) {
    void* t = nullptr;
    if (counted_malloc(&t, sizeof(float) * (size_t)2 * p.l * means_ld(p)) != cudaSuccess) {
      cudaGetLastError();
      set_last_error("allocation of the class means' float pairs failed");
      return GBCCA_ERR_OOM;
    }
    p.means_df = static_cast<float*>(t);
  }
  return GBCCA_OK;
}

// Makes the copies of the bound data (FDA: of the class-centred rows, after
// the class statistics).
int hilo_prepare(Plan& p, cudaStream_t st) {
  p.ts_ready = false;
  if (!p.opt.tensor_cores || p.ts_copy[0] == nullptr) return GBCCA_OK;
  const bool fda = p.kind == kLDA;
  const int ldm = means_ld(p);
  float* ml = p.means_df + (fda ? (int64_t)p.l * ldm : 0);
  if (fda) {
    split_means_kernel<<<ceil_div(p.l * ldm, 256), 256, 0, st>>>(p.means, p.l, p.v[0].d, ldm, p.means_df, ml);
    GB_CHECK_LAUNCH();
  }
  for (int v = 0; v < p.nviews; ++v) {
    const int d = p.v[v].d;
    const float* Z = static_cast<const float*>(p.v[v].Z);
    const bool vec = p.v[v].ld % 4 == 0 && (reinterpret_cast<uintptr_t>(Z) & 15) == 0;
    // rows per CTA: about two rounds of the threads' chunks
    const int rows = std::max(1, 2 * 256 * kChunks / ((d + 3) / 4));
    auto kern = fda ? (vec ? hilo_copy_kernel<true, true> : hilo_copy_kernel<false, true>)
                    : (vec ? hilo_copy_kernel<true, false> : hilo_copy_kernel<false, false>);
    kern<<<ceil_div(p.n, rows), 256, 0, st>>>(Z, p.v[v].ld, p.n, d, rows, p.labels, p.means_df, ml, ldm, p.ts_copy[v],
                                              p.ts_ld[v]);
    GB_CHECK_LAUNCH();
  }
  p.ts_ready = true;
  return GBCCA_OK;
}

}  // namespace gbcca
