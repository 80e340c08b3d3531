// The per-iteration data pass in FP64 on CUDA cores (FP64 data, and the
// FP64 Grams of the final refinement of FP32/BF16 plans; same products as
// pass.cu: W = [X Phi_x, Y Phi_y], Z^T W, W^T W; FDA with the class-mean rows
// subtracted, Sec. 4.2 and 5.1-5.2).
//
// What bounds these kernels is the FP64 rate: a warp-wide multiply-add
// occupies its scheduler for 64 cycles whether its lanes are used or not, and
// an SM completes one every 19, so four or five warps saturate an SM and the
// serial chain of one output costs no more than independent ones.  So every
// output is one thread's chain in the order of its terms (bitwise
// reproducible, and independent of the shapes of tiles and grids), lanes hold
// outputs only, and small inputs are spread over all SMs: the products of
// 2000 x 90 data with 10 columns per view run on 125 CTAs of 16 rows, where
// 64-row tiles with columns padded to a multiple of 8 took 55 us on 32 SMs
// (98 us for the whole call; 31 us now).  One refinement pass over 100000
// x 784 FP32 with 9 columns is most of what took an LDA solve from 15.2 to
// 14.0 ms.
#include "pass64.h"

namespace gbcca {

namespace {

constexpr int kJ = 64;      // columns of Z per step of the W kernel
constexpr int kGRows = 64;  // rows of a Gram tile (one chain of its sums)
constexpr int kRows = 32;   // rows per step of the G kernel
constexpr int kFlush = 4;   // G kernel: steps per partial chain
constexpr int kGE = 13;     // Gram entries per thread (80 * 81 / 2 of them at most)
constexpr int kCE = 10;     // class-sum entries per thread (l NC <= 2560)

__device__ __forceinline__ void cp_async8(double* dst, const double* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(ok ? 8u : 0u)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// W: thread (r, c) owns entry (row0 + r, c) of W, R rows per CTA (16, or 8
// beyond 40 columns).  Z (widened) and Phi are staged in steps of kJ columns
// of both views, one step ahead of the arithmetic.
template <typename Tin, int R>
__global__ void __launch_bounds__(R == 16 ? 640 : 1024) pass_w64_kernel(Pass64 a) {
  if (a.done != nullptr && *a.done) return;
  constexpr int kZ = 2 * R * kJ / 256;  // elements of Z per thread and step (at least 256 threads)
  extern __shared__ __align__(16) double sm64[];
  const int NC = a.NC, kc = a.kc, nt = blockDim.x, tid = threadIdx.x;
  double* Ps = sm64;                                                 // [2][2 views][kJ][kc]
  double* Zs = Ps + 4 * kJ * kc;                                     // [2][2 views][R][kJ + 1]
  const int64_t row0 = blockIdx.x * (int64_t)R;
  const int r = tid / NC, c = tid - r * NC, v = c >= kc ? 1 : 0, cv = c - v * kc;
  const bool own = r < R;
  const int d0 = a.d[0], d1 = a.nviews > 1 ? a.d[1] : 0;
  const int ns = (max(d0, d1) + kJ - 1) / kJ;
  Tin zr[kZ];
  auto load = [&](int s) {
    const int j0 = s * kJ;
#pragma unroll
    for (int i = 0; i < kZ; ++i) {
      const int e = tid + nt * i;  // [view][row][column]
      const int ev = e / (R * kJ), er = e / kJ % R, ec = e & (kJ - 1);
      const int64_t row = row0 + er;
      const bool in = ev < a.nviews && e < 2 * R * kJ && row < a.n && j0 + ec < (ev == 0 ? d0 : d1);
      zr[i] = in ? static_cast<const Tin*>(ev == 0 ? a.Z[0] : a.Z[1])[row * (ev == 0 ? a.ld[0] : a.ld[1]) + j0 + ec]
                 : Tin(0.0f);
    }
    double* pb = Ps + (s & 1) * 2 * kJ * kc;
    for (int e = tid; e < a.nviews * kJ * kc; e += nt) {
      const int ev = e / (kJ * kc), f = e - ev * kJ * kc, j = f / kc, q = f - j * kc;
      const double* Phi = ev == 0 ? a.Phi[0] : a.Phi[1];
      const bool ok = j0 + j < (ev == 0 ? d0 : d1);
      cp_async8(pb + e, ok ? Phi + (int64_t)(j0 + j) * a.phistride + q : Phi, ok);
    }
  };
  auto store = [&](int s) {
    double* zb = Zs + (s & 1) * 2 * R * (kJ + 1);
#pragma unroll
    for (int i = 0; i < kZ; ++i) {
      const int e = tid + nt * i;
      if (e < 2 * R * kJ) zb[(e / kJ) * (kJ + 1) + (e & (kJ - 1))] = widen(zr[i]);
    }
  };
  load(0);
  store(0);
  cp_async_wait();
  __syncthreads();
  double acc = 0.0;
  const int dv = v == 0 ? d0 : d1;
  for (int s = 0; s < ns; ++s) {
    if (s + 1 < ns) load(s + 1);
    if (own) {
      const double* zb = Zs + ((s & 1) * 2 * R + v * R + r) * (kJ + 1);
      const double* pb = Ps + ((s & 1) * 2 + v) * kJ * kc + cv;
      const int nj = min(kJ, dv - s * kJ);
#pragma unroll 4
      for (int j = 0; j < nj; ++j) acc += zb[j] * pb[j * kc];
    }
    if (s + 1 < ns) store(s + 1);
    cp_async_wait();
    __syncthreads();
  }
  const int64_t row = row0 + r;
  if (!own || row >= a.n) return;
  if (a.labels != nullptr) acc -= a.Cls[(int64_t)a.labels[row] * NC + c];  // FDA: minus the class mean's row
  a.W[row * NC + c] = acc;
}

// CTAs [0, gctas): W^T W (and the FDA class sums) over tiles of kGRows rows
// (tile b, b + gctas, ...), entries a <= b only (products commute, so the
// mirrored entry is the same number).  The other CTAs: Z^T W of (row chunk,
// kCols columns of Z), a thread per entry (column of Z, column of W) and KQ of
// them, one chain over the chunk's rows per entry, restarted every kFlush
// steps.  kCols = 8 where 32 would leave the SMs with one or two CTAs each (2000
// x 90, 10 columns per view: 16 us of a pass, one SM's two CTAs of 32 columns
// setting the time), 32 otherwise (a CTA copies all of its rows of W).
template <int KQ, int kCols>
__global__ void __launch_bounds__(256) pass_g64_kernel(Pass64 a, int gctas, int chunks, int64_t rows_per_chunk, int nb0,
                                                       int D, double* __restrict__ partG) {
  if (a.done != nullptr && *a.done) return;
  extern __shared__ __align__(16) double sm64[];
  const int NC = a.NC, tid = threadIdx.x;
  if ((int)blockIdx.x < gctas) {
    double* Wt = sm64;  // [kGRows][NC]
    int* ys = reinterpret_cast<int*>(Wt + kGRows * NC);
    const int ne = NC * (NC + 1) / 2;
    const bool cls = a.partCls != nullptr;
    double g_acc[kGE], c_acc[kCE];
#pragma unroll
    for (int i = 0; i < kGE; ++i) g_acc[i] = 0.0;
#pragma unroll
    for (int i = 0; i < kCE; ++i) c_acc[i] = 0.0;
    auto entry = [&](int e, int& x, int& y) {  // e = y (y + 1) / 2 + x, x <= y
      y = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
      while ((y + 1) * (y + 2) / 2 <= e) ++y;
      while (y * (y + 1) / 2 > e) --y;
      x = e - y * (y + 1) / 2;
    };
    const int64_t ntiles = (a.n + kGRows - 1) / kGRows;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gctas) {
      const int64_t row0 = tile * kGRows;
      const int nr = (int)min((int64_t)kGRows, a.n - row0);
      for (int e = tid; e < nr * NC; e += 256) cp_async8(Wt + e, a.W + row0 * NC + e, true);
      if (cls && tid < kGRows) ys[tid] = tid < nr ? a.labels[row0 + tid] : -1;
      cp_async_wait();
      __syncthreads();
#pragma unroll
      for (int i = 0; i < kGE; ++i) {
        const int e = tid + 256 * i;
        if (e < ne) {
          int x, y;
          entry(e, x, y);
          double s = 0.0;
#pragma unroll 4
          for (int r = 0; r < nr; ++r) s += Wt[r * NC + x] * Wt[r * NC + y];
          g_acc[i] += s;
        }
      }
      if (cls) {
#pragma unroll
        for (int i = 0; i < kCE; ++i) {
          const int e = tid + 256 * i;
          if (e < a.l * NC) {
            const int k = e / NC, c = e - k * NC;
            double s = 0.0;
            for (int r = 0; r < nr; ++r)
              if (ys[r] == k) s += Wt[r * NC + c];
            c_acc[i] += s;
          }
        }
      }
      __syncthreads();
    }
    double* pg = a.partGram + (int64_t)blockIdx.x * NC * NC;
#pragma unroll
    for (int i = 0; i < kGE; ++i) {
      const int e = tid + 256 * i;
      if (e < ne) {
        int x, y;
        entry(e, x, y);
        pg[x * NC + y] = g_acc[i];
        pg[y * NC + x] = g_acc[i];
      }
    }
    if (cls) {
#pragma unroll
      for (int i = 0; i < kCE; ++i) {
        const int e = tid + 256 * i;
        if (e < a.l * NC) a.partCls[(int64_t)blockIdx.x * a.l * NC + e] = c_acc[i];
      }
    }
    return;
  }
  double* Zs = sm64;                          // [2][kRows][kCols + 1]
  double* Ws = Zs + 2 * kRows * (kCols + 1);  // [2][kRows][NC]
  int zc[KQ], wc[KQ];  // this thread's entries: column of Z, column of W
#pragma unroll
  for (int q = 0; q < KQ; ++q) {
    const int e = tid + 256 * q;
    // (lanes along the columns of Z at 32, so that W is broadcast)
    zc[q] = kCols == 32 ? e % kCols : e / NC;
    wc[q] = kCols == 32 ? e / kCols : e - zc[q] * NC;
  }
  const int b = (int)blockIdx.x - gctas, chunk = b % chunks, block = b / chunks;
  const int v = block < nb0 ? 0 : 1;
  const int c0 = kCols * (block - (v == 0 ? 0 : nb0));
  const double* Z = static_cast<const double*>(v == 0 ? a.Z[0] : a.Z[1]);
  const int64_t ld = v == 0 ? a.ld[0] : a.ld[1];
  const int d = v == 0 ? a.d[0] : a.d[1];
  const int64_t r0 = chunk * rows_per_chunk, r1 = min(a.n, r0 + rows_per_chunk);
  const int ns = r1 > r0 ? (int)((r1 - r0 + kRows - 1) / kRows) : 0;
  auto load = [&](int s) {
    const int64_t i0 = r0 + (int64_t)s * kRows;
    double* zb = Zs + (s & 1) * kRows * (kCols + 1);
#pragma unroll
    for (int i = 0; i < kRows * kCols / 256; ++i) {
      const int e = tid + 256 * i, rr = e / kCols, cc = e % kCols;
      const int64_t r = i0 + rr;
      const bool ok = r < r1 && c0 + cc < d;
      cp_async8(zb + rr * (kCols + 1) + cc, ok ? Z + r * ld + c0 + cc : Z, ok);
    }
    double* wb = Ws + (s & 1) * kRows * NC;
    const int nw = (int)min((int64_t)kRows, r1 - i0) * NC;
    for (int e = tid; e < nw; e += 256) cp_async8(wb + e, a.W + i0 * NC + e, true);
  };
  double acc[KQ], acc64[KQ];
#pragma unroll
  for (int q = 0; q < KQ; ++q) acc[q] = acc64[q] = 0.0;
  if (ns > 0) load(0);
  cp_async_wait();
  __syncthreads();
  for (int s = 0; s < ns; ++s) {
    if (s + 1 < ns) load(s + 1);
    if (s > 0 && s % kFlush == 0) {
#pragma unroll
      for (int q = 0; q < KQ; ++q) acc64[q] += acc[q], acc[q] = 0.0;
    }
    const double* zb = Zs + (s & 1) * kRows * (kCols + 1);
    const double* wb = Ws + (s & 1) * kRows * NC;
    const int nr = (int)min((int64_t)kRows, r1 - r0 - (int64_t)s * kRows);
#pragma unroll 2
    for (int r = 0; r < nr; ++r) {
#pragma unroll
      for (int q = 0; q < KQ; ++q)
        if (tid + 256 * q < kCols * NC) acc[q] += zb[r * (kCols + 1) + zc[q]] * wb[r * NC + wc[q]];
    }
    cp_async_wait();
    __syncthreads();
  }
  double* out = partG + ((int64_t)chunk * D + (v == 0 ? 0 : a.d[0])) * NC;
#pragma unroll
  for (int q = 0; q < KQ; ++q)
    if (tid + 256 * q < kCols * NC && c0 + zc[q] < d) out[(int64_t)(c0 + zc[q]) * NC + wc[q]] = acc64[q] + acc[q];
}

template <typename Tin, int R>
int launch_w64(const Pass64& a, cudaStream_t st) {
  const size_t smem = sizeof(double) * (4 * kJ * (size_t)a.kc + 4 * R * (kJ + 1));
  auto kern = pass_w64_kernel<Tin, R>;
  GB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int threads = std::max(256, (R * a.NC + 31) / 32 * 32);
  kern<<<ceil_div(a.n, R), threads, smem, st>>>(a);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

template <typename Tin>
int w64(const Pass64& a, cudaStream_t st) {
  return a.NC <= 40 ? launch_w64<Tin, 16>(a, st) : launch_w64<Tin, 8>(a, st);
}

template <int KQ, int kCols>
int launch_g64(const Pass64& a, int gctas, int chunks, int D, double* partG, cudaStream_t st) {
  const size_t gram = sizeof(double) * kGRows * a.NC + sizeof(int) * kGRows;
  const size_t stage = sizeof(double) * (2 * kRows * (kCols + 1) + 2 * (size_t)kRows * a.NC);
  const size_t smem = std::max(gram, stage);
  const int nb0 = ceil_div(a.d[0], kCols), nb = nb0 + (a.nviews > 1 ? ceil_div(a.d[1], kCols) : 0);
  auto kern = pass_g64_kernel<KQ, kCols>;
  GB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int blocks = partG == nullptr ? 0 : chunks * nb;
  kern<<<gctas + blocks, 256, smem, st>>>(a, gctas, std::max(1, chunks), (a.n + chunks - 1) / chunks, nb0, D, partG);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

}  // namespace

int pass64(const Pass64& a, int dtype, int gctas, int chunks, int D, double* partG, cudaStream_t st) {
  switch (dtype) {
    case GBCCA_FP64: GB_TRY(w64<double>(a, st)); break;
    case GBCCA_FP32: GB_TRY(w64<float>(a, st)); break;
    default: GB_TRY(w64<__nv_bfloat16>(a, st));
  }
  const int blocks32 = chunks * (ceil_div(a.d[0], 32) + (a.nviews > 1 ? ceil_div(a.d[1], 32) : 0));
  if (partG != nullptr && blocks32 < 4 * 152) {
    switch (ceil_div(a.NC, 32)) {
      case 1: return launch_g64<1, 8>(a, gctas, chunks, D, partG, st);
      case 2: return launch_g64<2, 8>(a, gctas, chunks, D, partG, st);
      default: return launch_g64<3, 8>(a, gctas, chunks, D, partG, st);
    }
  }
  switch (ceil_div(a.NC, 8)) {
    case 1: return launch_g64<1, 32>(a, gctas, chunks, D, partG, st);
    case 2: return launch_g64<2, 32>(a, gctas, chunks, D, partG, st);
    case 3: return launch_g64<3, 32>(a, gctas, chunks, D, partG, st);
    case 4: return launch_g64<4, 32>(a, gctas, chunks, D, partG, st);
    case 5: return launch_g64<5, 32>(a, gctas, chunks, D, partG, st);
    case 6: return launch_g64<6, 32>(a, gctas, chunks, D, partG, st);
    case 7: return launch_g64<7, 32>(a, gctas, chunks, D, partG, st);
    case 8: return launch_g64<8, 32>(a, gctas, chunks, D, partG, st);
    case 9: return launch_g64<9, 32>(a, gctas, chunks, D, partG, st);
    default: return launch_g64<10, 32>(a, gctas, chunks, D, partG, st);
  }
}

}  // namespace gbcca
