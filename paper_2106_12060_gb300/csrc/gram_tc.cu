// Grams of sketched views on the tensor cores (tcgen05 + TMA, sm_103a), with
// about the error of FP64 sums: C = A^T B for the FP64 sketches A (s x d1)
// and B (s x d2) of FP32/BF16 plans (Alg. 1 steps 2-4, Alg. 2 step 3).
//
// Method (error-free splitting for matrix products: Ozaki, Ogita, Oishi, Rump,
// Numer. Algorithms 59, 2012): every column is scaled by a power of two to at
// most 1 and rounded to 55 bits, x = sum_t d_t 2^(-7 - 8 t) with seven integer
// digits |d_t| <= 128, each exact in BF16.  Products of digits at most 2^14,
// summed over at most 7 pairs (t, u) of a level t + u = l and kWindow = 128
// rows, stay below 2^24, so the FP32 accumulators of the 28 MMAs per K step
// (levels 0 .. 6) hold exact integers.  After every window the epilogue adds
// them, shifted by their levels, into one 64-bit integer per entry in units of
// 2^-50, up to kMaxRows rows per CTA (coarser units serve longer ranges).
//
// Error of an entry, in units of the product of its columns' largest entries:
// at most 2^-55 a row from the digits' rounding, 6 x 2^-56 a row from the levels
// left out (t + u >= 7), 2^-51 a window from the units (2^(drop - 51) with coarser
// ones): s 2^-53 and a thirty-second of it.  So it is bounded by the columns'
// norms, as an FP64 sum's is, not by the sum of an entry's own |terms|: where
// outlier rows dwarf the rest of a column, entries among the rest keep fewer
// bits than the double-float sums before gave them (2^-44 of each term).  For the
// factorization, whose error is relative to the columns' norms too, that does
// not matter.
//
// Bound by MMA issue (one thread issues an MMA about every 50 cycles; 56 per
// 32 rows) and the windows' epilogue, which the single set of 7 x 64
// accumulator columns does not hide.  FP32 double-float arithmetic is bound by
// FP32 issue (12 instructions a term): 690 us for 4096 x (512 + 512) and 370 us
// for each symmetric 512 x 512; 84 and 57 us now, and 26 us for the digits and
// the scaling of each.  Error of R^T R against FP64 over 24 to 1000 columns and
// both sketches, measured: 2.5e-15 of the columns' norms before, 5e-17 now.
#include "tc_ptx.cuh"

namespace gbcca {
namespace gram {

using namespace tc;

constexpr int kSlices = 7;
constexpr int kBox = 4096;                     // 64 columns x 32 rows of one slice
constexpr int kStageRows = 32;
constexpr int kWindow = 128;                   // rows between flushes
constexpr int kMaxRows = 4096;                 // rows of one CTA: |sum| < 2^63 in units of 2^-50
constexpr int kBBytes = kSlices * kBox;        // N = 64
constexpr int kABytes = 2 * kSlices * kBox;    // M = 128
constexpr int kStage = kABytes + kBBytes;
constexpr int kStages = 2;
constexpr int kN = 64;                         // TMEM columns of a level
constexpr int kThreads = 384;                  // producer, issuer, TMEM, spare, 8 epilogue warps
constexpr int kSmem = kStages * kStage + 1024 + 256;
constexpr uint32_t kTmemCols = 512;
static_assert(kSlices * kWindow * (1 << 14) < (1 << 24), "exact FP32 sums of a level");
static_assert(kSlices * kN <= (int)kTmemCols, "accumulators");
static_assert(kStages * kStage + 1280 <= 232448, "shared memory");

// Exponents (biased) at which the FP32 range ends for the entries of a column:
// beyond kMaxExp not finite; below kMinExp every square rounds to zero.
constexpr int kMaxExp = 1150, kMinExp = 948;

// Largest biased exponent of every column (zeroed before); 2047, as for a
// column that is not finite, where the column's squares sum to more than FP32
// holds over one of the row ranges of the double-float form.  The rest of a
// plan (M^{-1} as float pairs above all) has no more range than that, so both
// forms refuse the same sketches.  blockIdx.y: a range of `chunk` rows.
__global__ void __launch_bounds__(1024) col_exp_kernel(const double* __restrict__ A, int64_t s, int d, int64_t chunk,
                                                       int* __restrict__ ex) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, col = blockIdx.x * 32 + lane;
  __shared__ int red_m[32][32];
  __shared__ float red_q[32][32];
  const int64_t r1 = min(s, (int64_t)(blockIdx.y + 1) * chunk);
  int m = 0;
  float q = 0.f;
  if (col < d) {
#pragma unroll 4
    for (int64_t r = blockIdx.y * chunk + w; r < r1; r += 32) {
      const double x = A[r * d + col];
      const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
      const int e = (int)(hi >> 20 & 0x7ff);
      m = max(m, e);
      // |x| to 24 bits, by moving the bits (a conversion runs at the FP64 rate)
      const float a = e > kMaxExp ? INFINITY
                                  : (e < 897 ? 0.f : __uint_as_float((uint32_t)(e - 896) << 23 | (hi & 0xfffff) << 3 | lo >> 29));
      q = fmaf(a, a, q);
    }
  }
  red_m[w][lane] = m;
  red_q[w][lane] = q;
  __syncthreads();
  if (w != 0 || col >= d) return;
  for (int u = 1; u < 32; ++u) {
    m = max(m, red_m[u][lane]);
    q += red_q[u][lane];
  }
  atomicMax(&ex[col], q <= 3.402823466e38f ? m : 2047);
}

// Digits of every entry: slice t at S + t sp dp, rows s .. sp - 1 zero.  Two
// columns per thread; integer arithmetic only (FP64 instructions are slow).
__global__ void __launch_bounds__(256) slice_kernel(const double* __restrict__ A, int64_t s, int64_t sp, int d, int dp,
                                                    const int* __restrict__ ex, uint32_t* __restrict__ S) {
  const int64_t e = blockIdx.x * (int64_t)256 + threadIdx.x;
  const int half = dp / 2;
  if (e >= sp * half) return;
  const int64_t r = e / half;
  const int c = (int)(e - r * half) * 2;
  uint32_t w[kSlices] = {};
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (r >= s || c + u >= d) continue;
    const long long bits = __double_as_longlong(A[r * d + c + u]);
    int be = (int)(bits >> 52) & 0x7ff;
    long long m = bits & 0xfffffffffffffll;
    if (be != 0) m |= 1ll << 52;
    else be = 1;
    // x 2^55 / 2^(E - 1022), rounded to an integer, E the column's exponent
    const int sh = be - max(ex[c + u], 1) + 2;
    long long q = sh >= 0 ? m << sh : (sh > -54 ? (m + (1ll << (-sh - 1))) >> -sh : 0);
    if (bits < 0) q = -q;
#pragma unroll
    for (int t = kSlices - 1; t >= 0; --t) {
      const int dg = t > 0 ? (int)((q + 128) & 255) - 128 : (int)q;
      q = (q - dg) >> 8;
      w[t] |= (__float_as_uint((float)dg) >> 16) << (16 * u);
    }
  }
#pragma unroll
  for (int t = 0; t < kSlices; ++t) S[(t * sp + r) * half + c / 2] = w[t];
}

struct Args {
  int64_t sp;         // rows of a slice (a multiple of kStageRows)
  int64_t kchunk;     // rows per CTA (a multiple of kWindow)
  int d1, d2;
  int sym;            // only the tiles that reach the lower triangle
  int drop;           // sums in units of 2^(drop - 50)
  long long* part;    // [split][d1 x d2]
  int* err;
};

__global__ void __launch_bounds__(kThreads, 1)
gram_tc_kernel(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb, Args a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  struct Bars {
    uint64_t full[kStages], empty[kStages], acc_full, acc_free, final_bar;
    uint32_t tmem;
    volatile int abort_flag;
  };
  Bars* B = reinterpret_cast<Bars*>(smem + kStages * kStage);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // tile (128 columns of A, 64 of B)
  int ti, tj;
  if (a.sym) {  // row block ti holds 2 ti + 2 tiles (fewer at the matrix' edge)
    const int t = blockIdx.x, nb = (a.d2 + 63) / 64;
    ti = (int)((sqrtf(4.f * (float)t + 1.f) - 1.f) * 0.5f);
    while ((ti + 1) * (ti + 2) <= t) ++ti;
    while (ti * (ti + 1) > t) --ti;
    tj = t - ti * (ti + 1);
    if (tj >= nb) return;
  } else {
    const int nb = (a.d2 + 63) / 64;
    ti = blockIdx.x / nb;
    tj = blockIdx.x - ti * nb;
  }
  const int64_t r0 = (int64_t)blockIdx.y * a.kchunk, r1 = min(a.sp, r0 + a.kchunk);
  const int stages = (int)((r1 - r0) / kStageRows);
  auto bar = [](const uint64_t& b) { return smem_u32(&b); };
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(bar(B->full[s]), 1);
      mbar_init(bar(B->empty[s]), 1);
    }
    mbar_init(bar(B->acc_full), 1);
    mbar_init(bar(B->acc_free), 256);
    mbar_init(bar(B->final_bar), 1);
    B->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_proxy_async();
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&B->tmem)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = B->tmem;
  constexpr int kPer = kWindow / kStageRows;  // stages of a window
  const int windows = (stages + kPer - 1) / kPer;

  if (warp == 0 && lane == 0) {
    int u = 0;
    for (; u < stages; ++u) {
      const int slot = u % kStages;
      if (!mbar_wait(bar(B->empty[slot]), ((u / kStages) & 1) ^ 1, &B->abort_flag)) break;
      const uint32_t fb = bar(B->full[slot]), dst = smem_u32(smem + slot * kStage);
      mbar_expect_tx(fb, kStage);
      const int row = (int)r0 + u * kStageRows;
      for (int t = 0; t < kSlices; ++t) {
        const int y = (int)(t * a.sp) + row;
        tma_load_2d(dst + 2 * t * kBox, &ma, 128 * ti, y, fb);
        tma_load_2d(dst + (2 * t + 1) * kBox, &ma, 128 * ti + 64, y, fb);
        tma_load_2d(dst + kABytes + t * kBox, &mb, 64 * tj, y, fb);
      }
    }
    // the copies in flight arrive (bounded) before the CTA leaves
    for (int v = max(0, u - kStages); v < u; ++v) {
      const long long t0 = clock64();
      while (!mbar_try(bar(B->full[v % kStages]), (v / kStages) & 1) && clock64() - t0 < kWaitCycles) {
      }
    }
  } else if (warp == 1 && lane == 0) {
    constexpr uint32_t id = idesc_bf16(128, kN, 1, 1);
    bool ok = true;
    int u = 0;
    for (int w = 0; w < windows && ok; ++w) {
      if (w > 0 && !(ok = mbar_wait(bar(B->acc_free), (w - 1) & 1, &B->abort_flag))) break;
      tc_fence_after();
      const int u1 = min(stages, u + kPer);
      for (const int u0 = u; u < u1; ++u) {
        const int slot = u % kStages;
        if (!(ok = mbar_wait(bar(B->full[slot]), (u / kStages) & 1, &B->abort_flag))) break;
        tc_fence_after();
        const uint64_t ad = sdesc(smem_u32(smem + slot * kStage), kBox, 1024);
        const uint64_t bd = sdesc(smem_u32(smem + slot * kStage + kABytes), kBox, 1024);
        const uint32_t first = u > u0 ? 1u : 0u;
#pragma unroll
        for (int l = 0; l < kSlices; ++l)
#pragma unroll
          for (int t = 0; t <= l; ++t)
#pragma unroll
            for (int q = 0; q < kStageRows / 16; ++q)  // K steps of 16 rows
              mma_bf16(tmem + (uint32_t)(l * kN), ad + (uint64_t)((2 * t * kBox >> 4) + 128 * q),
                       bd + (uint64_t)(((l - t) * kBox >> 4) + 128 * q), id, t + q > 0 ? 1u : first);
        mma_commit(bar(B->empty[slot]));
      }
      if (ok) mma_commit(bar(B->acc_full));
    }
    if (u > 0) {
      mma_commit(bar(B->final_bar));
      const long long t0 = clock64();
      while (!mbar_try(bar(B->final_bar), 0) && clock64() - t0 < kWaitCycles) {
      }
    }
  } else if (warp >= 4) {
    // lane quadrant q: rows 32 q + lane of the tile; the two warps of a
    // quadrant take 32 columns each
    const int q = warp & 3, c0 = 32 * ((warp >> 2) - 1);
    const uint32_t acc = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c0;
    long long T[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) T[c] = 0;
    const long long half = (1ll << a.drop) >> 1;
    bool ok = true;
    for (int w = 0; w < windows; ++w) {
      if (!(ok = __all_sync(0xffffffffu, mbar_wait(bar(B->acc_full), w & 1, &B->abort_flag)))) break;
      tc_fence_after();
#pragma unroll
      for (int g = 0; g < 8; ++g) {
        uint32_t v[kSlices][4];
#pragma unroll
        for (int l = 0; l < kSlices; ++l)
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(v[l][0]), "=r"(v[l][1]), "=r"(v[l][2]), "=r"(v[l][3])
                       : "r"(acc + (uint32_t)(l * kN + 4 * g)));
        tmem_ld_wait();
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          int x[kSlices];
#pragma unroll
          for (int l = 0; l < kSlices; ++l) x[l] = __float2int_rn(__uint_as_float(v[l][c]));
          // units of 2^-50: level l weighs 2^(36 - 8 l)
          const long long low = ((long long)x[5] * 256 + x[6] + 2048) >> 12;
          const long long sum = ((long long)x[0] << 36) + ((long long)x[1] << 28) + ((long long)x[2] << 20) +
                                ((long long)x[3] << 12) + ((long long)x[4] << 4) + low;
          T[4 * g + c] += (sum + half) >> a.drop;
        }
      }
      tc_fence_before();
      mbar_arrive(bar(B->acc_free));
    }
    const int i = 128 * ti + 32 * q + lane;
    if (ok && i < a.d1) {
      long long* out = a.part + ((int64_t)blockIdx.y * a.d1 + i) * a.d2;
#pragma unroll
      for (int c = 0; c < 32; ++c)
        if (64 * tj + c0 + c < a.d2) out[64 * tj + c0 + c] = T[c];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && B->abort_flag) raise_flag(a.err, kFlagTimeout);
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// C = the splits' integers summed (exactly, as high and low words) and scaled
// back, + diag_add on the diagonal.  A column beyond the FP32 range (or not
// finite) makes its entries NaN, and columns whose products vanish in FP32 have
// none here either: the factorization reports both (the second with diag_add =
// 0), and the warm start a cross matrix of zeros.
__global__ void __launch_bounds__(256) gram_scale_kernel(const long long* __restrict__ part, int ks, int d1, int d2,
                                                         const int* __restrict__ ea, const int* __restrict__ eb,
                                                         int sym, int drop, double diag_add, double* __restrict__ C) {
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e >= d1 * d2) return;
  const int i = e / d2, j = e - i * d2;
  const int64_t o = sym && j > i ? (int64_t)j * d2 + i : e;
  long long hi = 0, lo = 0;
  for (int z = 0; z < ks; ++z) {
    const long long t = part[(int64_t)z * d1 * d2 + o];
    hi += t >> 32;
    lo += t & 0xffffffffll;
  }
  hi += lo >> 32;
  lo &= 0xffffffffll;
  const int Ei = max(ea[i], 1), Ej = max(eb[j], 1);
  double x = scalbn(fma((double)hi, 4294967296.0, (double)lo), Ei + Ej - 2 * 1022 - 50 + drop);
  if (Ei > kMaxExp || Ej > kMaxExp) x = __longlong_as_double(0x7ff8000000000000ll);
  if (Ei + Ej < 2 * kMinExp) x = 0.0;
  C[e] = x + (i == j ? diag_add : 0.0);
}

}  // namespace gram

int64_t gram_slice_rows(int64_t s) { return (s + gram::kStageRows - 1) / gram::kStageRows * gram::kStageRows; }
int64_t gram_slices_len(int64_t s, int d) { return gram::kSlices * gram_slice_rows(s) * ((d + 7) / 8 * 8); }

int gram_slice(const double* A, int64_t s, int d, int* ex, __nv_bfloat16* S, int64_t ws_len, cudaStream_t st) {
  const int dp = (d + 7) / 8 * 8;
  const int64_t sp = gram_slice_rows(s), chunk = gram_df_chunk(s, d, ws_len);
  GB_CUDA(cudaMemsetAsync(ex, 0, sizeof(int) * d, st));
  gram::col_exp_kernel<<<dim3(ceil_div(d, 32), ceil_div(s, chunk)), 1024, 0, st>>>(A, s, d, chunk, ex);
  GB_CHECK_LAUNCH();
  gram::slice_kernel<<<ceil_div(sp * (dp / 2), 256), 256, 0, st>>>(A, s, sp, d, dp, ex, reinterpret_cast<uint32_t*>(S));
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

int gram_sliced(const __nv_bfloat16* A, const int* ea, int d1, const __nv_bfloat16* B, const int* eb, int d2, int64_t s,
                double* C, double diag_add, double* ws, int64_t ws_len, int sm_count, int* err, cudaStream_t st) {
  const bool sym = A == B;
  const int64_t sp = gram_slice_rows(s), len = (int64_t)d1 * d2;
  const int rb = ceil_div(d1, 128), cb = ceil_div(d2, 64);
  const int tiles = sym ? rb * (rb + 1) : rb * cb;
  // splits of the rows: about one CTA per SM, whole windows, and partial sums
  // within the workspace
  int64_t ks = std::min<int64_t>(std::max<int64_t>(1, sm_count / tiles), (sp + gram::kWindow - 1) / gram::kWindow);
  ks = std::min(ks, ws_len / len);
  if (ks < 1) {
    set_last_error("gram_sliced: workspace too small");
    return GBCCA_ERR_INVALID_ARG;
  }
  gram::Args a{};
  a.sp = sp;
  a.kchunk = ((sp + ks - 1) / ks + gram::kWindow - 1) / gram::kWindow * gram::kWindow;
  ks = (sp + a.kchunk - 1) / a.kchunk;
  while (a.kchunk > (int64_t)gram::kMaxRows << a.drop) ++a.drop;
  a.d1 = d1;
  a.d2 = d2;
  a.sym = sym ? 1 : 0;
  a.part = reinterpret_cast<long long*>(ws);
  a.err = err;
  CUtensorMap ma, mb;
  GB_TRY(make_tma_map_bf16(&ma, A, gram::kSlices * sp, d1, (d1 + 7) / 8 * 8, gram::kStageRows));
  GB_TRY(make_tma_map_bf16(&mb, B, gram::kSlices * sp, d2, (d2 + 7) / 8 * 8, gram::kStageRows));
  GB_CUDA(cudaFuncSetAttribute(gram::gram_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, gram::kSmem));
  gram::gram_tc_kernel<<<dim3(tiles, (unsigned)ks), gram::kThreads, gram::kSmem, st>>>(ma, mb, a);
  GB_CHECK_LAUNCH();
  gram::gram_scale_kernel<<<ceil_div(len, 256), 256, 0, st>>>(a.part, (int)ks, d1, d2, ea, eb, sym ? 1 : 0, a.drop, diag_add, C);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

}  // namespace gbcca
