// The data pass in two sweeps on the tensor cores (tcgen05 + TMA, sm_103a), for
// plans whose working set does not fit the one-sweep kernel of pass_tc.cu:
// more than 24 columns of Phi per view (k > 12), or a CCA view wider than 512
// columns.  Same products (Sec. 4.2 gradient, Sec. 5.1-5.2 for FDA; Cor. 4.6,
// Cor. 5.6): W = Z Phi, then G = Z^T W, with W kept as bf16 hi + lo parts
// between the sweeps.
//
// Why two sweeps: with wide views the one-sweep kernel needs the columns of a
// row tile on several CTAs, whose partial W must be exchanged before the
// second product, and with many columns its accumulators do not fit and the
// data was read once per group of columns; both stalled it (254 us per group
// for 200000 x (1024 + 256) BF16, 2.0 TB/s, two groups at k = 20).  Here the
// data is read exactly twice at the rate of memory, no CTA waits for another,
// and the work splits evenly whatever the widths of the views:
//
// Sweep 1 (w_kernel): a CTA takes a range of 64-row tiles, four at a time.
//   Every 64-column box of the four (TMA) arrives in a ring slot together with
//   that box of the Phi image (bulk copy from L2; per 128 rows it was 60% as
//   many bytes as the data, and the sweep ran at 138 us for the shape above),
//   M = 128, N = 2h MMAs accumulate W_v (bf16 hi and lo columns of Phi, h
//   each) in TMEM; eight epilogue warps (a row per lane) add hi and lo columns
//   (FP32 data: and the product rows of a hi/lo row pair), split W into bf16
//   hi + lo and store it as the K-major, 128B-swizzled operand of sweep 2, one
//   image of [hi rows | lo rows] x 64 tile rows per 64 rows of data.
// Sweep 2 (g_kernel): a CTA owns a block of at most three 128-column pairs of
//   one view and a range of 64-row tiles: per tile one bulk copy of the W image
//   and two TMA boxes per pair, M = 128 (data columns, MN-major from the same
//   boxes), N = 2 nw, K = 64; G stays in TMEM for at most kChain tiles (the
//   truncation of each step adds up: with ranges of 100 tiles the error was
//   1.15 times the one-sweep kernel's over its 82) and is drained to a partial
//   slab (column-major, as in pass_tc.cu), which tc_post_kernel sums per pair.
//
// Bound by HBM in both sweeps (2 x 513 MB + the W image of 64 MB, which mostly
// stays in L2: 151 us at the copy rate for the shape above; 106 us each, 4.9
// TB/s, and 278 us for the whole call, 579 in 4-CTA clusters).  Every wait is
// bounded in time; on expiry a CTA records an error code, waits (bounded) for
// its own copies and MMAs and frees its TMEM.
#include "pass_two.h"

namespace gbcca {
namespace two {

using namespace tc;

constexpr int kThreads = 384;        // producer, issuer, TMEM, spare, 8 epilogue warps
constexpr int kBox = 8192;           // 64 x 64 BF16
constexpr int kPair = 2 * kBox;      // 128 columns of a 64-row tile
constexpr int kAccW = 80;            // TMEM columns of one W accumulator (128 rows of one view)
constexpr int kUnit = 4;             // 64-row tiles of a unit of sweep 1: two accumulators
constexpr int kBufs = 3;             // TMEM buffers between MMA and epilogue
constexpr int kPart = 4;             // boxes of one accumulation in TMEM
constexpr int kChain = 64;           // 64-row tiles of one accumulation of G in TMEM, if the slabs allow
constexpr int kGroups = 3;           // 16-column groups of Phi (at most 40 columns)
constexpr int kMaxStages = 12;
constexpr int kSmem = 232448;        // dynamic shared memory of one CTA
constexpr uint32_t kTmemCols = 512;

struct Bars {
  uint64_t full[kMaxStages], empty[kMaxStages], acc_full[kBufs], acc_free[kBufs], final_bar;
  uint32_t tmem;
  volatile int abort_flag;
};

// Segment s of this CTA: the instance, its first tile and count, the block and
// slab (sweep 2).
struct View {
  const Inst* I;
  int first, count, block, slab;
};
__device__ __forceinline__ int block_of_cta(const Args& a) {
  int b = 0;
  while (b + 1 < a.nblk && (int)blockIdx.x >= a.cta0[b + 1]) ++b;
  return b;
}
__device__ __forceinline__ int seg_count(const Args& a) {
  return a.insts == nullptr ? a.nseg[block_of_cta(a)] : a.seg_off[blockIdx.x + 1] - a.seg_off[blockIdx.x];
}
__device__ __forceinline__ View seg_view(const Args& a, const Inst* one, int s) {
  View v;
  if (a.insts != nullptr) {
    const Seg g = a.segs[a.seg_off[blockIdx.x] + s];
    v = View{a.insts + g.inst, g.first, g.count, g.block, g.slab};
  } else {
    const int b = block_of_cta(a), n = (a.cta0[b + 1] - a.cta0[b]) * a.nseg[b];  // ranges of the block
    const int i = ((int)blockIdx.x - a.cta0[b]) * a.nseg[b] + s;
    const int t0 = (int)((int64_t)one->ntiles * i / n), t1 = (int)((int64_t)one->ntiles * (i + 1) / n);
    v = View{one, t0, t1 - t0, b, i};
  }
  if (v.I->done != nullptr && *v.I->done) v.count = 0;
  return v;
}

// Common prologue and epilogue of both kernels.
__device__ __forceinline__ uint32_t prologue(Bars* B, int stages, int acc_free_count) {
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(smem_u32(&B->full[s]), 1);
      mbar_init(smem_u32(&B->empty[s]), 1);
    }
    for (int b = 0; b < kBufs; ++b) {
      mbar_init(smem_u32(&B->acc_full[b]), 1);
      mbar_init(smem_u32(&B->acc_free[b]), acc_free_count);
    }
    mbar_init(smem_u32(&B->final_bar), 1);
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
  return B->tmem;
}
__device__ __forceinline__ void epilogue(Bars* B, uint32_t tmem, int* err) {
  __syncthreads();
  if (threadIdx.x == 0 && B->abort_flag) raise_flag(err, kFlagTimeout);
  if ((threadIdx.x >> 5) == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}
// Before the CTA leaves, whether it finished or gave up, the producer waits
// (bounded) for the copies it has issued (`uses` slots in ring order) and the
// issuer for its MMAs.  After a complete run they have all arrived.
__device__ __forceinline__ void drain_copies(Bars* B, int uses, int stages) {
  for (int u = max(0, uses - stages); u < uses; ++u) {
    const long long t0 = clock64();
    while (!mbar_try(smem_u32(&B->full[u % stages]), (u / stages) & 1) && clock64() - t0 < kWaitCycles) {
    }
  }
}
__device__ __forceinline__ void drain_mmas(Bars* B) {
  mma_commit(smem_u32(&B->final_bar));
  const long long t0 = clock64();
  while (!mbar_try(smem_u32(&B->final_bar), 0) && clock64() - t0 < kWaitCycles) {
  }
}

// ------------------------------------------------------------------ sweep 1
// A unit is up to kUnit 64-row tiles of one view: its boxes share one box of
// the Phi image.  Its columns are summed in TMEM in parts of kPart boxes, as in
// the one-sweep kernel (the tensor cores truncate as they accumulate: one chain
// over 1024 columns had 1.15 times the error), each part's accumulators (two
// MMA row groups) in the next of the buffers; the epilogue adds the parts.
__global__ void __launch_bounds__(kThreads, 1) w_kernel(const __grid_constant__ Inst one, Args a) {
  if (a.insts == nullptr && one.done != nullptr && *one.done) return;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int S = a.stages, stage = a.stage_bytes, h = a.h, phib = 2 * h * 128;
  Bars* B = reinterpret_cast<Bars*>(smem + S * stage);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t tmem = prologue(B, S, 256);
  const int nseg = seg_count(a);
  auto bar = [](const uint64_t& b) { return smem_u32(&b); };
  if (warp == 0 && lane == 0) {
    bool ok = true;
    int u = 0;  // ring uses
    for (int s = 0; s < nseg && ok; ++s) {
      const View v = seg_view(a, &one, s);
      const CUtensorMap* map = v.I->map;
      const uint8_t* img = v.I->phi_img;
      const int64_t img_view = v.I->img_view;
      const int nv = v.I->nv, nb0 = (v.I->d[0] + 63) >> 6, nb1 = (v.I->d[1] + 63) >> 6;
      const long long wait = v.I->wait;
      for (int t = 0; t < v.count && ok; t += kUnit) {
        const int m = min(kUnit, v.count - t), row0 = (v.first + t) * 64;
        for (int w = 0; w < nv && ok; ++w) {
          const int nb = w == 0 ? nb0 : nb1;
          const uint8_t* phi = img + w * img_view;
          for (int b = 0; b < nb; ++b, ++u) {
            const int slot = u % S;
            if (!(ok = mbar_wait(bar(B->empty[slot]), ((u / S) & 1) ^ 1, &B->abort_flag, wait))) break;
            const uint32_t fb = bar(B->full[slot]), dst = smem_u32(smem + slot * stage);
            mbar_expect_tx(fb, m * kBox + phib);
            for (int i = 0; i < m; ++i) tma_load_2d(dst + i * kBox, map + w, 64 * b, row0 + 64 * i, fb);
            bulk_g2s(dst + kUnit * kBox, phi + (int64_t)b * phib, phib, fb);
          }
        }
      }
    }
    drain_copies(B, u, S);
  } else if (warp == 1 && lane == 0) {
    const uint32_t id = idesc_bf16(128, 2 * h, 0, 0);
    bool ok = true;
    int u = 0, j = 0;
    for (int s = 0; s < nseg && ok; ++s) {
      const View v = seg_view(a, &one, s);
      const int nv = v.I->nv, nb0 = (v.I->d[0] + 63) >> 6, nb1 = (v.I->d[1] + 63) >> 6;
      const long long wait = v.I->wait;
      for (int t = 0; t < v.count && ok; t += kUnit) {
        const bool both = v.count - t > 2;  // more than one row group
        for (int w = 0; w < nv && ok; ++w) {
          const int nb = w == 0 ? nb0 : nb1;
          for (int b = 0; b < nb && ok; ++j) {  // a part
            const int buf = j % kBufs, b0 = b, b1 = min(nb, b + kPart);
            if (j >= kBufs && !(ok = mbar_wait(bar(B->acc_free[buf]), (j / kBufs - 1) & 1, &B->abort_flag, wait)))
              break;
            tc_fence_after();
            const uint32_t acc = tmem + (uint32_t)(2 * buf * kAccW);
            for (; b < b1; ++b, ++u) {
              const int slot = u % S;
              if (!(ok = mbar_wait(bar(B->full[slot]), (u / S) & 1, &B->abort_flag, wait))) break;
              tc_fence_after();
              const uint64_t ad = sdesc(smem_u32(smem + slot * stage), 16, 1024);
              const uint64_t bd = sdesc(smem_u32(smem + slot * stage + kUnit * kBox), 16, 1024);
#pragma unroll
              for (int q = 0; q < 4; ++q)  // K steps of 16 columns: 32 bytes inside the swizzled rows
                mma_bf16(acc, ad + (uint64_t)(2 * q), bd + (uint64_t)(2 * q), id, (b - b0 | q) != 0 ? 1u : 0u);
              if (both) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                  mma_bf16(acc + kAccW, ad + (uint64_t)((2 * kBox >> 4) + 2 * q), bd + (uint64_t)(2 * q), id,
                           (b - b0 | q) != 0 ? 1u : 0u);
              }
              mma_commit(bar(B->empty[slot]));
            }
            if (ok) mma_commit(bar(B->acc_full[buf]));
          }
        }
      }
    }
    if (u > 0) drain_mmas(B);
  } else if (warp >= 4) {
    const int q = warp & 3, grp = (warp >> 2) - 1;  // row group of the unit
    const int rr = 32 * q + lane, e = rr & 62;      // row within the group; even row of its pair within the tile
    const uint32_t lane_off = (uint32_t)(32 * q) << 16;
    const bool odd = (lane & 1) != 0;
    bool ok = true;
    int j = 0;
    for (int s = 0; s < nseg && ok; ++s) {
      const View v = seg_view(a, &one, s);
      const int ncol = v.I->ncol, nw = v.I->nw, nv = v.I->nv, pair_sum = v.I->pair_sum;
      const int nb0 = (v.I->d[0] + 63) >> 6, nb1 = (v.I->d[1] + 63) >> 6;
      const long long wait = v.I->wait;
      uint8_t* wimg = v.I->wimg + (odd ? nw * 128 : 0);
      for (int t = 0; t < v.count && ok; t += kUnit) {
        const int tile = 2 * grp + (rr >> 6);  // of the unit (uniform over the warp)
        uint8_t* img = wimg + (int64_t)(v.first + t + tile) * (2 * nw * 128);
        for (int w = 0; w < nv && ok; ++w) {
          float x[kGroups][16];
#pragma unroll
          for (int g = 0; g < kGroups; ++g)
#pragma unroll
            for (int c = 0; c < 16; ++c) x[g][c] = 0.f;
          const int parts = ((w == 0 ? nb0 : nb1) + kPart - 1) / kPart;
          for (int p = 0; p < parts; ++p, ++j) {
            const int buf = j % kBufs;
            if (!(ok = __all_sync(0xffffffffu,
                                  mbar_wait(bar(B->acc_full[buf]), (j / kBufs) & 1, &B->abort_flag, wait))))
              break;
            tc_fence_after();
            if (t + tile < v.count) {
              const uint32_t acc = tmem + lane_off + (uint32_t)((2 * buf + grp) * kAccW);
#pragma unroll
              for (int g = 0; g < kGroups; ++g)
                if (16 * g < ncol) {
                  float hi[16], lo[16];
                  tmem_ld16(acc + (uint32_t)(16 * g), hi);
                  tmem_ld16(acc + (uint32_t)(h + 16 * g), lo);
                  tmem_ld_wait();
#pragma unroll
                  for (int c = 0; c < 16; ++c) x[g][c] += hi[c] + lo[c];
                }
            }
            tc_fence_before();
            mbar_arrive(bar(B->acc_free[buf]));
          }
          if (!ok || t + tile >= v.count) continue;
#pragma unroll
          for (int g = 0; g < kGroups; ++g)
            if (16 * g < ncol) {
              if (pair_sum) {  // FP32 data: the data row's W = hi-row product + lo-row product
#pragma unroll
                for (int c = 0; c < 16; ++c) x[g][c] += __shfl_xor_sync(0xffffffffu, x[g][c], 1);
              }
              // hi and lo parts of the lane's row; even lanes store the hi
              // parts of rows rr, rr + 1 (adjacent in the K-major operand),
              // odd lanes the lo parts of rows rr - 1, rr
              uint32_t own[16];
#pragma unroll
              for (int c = 0; c < 16; ++c) {
                const __nv_bfloat16 xh = __float2bfloat16_rn(x[g][c]);
                const __nv_bfloat16 xl = __float2bfloat16_rn(x[g][c] - __bfloat162float(xh));
                own[c] = (uint32_t)__bfloat16_as_ushort(xh) | (uint32_t)__bfloat16_as_ushort(xl) << 16;
              }
#pragma unroll
              for (int c = 0; c < 16; ++c) {
                const uint32_t other = __shfl_xor_sync(0xffffffffu, own[c], 1);
                const uint32_t word = odd ? __byte_perm(other, own[c], 0x7632) : __byte_perm(own[c], other, 0x5410);
                if (16 * g + c < ncol) *reinterpret_cast<uint32_t*>(img + swz(w * ncol + 16 * g + c, e)) = word;
              }
            }
        }
      }
    }
  }
  epilogue(B, tmem, a.err);
}

// ------------------------------------------------------------------ sweep 2
__global__ void __launch_bounds__(kThreads, 1) g_kernel(const __grid_constant__ Inst one, Args a) {
  if (a.insts == nullptr && one.done != nullptr && *one.done) return;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int S = a.stages, stage = a.stage_bytes;
  Bars* B = reinterpret_cast<Bars*>(smem + S * stage);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t tmem = prologue(B, S, 256);
  const int nseg = seg_count(a);
  auto bar = [](const uint64_t& b) { return smem_u32(&b); };
  if (warp == 0 && lane == 0) {
    bool ok = true;
    int u = 0;
    for (int s = 0; s < nseg && ok; ++s) {
      const View v = seg_view(a, &one, s);
      const Inst* I = v.I;
      int w, p0, np;
      block_of(I->d, I->nv, v.block, &w, &p0, &np);
      const uint32_t wbytes = 2 * I->nw * 128;
      const CUtensorMap* map = I->map + w;
      const uint8_t* wimg = I->wimg;
      const long long wait = I->wait;
      for (int t = 0; t < v.count; ++t, ++u) {
        const int tile = v.first + t, slot = u % S;
        if (!(ok = mbar_wait(bar(B->empty[slot]), ((u / S) & 1) ^ 1, &B->abort_flag, wait))) break;
        const uint32_t fb = bar(B->full[slot]), dst = smem_u32(smem + slot * stage);
        mbar_expect_tx(fb, np * kPair + wbytes);
        for (int p = 0; p < np; ++p) {
          tma_load_2d(dst + p * kPair, map, 128 * (p0 + p), tile * 64, fb);
          tma_load_2d(dst + p * kPair + kBox, map, 128 * (p0 + p) + 64, tile * 64, fb);
        }
        bulk_g2s(dst + kMaxPairs * kPair, wimg + (int64_t)tile * wbytes, wbytes, fb);
      }
    }
    drain_copies(B, u, S);
  } else if (warp == 1 && lane == 0) {
    bool ok = true;
    int u = 0, sp = 0;
    for (int s = 0; s < nseg && ok; ++s) {
      const View v = seg_view(a, &one, s);
      if (v.count == 0) continue;
      const Inst* I = v.I;
      int w, p0, np;
      block_of(I->d, I->nv, v.block, &w, &p0, &np);
      const int N2 = 2 * I->nw;
      const long long wait = I->wait;
      const uint32_t id = idesc_bf16(128, N2, 1, 0);
      // the accumulators of the previous segment have been drained
      if (sp > 0 && !(ok = mbar_wait(bar(B->acc_free[0]), (sp - 1) & 1, &B->abort_flag, wait))) break;
      tc_fence_after();
      ++sp;
      for (int t = 0; t < v.count; ++t, ++u) {
        const int slot = u % S;
        if (!(ok = mbar_wait(bar(B->full[slot]), (u / S) & 1, &B->abort_flag, wait))) break;
        tc_fence_after();
        const uint64_t wd = sdesc(smem_u32(smem + slot * stage + kMaxPairs * kPair), 16, 1024);
        for (int p = 0; p < np; ++p) {
          const uint64_t ad = sdesc(smem_u32(smem + slot * stage + p * kPair), kBox, 1024);
#pragma unroll
          for (int q = 0; q < 4; ++q)  // K steps of 16 rows: 2048 bytes of A, 32 bytes of B
            mma_bf16(tmem + (uint32_t)(p * N2), ad + (uint64_t)(128 * q), wd + (uint64_t)(2 * q), id,
                     (t | q) != 0 ? 1u : 0u);
        }
        mma_commit(bar(B->empty[slot]));
      }
      if (ok) mma_commit(bar(B->acc_full[0]));
    }
    if (u > 0) drain_mmas(B);
  } else if (warp >= 4) {
    const int q = warp & 3;
    const uint32_t lane_off = (uint32_t)(32 * q) << 16;
    bool ok = true;
    int sp = 0;
    for (int s = 0; s < nseg && ok; ++s) {
      const View v = seg_view(a, &one, s);
      if (v.count == 0) continue;
      const Inst* I = v.I;
      int w, p0, np;
      block_of(I->d, I->nv, v.block, &w, &p0, &np);
      if (!(ok = __all_sync(0xffffffffu, mbar_wait(bar(B->acc_full[0]), sp & 1, &B->abort_flag, I->wait)))) break;
      tc_fence_after();
      ++sp;
      // column-major slab: the lanes of a warp hold 32 consecutive rows, so
      // every store of a column is one 128-byte line
      const int o0 = pad_rows(I->d[0]), D = o0 + (I->nv > 1 ? pad_rows(I->d[1]) : 0), cols = I->nv * I->ncol;
      float* out = I->part + (int64_t)v.slab * I->slab + w * o0;
      const int nw = I->nw, dw = I->d[w];
      for (int p = 0; p < np; ++p) {
        const int col = 128 * (p0 + p) + 32 * q + lane;
        // the two warps of a lane quadrant take alternate groups of 16 columns
        for (int c0 = 16 * ((warp >> 2) - 1); c0 < cols; c0 += 32) {
          float hi[16], lo[16];
          tmem_ld16(tmem + lane_off + (uint32_t)(p * 2 * nw + c0), hi);
          tmem_ld16(tmem + lane_off + (uint32_t)(p * 2 * nw + nw + c0), lo);
          tmem_ld_wait();
          if (col < dw) {
#pragma unroll
            for (int c = 0; c < 16; ++c)
              if (c0 + c < cols) out[(int64_t)(c0 + c) * D + col] = hi[c] + lo[c];  // hi + lo products
          }
        }
      }
      tc_fence_before();
      mbar_arrive(bar(B->acc_free[0]));
    }
  }
  epilogue(B, tmem, a.err);
}

namespace {

int ring_stages(int stage_bytes) {
  return std::min(kMaxStages, (kSmem - 1024 - (int)sizeof(Bars)) / stage_bytes);
}
int ring_smem(int stages, int stage_bytes) { return stages * stage_bytes + (int)sizeof(Bars) + 1024; }

template <typename K>
int launch(K kern, const Inst& one, Args a, int stage_bytes, int ctas, cudaStream_t st) {
  a.stage_bytes = stage_bytes;
  a.stages = ring_stages(stage_bytes);
  const int smem = ring_smem(a.stages, stage_bytes);
  GB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  kern<<<ctas, kThreads, smem, st>>>(one, a);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// Bytes a 64-row tile of block b moves (its pairs from HBM; the W image, from
// L2, at half weight): the unit in which CTAs are shared out.
int64_t block_weight(const Inst& I, int b) {
  int w, p0, np;
  block_of(I.d, I.nv, b, &w, &p0, &np);
  return (int64_t)np * kPair + I.nw * 128;
}

}  // namespace

int sweep_w(const Inst& one, int h, int* err, int sm_count, cudaStream_t st) {
  Args a{};
  a.err = err;
  a.h = h;
  a.nblk = 1;
  a.cta0[1] = std::min(sm_count, one.ntiles);
  a.nseg[0] = 1;
  return launch(w_kernel, one, a, kUnit * kBox + 2 * h * 128, a.cta0[1], st);
}

int sweep_g(const Inst& one, int* err, int sm_count, int max_slabs, int* np, cudaStream_t st) {
  Args a{};
  a.err = err;
  a.nblk = block_count(one.d, one.nv);
  int64_t total = 0;
  for (int b = 0; b < a.nblk; ++b) total += block_weight(one, b);
  // CTAs per block in proportion to its weight, at least one, at most a CTA
  // per tile and a slab each
  int left = std::max(sm_count, a.nblk);
  for (int b = 0; b < a.nblk; ++b) {
    const int64_t w = block_weight(one, b);
    int nc = (int)std::min<int64_t>((left * w + total / 2) / total, left - (a.nblk - 1 - b));
    nc = std::max(1, std::min(std::min(nc, max_slabs), one.ntiles));
    left -= nc;
    total -= w;
    a.cta0[b + 1] = a.cta0[b] + nc;
    a.nseg[b] = std::max(1, std::min(max_slabs / nc, (one.ntiles + nc * kChain - 1) / (nc * kChain)));
    int v, p0, n;
    block_of(one.d, one.nv, b, &v, &p0, &n);
    for (int p = 0; p < n; ++p) np[8 * v + p0 + p] = nc * a.nseg[b];
  }
  return launch(g_kernel, one, a, kMaxPairs * kPair + 2 * one.nw * 128, a.cta0[a.nblk], st);
}

// ------------------------------------------------------------------- batch
Batch* batch_create(const std::vector<Inst>& insts, int h, int sm, cudaStream_t st, int* rc) {
  *rc = GBCCA_OK;
  auto* b = new (std::nothrow) Batch();
  if (b == nullptr) {
    *rc = GBCCA_ERR_OOM;
    return nullptr;
  }
  b->n = (int)insts.size();
  b->h = h;
  b->sm = sm;
  int blocks = 0;
  for (const Inst& I : insts) {
    blocks += block_count(I.d, I.nv);
    b->nw = std::max(b->nw, I.nw);
  }
  // a contiguous partition has at most CTAs + blocks pieces, cut further to
  // kChain tiles
  b->max_segs = sm + blocks + 1;
  for (const Inst& I : insts) b->max_segs += block_count(I.d, I.nv) * (I.ntiles / kChain + 1);
  bool ok = cudaMallocHost(&b->inst_h, sizeof(Inst) * b->n) == cudaSuccess &&
            cudaMalloc(&b->inst_d, sizeof(Inst) * b->n) == cudaSuccess;
  for (int k = 0; k < 2; ++k)
    ok = ok && cudaMallocHost(&b->seg_h[k], sizeof(Seg) * b->max_segs) == cudaSuccess &&
         cudaMallocHost(&b->off_h[k], sizeof(int) * (sm + 1)) == cudaSuccess &&
         cudaMalloc(&b->seg_d[k], sizeof(Seg) * b->max_segs) == cudaSuccess &&
         cudaMalloc(&b->off_d[k], sizeof(int) * (sm + 1)) == cudaSuccess;
  ok = ok && cudaMallocHost(&b->np_h, sizeof(int) * 16 * b->n) == cudaSuccess &&
       cudaMalloc(&b->np_d, sizeof(int) * 16 * b->n) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    batch_destroy(b);
    set_last_error("allocation of the batch schedule failed");
    *rc = GBCCA_ERR_OOM;
    return nullptr;
  }
  for (int i = 0; i < b->n; ++i) b->inst_h[i] = insts[i];
  cudaError_t e = cudaMemcpyAsync(b->inst_d, b->inst_h, sizeof(Inst) * b->n, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    set_last_error(std::string("batch table upload: ") + cudaGetErrorString(e));
    batch_destroy(b);
    *rc = GBCCA_ERR_CUDA;
    return nullptr;
  }
  return b;
}

void batch_destroy(Batch* b) {
  if (b == nullptr) return;
  cudaFreeHost(b->inst_h);
  cudaFree(b->inst_d);
  for (int k = 0; k < 2; ++k) {
    cudaFreeHost(b->seg_h[k]);
    cudaFreeHost(b->off_h[k]);
    cudaFree(b->seg_d[k]);
    cudaFree(b->off_d[k]);
  }
  cudaFreeHost(b->np_h);
  cudaFree(b->np_d);
  delete b;
}

// Both sweeps' schedules of the active instances over `ctas` CTAs: the items
// (64-row tiles, weighted by their boxes in sweep 1, of every block in sweep
// 2) are cut into contiguous ranges of near-equal weight.  The
// pieces of a block write its slabs 0, 1, ... in order.  The pinned host
// tables are rewritten only by the next schedule, after the caller has
// synchronized `st`.
int batch_schedule(Batch* b, const bool* active, int ctas, cudaStream_t st) {
  ctas = std::max(1, std::min(ctas, b->sm));
  struct Item {
    int inst, block, tiles;
    int64_t weight;
  };
  for (int k = 0; k < 2; ++k) {
    std::vector<Item> items;
    int64_t total = 0;
    for (int i = 0; i < b->n; ++i) {
      if (!active[i]) continue;
      const Inst& I = b->inst_h[i];
      if (k == 0) {
        // a tile costs its boxes, but at least its epilogue (about a box per 8
        // columns of Phi and view)
        int boxes = 0;
        for (int v = 0; v < I.nv; ++v) boxes += (I.d[v] + 63) / 64;
        items.push_back(Item{i, 0, I.ntiles, std::max(boxes, I.nv * I.ncol / 8) + 1});
      } else {
        for (int c = 0; c < block_count(I.d, I.nv); ++c)
          items.push_back(Item{i, c, I.ntiles, block_weight(I, c)});
      }
    }
    for (const Item& it : items) total += it.tiles * it.weight;
    if (k == 1)
      for (int i = 0; i < 16 * b->n; ++i) b->np_h[i] = 0;
    int c = 0, nseg = 0;
    int64_t cum = 0;
    b->off_h[k][0] = 0;
    auto bound = [&](int cc) { return (total * (cc + 1) + ctas - 1) / ctas; };
    for (const Item& it : items) {
      int pieces = 0, t = 0;
      // CTAs that take a piece of this item, and the tiles of a piece that
      // leave the pieces within the slabs (one per SM)
      const int64_t share = it.tiles * it.weight * ctas / total + 2;
      int64_t most = it.tiles;
      if (k == 1 && share < b->sm) most = std::max<int64_t>(kChain, (it.tiles + b->sm - share - 1) / (b->sm - share));
      while (t < it.tiles) {
        int64_t take = std::min<int64_t>(it.tiles - t, most);
        if (c < ctas - 1) take = std::min<int64_t>(take, (bound(c) - cum) / it.weight);
        if (take <= 0) {  // this CTA is full: close it
          b->off_h[k][++c] = nseg;
          continue;
        }
        b->seg_h[k][nseg++] = Seg{it.inst, t, (int)take, pieces++, it.block};
        t += (int)take;
        cum += take * it.weight;
        if (c < ctas - 1 && cum >= bound(c)) b->off_h[k][++c] = nseg;
      }
      if (k == 1) {
        int v, p0, n;
        block_of(b->inst_h[it.inst].d, b->inst_h[it.inst].nv, it.block, &v, &p0, &n);
        for (int p = 0; p < n; ++p) b->np_h[16 * it.inst + 8 * v + p0 + p] = pieces;
      }
    }
    while (c < ctas) b->off_h[k][++c] = nseg;
    GB_CUDA(cudaMemcpyAsync(b->seg_d[k], b->seg_h[k], sizeof(Seg) * std::max(nseg, 1), cudaMemcpyHostToDevice, st));
    GB_CUDA(cudaMemcpyAsync(b->off_d[k], b->off_h[k], sizeof(int) * (ctas + 1), cudaMemcpyHostToDevice, st));
  }
  GB_CUDA(cudaMemcpyAsync(b->np_d, b->np_h, sizeof(int) * 16 * b->n, cudaMemcpyHostToDevice, st));
  b->ctas = ctas;
  return GBCCA_OK;
}

int batch_launch(const Batch* b, int* err, cudaStream_t st) {
  Args a{};
  a.err = err;
  a.h = b->h;
  a.insts = b->inst_d;
  a.segs = b->seg_d[0];
  a.seg_off = b->off_d[0];
  // (the instance parameter is unused with a table)
  GB_TRY(launch(w_kernel, b->inst_h[0], a, kUnit * kBox + 2 * b->h * 128, b->ctas, st));
  a.segs = b->seg_d[1];
  a.seg_off = b->off_d[1];
  return launch(g_kernel, b->inst_h[0], a, kMaxPairs * kPair + 2 * b->nw * 128, b->ctas, st);
}

}  // namespace two
}  // namespace gbcca
