// Tensor-core (tcgen05 + TMA) fused CCA data pass for BF16 data on sm_103a,
// and for FP32 data streamed as a row-interleaved BF16 hi/lo copy (row 2i =
// bf16(z_i), row 2i + 1 = bf16(z_i - bf16(z_i)); see `pair_sum`).  The FDA
// pass (Sec. 5.1-5.2, Cor. 5.6: S_w Phi = Xhat^T (Xhat Phi) over the copy of
// the class-centred rows) is the same kernel in one-view clusters (kSolo):
// both CTAs stream the one view, each half of its 128-column pairs, and add
// their partial products W of every tile before GEMM 2.
//
// One Riemannian-CG iteration of the CCA solver needs, for the block-diagonal
// Phi = blkdiag([U, eta_U], [V, eta_V]) (Sec. 4.2 gradient, Table 1
// retraction, Cor. 4.6 per-iteration cost O(p (nnz X + nnz Y))):
//     W = Z Phi  (Z = [X | Y], n x 4k, never leaves the chip)
//     G = Z^T W  (D x 4k)
// and W^T W, which equals Phi^T G and is formed afterwards in FP64 from G.
//
// Persistent kernel of 2-CTA clusters; both CTAs of a cluster work on the
// same 64-row tile, CTA v on view v (X or Y), so that each CTA keeps its
// 64 x d_v BF16 block (<= 64 KB) in shared memory for both GEMMs and every
// byte of the data is read from HBM exactly once.  Two tiles are resident per
// CTA (double buffering): the next tile streams in while the current one is
// in its epilogue and second GEMM.  Per tile (h = 20 for 2k <= 20, else 24):
//   GEMM 1  (tcgen05, M = 64, per CTA): W_v = Z_v Phi_v, 64 x 2h FP32 in TMEM
//           (B = Phi_v split into bf16 hi|lo columns, h each; rows 16 q ..
//           16 q + 15 of the M = 64 result sit in lanes 32 q .. 32 q + 15);
//   epilogue warps read W_v from TMEM, add the hi and lo halves, split W_v
//           into bf16 hi/lo and write it into the K-major B operand of GEMM 2
//           (rows h v .. h v + h - 1 of the hi part and of the lo part) of
//           their own CTA, then push those rows into the peer CTA's operand
//           with bulk shared::cluster copies;
//   GEMM 2  (tcgen05, M = 128, N = 4h, per CTA): G_v += Z_v^T [W_x | W_y]
//           for the hi and the lo parts at once (separate accumulator
//           columns, added when G is drained), over the same shared-memory
//           blocks read as MN-major A (128 columns of Z_v per MMA),
//           accumulated in TMEM over all tiles of the cluster.  One MMA per
//           K step reads each block of the tile once: the operand reads from
//           shared memory, not the tensor arithmetic, bound these small-N
//           products.
// The end of GEMM 2 is signalled to both CTAs (multicast commit), which
// frees both CTAs' W operand buffer of that tile.  At the end the epilogue
// warps drain G to a per-cluster FP32 partial; a second kernel sums the
// partials in fixed order.
//
// Roles per CTA: warp 0 lane 0 = TMA producer (it first issues the bulk copy
// of the own view's Phi image, so the ring starts filling at once); warp 1
// lane 0 = GEMM 1 issuer (with 2k <= 20: for the first half of the pairs,
// warp 2 lane 0 for the second half, into a second accumulator that the
// epilogue adds); warp 3 lane 0 = GEMM 2 issuer; warp 2 = TMEM allocator;
// warps 4-7 and 8-11 = two epilogue groups (even and odd tiles; TMEM lane
// quarters 0-3 each), whose per-tile chains of dependent steps overlap.
// Every mbarrier wait is bounded in time; on expiry the CTA records an error
// code, waits (bounded) for its own copies and MMAs, frees TMEM and leaves
// after a cluster barrier (no remote access can target an exited CTA).
#include <cstring>
#include <vector>

#include "pass_two.h"

namespace gbcca {

namespace tc {

constexpr int kRows = 64;             // rows per tile (MMA M of GEMM 1, K of GEMM 2)
constexpr int kHalfMax = 24;          // W rows of a view at most (2k <= 24)
constexpr int kTileSlots = 4;         // pair slots of one tile (512 columns)
constexpr int kSlot = 16384;          // two 64 x 64 BF16 boxes
constexpr int kBox = 8192;
constexpr int kPhiView = 49152;       // stride of the views' Phi images in the plan buffer
constexpr int kMaxSmem = 232448;      // dynamic shared memory of one CTA
constexpr uint32_t kTmemCols = 512;   // W: columns kTW (nacc b + a); G: kTG + kN2 p (p < 4 pairs)
constexpr int kTW = 48;               // TMEM column stride of the W accumulators
constexpr long long kTimeout = kWaitCycles;       // cycles (~1 s)

// Shared-memory layout and barriers for GEMM 1 with N = 2 kH1 (Phi columns as
// bf16 hi rows 0 .. kH1 - 1 and lo rows kH1 .. 2 kH1 - 1; kH1 = 20 serves
// 2k <= 20 and leaves room for a 10-slot ring, kH1 = 24 a 9-slot ring).
template <int kH1, bool kSolo = false>
struct Lay {
  static constexpr int kN1 = 2 * kH1;
  static constexpr int kKBox1 = kN1 * 128;       // one K-box (64 columns) of the Phi image
  static constexpr int kPhiBytes = 8 * kKBox1;   // 512 columns
  // W operand of GEMM 2 (K-major, one K-box of 64 tile rows): rows
  // [W_x | W_y] of the hi parts (kH1 rows per view; rows 2k .. kH1 - 1 stay
  // zero), then the same rows of the lo parts, so that one MMA with
  // N = kN2 reads the tile's columns once for both parts.  One view (FDA):
  // its rows padded to 24 per part (an M = 128 MMA needs N a multiple of 16).
  static constexpr int kHalf = kH1;              // W rows of a view
  static constexpr int kNW = kSolo ? 24 : 2 * kH1;  // rows of one part (hi or lo)
  static constexpr int kN2 = 2 * kNW;            // N of GEMM 2
  static constexpr int kWs = kNW * 128;          // bytes of one part
  static constexpr int kWBuf = 2 * kWs;          // hi + lo
  static constexpr int kWHalf = kHalf * 128;     // one view's rows of one part
  static constexpr int kD1Cols = ((kN1 + 15) / 16) * 16;  // TMEM columns read back for W
  // GEMM 1 is issued by two threads (pairs [0, ceil(np / 2)) and the rest),
  // each into its own accumulator, when TMEM has room for 2 x 2 W
  // accumulators and the G accumulators: one thread issues an MMA only about
  // every 50 cycles, two streams overlap in the tensor pipe.
  static constexpr int kNAcc = (4 * kTW + kTileSlots * kN2 <= (int)kTmemCols) ? 2 : 1;
  static constexpr int kTG = 2 * kNAcc * kTW;    // first TMEM column of the G accumulators
  // one-view clusters (FDA: the view's columns split over the two CTAs): two
  // FP32 buffers that receive the other half's partial W of a tile
  static constexpr bool kHalves = kSolo;  // a view's pairs over two CTAs
  static constexpr int kXC = 24;                 // floats per row of an exchange buffer
  static constexpr int kXBytes = kHalves ? 2 * kRows * kXC * 4 : 0;
  static constexpr int kStages = (kMaxSmem - kPhiBytes - 2 * kWBuf - kXBytes - 512 - 1024) / kSlot;
  static constexpr int kRingOff = kPhiBytes;
  static constexpr int kWsOff = kRingOff + kStages * kSlot;
  static constexpr int kXOff = kWsOff + 2 * kWBuf;
  static constexpr int kBarOff = kXOff + kXBytes;
  static constexpr int kSmemBytes = kBarOff + 512 + 1024;  // barriers + alignment slack
  // barrier indices
  static constexpr int kFull = 0, kEmpty = kStages, kD1Full = 2 * kStages;  // [stages], [stages], [2]
  static constexpr int kD1Free = kD1Full + 2, kEpiSync = kD1Free + 2, kWReady = kEpiSync + 1;  // [2], 1, [2]
  static constexpr int kWPeer = kWReady + 2, kWFree = kWPeer + 2, kGDone = kWFree + 2;      // [2], [2], 1
  static constexpr int kFinal = kGDone + 1;                         // [3]: one per MMA-issuing thread
  static constexpr int kPhiFull = kFinal + 3;  // Phi image in shared memory
  static constexpr int kGFree = kPhiFull + 1;   // G drained (128 arrivals)
  static constexpr int kPhiFree = kGFree + 1;  // GEMM 1 done with a segment's Phi
  static constexpr int kXFull = kPhiFree + 1, kXFree = kXFull + 2;  // [2], [2]: partial-W exchange
  static constexpr int kEpiSyncB = kXFree + 2;  // the second epilogue group's kEpiSync
  static constexpr int kNumBars = kEpiSyncB + 1;
  static_assert(kStages >= 2 * kTileSlots, "two resident tiles");
  static_assert(kN1 <= kTW && kD1Cols <= kTW, "W buffers in TMEM");
  static_assert(kN2 % 16 == 0 && kTG + kTileSlots * kN2 <= (int)kTmemCols, "G accumulators in TMEM");
  static_assert(kPhiBytes % 16 == 0 && kWHalf % 16 == 0 && kWs % 1024 == 0, "bulk copy and swizzle alignment");
  static_assert(kRows == 64, "GEMM 2 issues four K steps of 16 rows");
  static_assert(kNumBars * 8 + 8 <= 512, "barrier area");
  static_assert(kSmemBytes <= kMaxSmem, "shared memory");
};

// One instance of a batched pass (device memory; the tensor maps are read by
// the TMA unit from there; CUtensorMap carries its own 128-byte alignment).
struct Inst {
  CUtensorMap map[2];      // views X, Y (BF16 data, or the interleaved hi/lo copy)
  const uint8_t* phi_img;  // [view][K-box][2 kH1][128 B], pre-swizzled
  float* partG;            // partial slabs of this instance
  const int* done;         // the instance's convergence flag: skip it when set
  int64_t slab;            // floats per partial slab (see tc_slab)
  int64_t img_view;        // bytes between the two views' Phi images
  int d[2];
  int pairs[2];
  int k2;
  int pair_sum;
};

// A contiguous range of one instance's 64-row tiles, processed by one cluster
// into partial slab `slab` of that instance.
struct Seg {
  int inst;
  int first;
  int count;
  int slab;
};

struct Args {
  // one instance (insts == nullptr): cluster c takes tiles c, c + clusters,
  // ... of the pair of matrices in the kernel's tensor-map parameters
  int64_t n;
  int d[2];
  int pairs[2];
  int k2;        // columns of Phi per view (2k)
  int ntiles;
  const uint8_t* phi_img;  // [view][K-box][2 kH1][128 B], pre-swizzled
  float* partG;            // [cluster][column][padded rows of the views]
  int64_t slab;            // floats between the clusters' partial slabs
  int* err;
  const int* done;
  int64_t img_view;        // bytes between the two views' Phi images
  int pair_sum;            // 1: rows 2i and 2i+1 of the streamed matrix are the bf16
                           // hi and lo parts of one data row (FP32 data): W of the
                           // row is the sum of the two product rows, and both rows
                           // of GEMM 2's operand carry it
  long long wait_limit;    // one-view clusters: cycles of one pipeline wait before the
                           // kernel gives up (the other shapes use kWaitCycles)
  // several instances (insts != nullptr): cluster c takes the segments
  // seg_off[c] .. seg_off[c + 1] - 1 in order
  const Inst* insts;
  const Seg* segs;
  const int* seg_off;      // [clusters + 1]
};

// What one CTA needs of the segment it is on.
struct SegView {
  const CUtensorMap* map;  // this CTA's view
  const uint8_t* phi;      // this view's Phi image
  float* out;              // partial slab of the segment
  int first, stride, count;
  int d0, d1, npairs, k2, pair_sum;
  int pb;                  // first 128-column pair of this CTA
  bool skip;
};

// The 128-column pairs of a view of P pairs that CTA half h takes: all of
// them in a cluster of two views; in a one-view cluster the first ceil(P / 2)
// for h = 0 and the rest for h = 1, at least
// one (a pair past the view's last column reads zeros from the tensor map and
// the image, and drains nothing).
__device__ __forceinline__ void half_pairs(int P, bool split, int h, int* pb, int* np) {
  if (!split) {
    *pb = 0;
    *np = P;
    return;
  }
  const int p0 = (P + 1) / 2;
  *pb = h == 0 ? 0 : p0;
  *np = h == 0 ? p0 : max(1, P - p0);
}

__device__ __forceinline__ int seg_count(const Args& a, int cid, int ncl) {
  if (a.insts == nullptr) return 1;
  return a.seg_off[cid + 1] - a.seg_off[cid];
}

// (split: the view's pairs are split over two CTAs)
__device__ __forceinline__ SegView seg_view(const Args& a, const CUtensorMap* tmx, const CUtensorMap* tmy, int view,
                                            int cid, int ncl, int s, bool split = false, int half = 0) {
  SegView v;
  if (a.insts == nullptr) {
    v.map = view == 0 ? tmx : tmy;
    v.phi = a.phi_img + view * a.img_view;
    v.d0 = a.d[0];
    v.d1 = a.d[1];
    v.out = a.partG + (int64_t)cid * a.slab;
    v.first = cid;
    v.stride = ncl;
    v.count = (a.ntiles - cid + ncl - 1) / ncl;
    half_pairs(a.pairs[view], split, half, &v.pb, &v.npairs);
    v.k2 = a.k2;
    v.pair_sum = a.pair_sum;
    v.skip = false;
  } else {
    const Seg sg = a.segs[a.seg_off[cid] + s];
    const Inst* I = a.insts + sg.inst;
    v.map = &I->map[view];
    v.phi = I->phi_img + view * I->img_view;
    v.out = I->partG + (int64_t)sg.slab * I->slab;
    v.d0 = I->d[0];
    v.d1 = I->d[1];
    v.first = sg.first;
    v.stride = 1;
    v.count = sg.count;
    half_pairs(I->pairs[view], split, half, &v.pb, &v.npairs);
    v.k2 = I->k2;
    v.pair_sum = I->pair_sum;
    v.skip = I->done != nullptr && *I->done != 0;
  }
  if (v.skip) v.count = 0;
  return v;
}

constexpr int kThreads = 384;  // 4 role warps + two epilogue groups of 4 warps

template <int kH1, bool kSolo = false>
__global__ void __launch_bounds__(kThreads, 1)
tc_pass_kernel(const __grid_constant__ CUtensorMap tmx, const __grid_constant__ CUtensorMap tmy, Args a) {
  using L = Lay<kH1, kSolo>;
  constexpr bool kHalves = L::kHalves;
  constexpr int kStages = L::kStages;
  constexpr int kFull = L::kFull, kEmpty = L::kEmpty, kD1Full = L::kD1Full, kD1Free = L::kD1Free;
  constexpr int kEpiSync = L::kEpiSync, kWReady = L::kWReady, kWPeer = L::kWPeer, kWFree = L::kWFree;
  constexpr int kGDone = L::kGDone, kFinal = L::kFinal, kPhiFull = L::kPhiFull, kGFree = L::kGFree;
  constexpr int kPhiFree = L::kPhiFree, kXFull = L::kXFull, kXFree = L::kXFree, kEpiSyncB = L::kEpiSyncB;
  constexpr int kNumBars = L::kNumBars;
  constexpr int kTG = L::kTG;
  if (a.done != nullptr && *a.done) return;  // uniform over the cluster: no remote access yet
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* phi_s = smem;
  uint8_t* ring = smem + L::kRingOff;
  uint8_t* ws = smem + L::kWsOff;  // [buffer][hi | lo][kNW rows][128 B]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kNumBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* xbuf = reinterpret_cast<float*>(smem + L::kXOff);  // [buffer][64 rows][kXC]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // rank = view: the two CTAs share the tile's W (views X and Y).  A one-view
  // cluster (FDA): rank = half, the two CTAs add their partial W.
  const uint32_t rank = cluster_ctarank();
  const int view = kSolo ? 0 : (int)(rank & 1u);  // 0: X, 1: Y
  const int half = kSolo ? (int)rank : 0;
  const uint32_t peer = rank ^ 1u;
  const uint32_t hpeer = peer;  // the CTA with the other half
  (void)hpeer;
  (void)xbuf;
  // bound of one pipeline wait: the plan's for a one-view cluster, whose only
  // remote operations are synchronous stores and arrivals (an abort leaves no
  // copy in flight towards the peer); the default otherwise
  const long long wl = kSolo ? a.wait_limit : kWaitCycles;
  const int cid = (int)cluster_id_x(), ncl = (int)cluster_count_x();
  const int nseg = seg_count(a, cid, ncl);
  auto bar = [&](int i) { return smem_u32(&bars[i]); };

  // zero the W operands (each view's Phi image arrives by bulk copies that
  // the producer issues ahead of the first tile of each segment)
  {
    uint4* wz = reinterpret_cast<uint4*>(ws);
    for (int i = threadIdx.x; i < 2 * L::kWBuf / 16; i += blockDim.x) wz[i] = make_uint4(0, 0, 0, 0);
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(bar(kFull + s), 1);
      mbar_init(bar(kEmpty + s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar(kD1Full + b), L::kNAcc);  // one arrival per GEMM 1 issuer
      mbar_init(bar(kD1Free + b), 128);
      mbar_init(bar(kWReady + b), 1);
      mbar_init(bar(kWPeer + b), 1);   // + the peer's bytes
      mbar_init(bar(kWFree + b), kSolo ? 1 : 2);  // own (and the peer's) end of GEMM 2
    }
    mbar_init(bar(kEpiSync), 128);
    mbar_init(bar(kEpiSyncB), 128);
    mbar_init(bar(kGDone), 1);
    mbar_init(bar(kGFree), 128);
    mbar_init(bar(kPhiFree), L::kNAcc);  // one arrival per GEMM 1 issuer
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar(kXFull + b), 4);  // the other half's epilogue warps
      mbar_init(bar(kXFree + b), 4);
    }
    mbar_init(bar(kFinal), 1);
    mbar_init(bar(kFinal + 1), 1);
    mbar_init(bar(kFinal + 2), 1);
    mbar_init(bar(kPhiFull), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_proxy_async();
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers and W operands are initialised
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // Every role walks the same segments and tiles; jg counts the tiles and ig
  // the (tile, pair) items this CTA has processed (barrier phases and ring
  // slots run on across segments), sp the segments with tiles.
  if (warp == 0 && lane == 0) {
    // ------------------------------------------------------------ producer
    bool ok = true;
    int last_use[kStages];
    for (int s = 0; s < kStages; ++s) last_use[s] = -1;
    int jg = 0, ig = 0, sp = 0;
    for (int s = 0; s < nseg && ok; ++s) {
      const SegView sv = seg_view(a, &tmx, &tmy, view, cid, ncl, s, kHalves, half);
      if (sv.count == 0) continue;
      // the Phi image is rewritten only after every GEMM 1 MMA of the
      // previous segment has completed (its issuers signal that once per
      // segment; the barrier of a tile could already be two phases behind
      // this thread, whose parity test would then pass too early)
      if (sp > 0 && !(ok = mbar_wait(bar(kPhiFree), (sp - 1) & 1, abort_flag, wl))) break;
      // this segment's Phi image (GEMM 1's B operand), one bulk copy per K-box
      const uint32_t pb = bar(kPhiFull);
      mbar_expect_tx(pb, L::kPhiBytes);
      // (this CTA's pairs: K-boxes 2 pb .. 2 pb + 7 of the image)
      for (int kb = 0; kb < 8; ++kb)
        bulk_g2s(smem_u32(phi_s + kb * L::kKBox1), sv.phi + (2 * sv.pb + kb) * L::kKBox1, L::kKBox1, pb);
      ++sp;
      for (int t = 0; t < sv.count && ok; ++t, ++jg) {
        const int row0 = (sv.first + t * sv.stride) * kRows;
        for (int p = 0; p < sv.npairs; ++p, ++ig) {
          const int slot = ig % kStages, use = ig / kStages;
          if (!(ok = mbar_wait(bar(kEmpty + slot), (use & 1) ^ 1, abort_flag, wl))) break;
          const uint32_t fb = bar(kFull + slot);
          mbar_expect_tx(fb, kSlot);
          const uint32_t dst = smem_u32(ring + slot * kSlot);
          tma_load_2d(dst, sv.map, 128 * (sv.pb + p), row0, fb);
          tma_load_2d(dst + kBox, sv.map, 128 * (sv.pb + p) + 64, row0, fb);
          last_use[slot] = use;
        }
      }
    }
    if (!ok) {
      // wait (bounded) for the copies this thread issued before leaving
      if (sp > 0) {
        const long long t0 = clock64();
        while (!mbar_try(bar(kPhiFull), (sp - 1) & 1) && clock64() - t0 < kTimeout) {
        }
      }
      for (int s = 0; s < kStages; ++s) {
        if (last_use[s] < 0) continue;
        const long long t0 = clock64();
        while (!mbar_try(bar(kFull + s), last_use[s] & 1) && clock64() - t0 < kTimeout) {
        }
      }
    }
  } else if ((warp == 1 || warp == 3 || (warp == 2 && L::kNAcc == 2)) && lane == 0) {
    // ------------------------------------------------------------ MMA issuers
    // warps 1 and 2: GEMM 1 of every tile (half of the pairs each when there
    // are two accumulators); warp 3: GEMM 2 of every tile.  Separate issuers
    // keep GEMM 2 of tile j (which frees its ring slots) from waiting behind
    // the arrival of tile j + 1's data.
    constexpr uint32_t id1 = idesc_bf16(64, L::kN1, 0, 0);
    constexpr uint32_t id2 = idesc_bf16(128, L::kN2, 1, 0);
    bool ok = true;
    int issued = 0;  // MMAs this thread has issued
    int jg = 0, ig = 0, sp = 0;
    // One thread issues an MMA only about every 50 cycles at best, which for
    // these small shapes is slower than the tensor pipe; the issue loops
    // therefore do no descriptor arithmetic beyond one add of a compile-time
    // offset (a descriptor's low bits are the shared-memory address / 16,
    // and every operand address here is below 2^18).
    if (warp == 1 || warp == 2) {
      const int acc_i = warp - 1;  // accumulator of this issuer
      const uint64_t bdesc0 = sdesc(smem_u32(phi_s), 16, 1024);
      for (int s = 0; s < nseg && ok; ++s) {
        const SegView sv = seg_view(a, &tmx, &tmy, view, cid, ncl, s, kHalves, half);
        if (sv.count == 0) continue;
        const int npairs = sv.npairs;
        const int split = L::kNAcc == 2 ? (npairs + 1) / 2 : npairs;
        const int pb = acc_i == 0 ? 0 : split, pe = acc_i == 0 ? split : npairs;
        if (!(ok = mbar_wait(bar(kPhiFull), sp & 1, abort_flag, wl))) break;
        ++sp;
        for (int t = 0; t < sv.count && ok; ++t, ++jg, ig += npairs) {
          const int b = jg & 1;
          // W buffer b was last read by the epilogue of tile jg - 2
          if (jg >= 2 && !(ok = mbar_wait(bar(kD1Free + b), ((jg - 2) >> 1) & 1, abort_flag, wl))) break;
          tc_fence_after();
          const uint32_t d1 = tmem + (uint32_t)((L::kNAcc * b + acc_i) * kTW);
          for (int p = pb; p < pe; ++p) {
            const int it = ig + p;
            const int slot = it % kStages, use = it / kStages;
            if (!(ok = mbar_wait(bar(kFull + slot), use & 1, abort_flag, wl))) break;
            tc_fence_after();
            const uint64_t ad0 = sdesc(smem_u32(ring + slot * kSlot), 16, 1024);
            const uint64_t bd0 = bdesc0 + (uint64_t)((2 * p * L::kKBox1) >> 4);
            // K steps of 16 columns: box s / 4 of the slot, 32-byte step s % 4
            // inside its 128-byte swizzled rows
#define GB_G1_MMA(s, acc)                                                                        \
  mma_bf16(d1, ad0 + (uint64_t)((((s) >> 2) * kBox + ((s) & 3) * 32) >> 4),                      \
           bd0 + (uint64_t)((((s) >> 2) * L::kKBox1 + ((s) & 3) * 32) >> 4), id1, acc)
            if (p == pb) {
              GB_G1_MMA(0, 0u);
            } else {
              GB_G1_MMA(0, 1u);
            }
            GB_G1_MMA(1, 1u);
            GB_G1_MMA(2, 1u);
            GB_G1_MMA(3, 1u);
            GB_G1_MMA(4, 1u);
            GB_G1_MMA(5, 1u);
            GB_G1_MMA(6, 1u);
            GB_G1_MMA(7, 1u);
#undef GB_G1_MMA
            issued += 8;
          }
          if (!ok) break;
          // an issuer without pairs in this segment arrives plainly; the
          // barrier then completes with the other issuer's MMAs
          if (pe > pb) {
            mma_commit(bar(kD1Full + b));
          } else {
            mbar_arrive(bar(kD1Full + b));
          }
        }
        if (!ok) break;
        // release the Phi image when a later segment will load its own
        bool more = false;
        for (int s2 = s + 1; s2 < nseg && !more; ++s2)
          more = seg_view(a, &tmx, &tmy, view, cid, ncl, s2, kHalves, half).count > 0;
        if (more) {
          if (pe > pb) {
            mma_commit(bar(kPhiFree));
          } else {
            mbar_arrive(bar(kPhiFree));
          }
        }
      }
    } else {
      for (int s = 0; s < nseg && ok; ++s) {
        const SegView sv = seg_view(a, &tmx, &tmy, view, cid, ncl, s, kHalves, half);
        if (sv.count == 0) continue;
        const int npairs = sv.npairs;
        // the epilogue has drained the G accumulators of the previous segment
        if (sp > 0 && !(ok = mbar_wait(bar(kGFree), (sp - 1) & 1, abort_flag, wl))) break;
        tc_fence_after();
        ++sp;
        for (int t = 0; t < sv.count && ok; ++t, ++jg, ig += npairs) {
          const int b = jg & 1;
          // both halves of this tile's W operand: ours and the peer's (one
          // view: ours alone)
          if (!kSolo) mbar_expect_tx(bar(kWPeer + b), 2 * L::kWHalf);
          if (!(ok = mbar_wait(bar(kWReady + b), (jg >> 1) & 1, abort_flag, wl))) break;
          if (!kSolo && !(ok = mbar_wait(bar(kWPeer + b), (jg >> 1) & 1, abort_flag, wl))) break;
          tc_fence_after();
          const uint64_t wd0 = sdesc(smem_u32(ws + b * L::kWBuf), 16, 1024);
          const uint32_t acc0 = t > 0 ? 1u : 0u;
          for (int p = 0; p < npairs; ++p) {
            const int it = ig + p;
            const int slot = it % kStages;
            const uint32_t g = tmem + (uint32_t)(kTG + p * L::kN2);
            const uint64_t ad0 = sdesc(smem_u32(ring + slot * kSlot), kBox, 1024);
            // B = the hi rows and then the lo rows of W (N = kN2): the tile's
            // columns are read once per K step of 16 rows (A: 8-row groups of
            // 1024 bytes, B: 32-byte steps inside the swizzled rows); the lo
            // products accumulate in their own columns of G
            mma_bf16(g, ad0, wd0, id2, acc0);
            mma_bf16(g, ad0 + (uint64_t)(2048 >> 4), wd0 + (uint64_t)(32 >> 4), id2, 1u);
            mma_bf16(g, ad0 + (uint64_t)(4096 >> 4), wd0 + (uint64_t)(64 >> 4), id2, 1u);
            mma_bf16(g, ad0 + (uint64_t)(6144 >> 4), wd0 + (uint64_t)(96 >> 4), id2, 1u);
            mma_commit(bar(kEmpty + slot));
            issued += 4;
          }
          // both CTAs learn that this CTA's GEMM 2 has consumed buffer b (one
          // view: this CTA alone reads its W operand)
          if constexpr (kSolo) {
            mma_commit(bar(kWFree + b));
          } else {
            mma_commit_mc(bar(kWFree + b), (uint16_t)0x3u);
          }
        }
        if (ok) mma_commit(bar(kGDone));  // this segment's G is complete
      }
    }
    if (!ok && issued > 0) {
      // let the MMAs this thread issued finish before the CTA frees its memory
      const int f = kFinal + (warp == 3 ? 1 : (warp == 2 ? 2 : 0));
      mma_commit(bar(f));
      const long long t0 = clock64();
      while (!mbar_try(bar(f), 0) && clock64() - t0 < kTimeout) {
      }
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------------ epilogue
    // Two groups of four warps: group g takes the tiles jg with jg % 2 == g
    // (their W and GEMM 1 accumulator buffer g), so that the epilogues of
    // two consecutive tiles run at once; group 0 drains G at segment ends.
    const int grp = (warp - 4) >> 2;
    const int q = warp & 3;             // TMEM lane quarter (a warp reaches lanes 32 (warp % 4) ..)
    const int esync = grp == 0 ? kEpiSync : kEpiSyncB;
    const int lead = 128 * (grp + 1);   // the group's first thread
    const uint32_t lane_off = (uint32_t)(32 * q) << 16;
    const int rg = 32 * q + lane;       // Z column of a G pair block (M = 128 layout)
    bool ok = true;
    int jg = 0, sp = 0;
    for (int s = 0; s < nseg && ok; ++s) {
      const SegView sv = seg_view(a, &tmx, &tmy, view, cid, ncl, s, kHalves, half);
      if (sv.count == 0) continue;
      const int npairs = sv.npairs;
      const bool two_acc = L::kNAcc == 2 && (npairs + 1) / 2 < npairs;
      for (int t = 0; t < sv.count; ++t, ++jg) {
        const int b = jg & 1;
        if (b != grp) continue;
        if (!(ok = mbar_wait(bar(kD1Full + b), (jg >> 1) & 1, abort_flag, wl))) break;
        tc_fence_after();
        float d1[L::kD1Cols];
#pragma unroll
        for (int c = 0; c < L::kD1Cols; c += 16)
          tmem_ld16(tmem + lane_off + (uint32_t)(L::kNAcc * b * kTW + c), &d1[c]);
        if (two_acc) {
          // second GEMM 1 accumulator (the other half of the pairs)
          float d2[L::kD1Cols];
#pragma unroll
          for (int c = 0; c < L::kD1Cols; c += 16)
            tmem_ld16(tmem + lane_off + (uint32_t)((L::kNAcc * b + 1) * kTW + c), &d2[c]);
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < L::kD1Cols; ++c) d1[c] += d2[c];
        }
        tmem_ld_wait();
        tc_fence_before();
        mbar_arrive(bar(kD1Free + b));
        // both CTAs' GEMM 2 of tile jg - 2 must be done with both halves of buffer b
        if (jg >= 2 && !(ok = mbar_wait(bar(kWFree + b), ((jg - 2) >> 1) & 1, abort_flag, wl))) break;
        uint8_t* wb = ws + b * L::kWBuf;
        {
          // W_v row rr = hi part (TMEM column c) + lo part (column kH1 + c),
          // c < 2k.  Lanes 0..15 hold the rows (M = 64 layout, rows 16 q ..
          // 16 q + 15).  Lanes 0..15 convert column c, lanes 16..31 column
          // c + kH1/2 of the same rows (by shuffle); then even lanes store the
          // bf16 pair of rows (rr, rr + 1), which are adjacent in the K-major
          // operand.  Rows 2k .. kH1 - 1 of the operand hold zeros or values
          // of an earlier segment: they only reach G columns that are not
          // drained.
          constexpr int kLaneCols = kH1 / 2;
          const bool upper = lane >= 16;
          const int rr = 16 * q + (lane & 15);
          // in phases over all columns, so that the shuffles of different
          // columns are in flight together
          float w[kLaneCols];
          uint32_t hs[kLaneCols], ls[kLaneCols];
#pragma unroll
          for (int c0 = 0; c0 < kLaneCols; ++c0) w[c0] = d1[c0 + kLaneCols] + d1[kH1 + c0 + kLaneCols];
#pragma unroll
          for (int c0 = 0; c0 < kLaneCols; ++c0) w[c0] = __shfl_sync(0xffffffffu, w[c0], lane & 15);
          float xs[kLaneCols];
#pragma unroll
          for (int c0 = 0; c0 < kLaneCols; ++c0) {
            float x = upper ? w[c0] : d1[c0] + d1[kH1 + c0];
            // FP32 data: the data row's W = hi-row product + lo-row product
            // (adjacent rows sit in adjacent lanes; a + b == b + a, so both
            // lanes hold the same value)
            if (sv.pair_sum) x += __shfl_xor_sync(0xffffffffu, x, 1);
            xs[c0] = x;
          }
          if constexpr (kHalves) {
            // W of the view = this half's product + the other half's: send
            // ours into the other half's buffer b (once it has read the one
            // of tile jg - 2), take theirs from ours; both CTAs add the same
            // two numbers (a + b == b + a), so they hold the same W
            // Row rr of a buffer holds the lanes' column halves at floats
            // 0 .. 11 and 12 .. 23 (three 16-byte stores each, padded with
            // zeros when kH1 = 20).  The stores of a warp are released by one
            // arrival from lane 0 after the warp's barrier, so a barrier
            // phase counts the four epilogue warps.
            static_assert(2 * ((kLaneCols + 3) / 4 * 4) <= L::kXC && kLaneCols <= 12, "exchange row");
            const int xo = rr * L::kXC + (upper ? 12 : 0);
            // (the waits' verdicts are made warp-uniform: the shuffles below
            // need every lane)
            if (jg >= 2 &&
                !(ok = __all_sync(0xffffffffu, mbar_wait_cluster(bar(kXFree + b), ((jg - 2) >> 1) & 1, abort_flag, wl))))
              break;
            {
              float v[12];
#pragma unroll
              for (int c0 = 0; c0 < 12; ++c0) v[c0] = c0 < kLaneCols ? xs[c0 < kLaneCols ? c0 : 0] : 0.f;
              const uint32_t rx = map_peer(smem_u32(xbuf + b * kRows * L::kXC + xo), hpeer);
#pragma unroll
              for (int u = 0; u < 3; ++u) st_cluster_v4(rx + 16 * u, v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(map_peer(bar(kXFull + b), hpeer));
            if (!(ok = __all_sync(0xffffffffu, mbar_wait_cluster(bar(kXFull + b), (jg >> 1) & 1, abort_flag, wl))))
              break;
            {
              const float4* mine = reinterpret_cast<const float4*>(xbuf + b * kRows * L::kXC + xo);
              float v[12];
#pragma unroll
              for (int u = 0; u < 3; ++u) {
                const float4 t = mine[u];
                v[4 * u] = t.x;
                v[4 * u + 1] = t.y;
                v[4 * u + 2] = t.z;
                v[4 * u + 3] = t.w;
              }
#pragma unroll
              for (int c0 = 0; c0 < kLaneCols; ++c0) xs[c0] += v[c0];
            }
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(map_peer(bar(kXFree + b), hpeer));
          }
#pragma unroll
          for (int c0 = 0; c0 < kLaneCols; ++c0) {
            const __nv_bfloat16 hi = __float2bfloat16_rn(xs[c0]);
            const __nv_bfloat16 lo = __float2bfloat16_rn(xs[c0] - __bfloat162float(hi));
            hs[c0] = __bfloat16_as_ushort(hi);
            ls[c0] = __bfloat16_as_ushort(lo);
          }
#pragma unroll
          for (int c0 = 0; c0 < kLaneCols; ++c0) {
            hs[c0] |= __shfl_down_sync(0xffffffffu, hs[c0], 1) << 16;
            ls[c0] |= __shfl_down_sync(0xffffffffu, ls[c0], 1) << 16;
          }
          if ((lane & 1) == 0) {
#pragma unroll
            for (int c0 = 0; c0 < kLaneCols; ++c0) {
              const int c = upper ? c0 + kLaneCols : c0;
              if (c < sv.k2) {
                const uint32_t off = swz(view * L::kHalf + c, rr);
                *reinterpret_cast<uint32_t*>(wb + off) = hs[c0];
                *reinterpret_cast<uint32_t*>(wb + L::kWs + off) = ls[c0];
              }
            }
          }
        }
        fence_proxy_async();
        mbar_arrive(bar(esync));
        if (threadIdx.x == lead) {
          // all rows written: push this view's rows (hi and lo) into the peer's
          // buffer b (two views), then release our own GEMM 2 (the group's
          // barrier completes once per tile of the group)
          if (!(ok = mbar_wait(bar(esync), (jg >> 1) & 1, abort_flag, wl))) break;
          if constexpr (!kSolo) {
            const uint32_t pbar = map_peer(bar(kWPeer + b), peer);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const uint32_t src = smem_u32(wb + h * L::kWs + view * L::kWHalf);
              bulk_to_peer(map_peer(src, peer), src, L::kWHalf, pbar);
            }
          }
          mbar_arrive(bar(kWReady + b));
        }
      }
      if (!ok) break;
      // this segment's G (group 0): drain to its partial slab, then free the
      // accumulators for the next segment's GEMM 2
      if (grp == 0) {
      if (!(ok = mbar_wait(bar(kGDone), sp & 1, abort_flag, wl))) break;
      tc_fence_after();
      {
        // the slab is column-major (D rows, nv k2 columns): the 32 lanes
        // of a warp hold 32 consecutive rows, so every store of a column is
        // one 128-byte line
        // (each view's rows padded to kPostRows)
        const int o0 = pad_rows(sv.d0);
        const int D = o0 + pad_rows(sv.d1);
        const int dv = view == 0 ? sv.d0 : sv.d1;
        for (int p = 0; p < npairs; ++p) {
          float g[L::kN2];
#pragma unroll
          for (int c = 0; c < L::kN2; c += 16) tmem_ld16(tmem + lane_off + (uint32_t)(kTG + p * L::kN2 + c), &g[c]);
          tmem_ld_wait();
          const int col = 128 * (sv.pb + p) + rg;
          if (col < dv) {
            float* o = sv.out + view * o0 + col;
#pragma unroll
            for (int c = 0; c < (kSolo ? L::kHalf : L::kNW); ++c) {
              const int vv = c / L::kHalf, cc = c - vv * L::kHalf;
              if (cc < sv.k2) o[(int64_t)(vv * sv.k2 + cc) * D] = g[c] + g[L::kNW + c];  // hi + lo products
            }
          }
        }
      }
      tc_fence_before();
      mbar_arrive(bar(kGFree));
      }
      ++sp;
    }
    if (ok) {
      // the peer's last end-of-GEMM-2 signal of this group's buffer (tile
      // jg - 2 or jg - 1, not waited in the loop) must have reached us
      // before we leave
      for (int j = max(0, jg - 2); j < jg; ++j)
        if ((j & 1) == grp) mbar_wait(bar(kWFree + (j & 1)), (j >> 1) & 1, abort_flag);
    }
    tc_fence_before();
  }
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) raise_flag(a.err, kFlagTimeout);
  cluster_sync();  // no bulk copy or remote arrive targets a CTA that has left
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// Phi image: per view, K-boxes of 64 columns; B rows 0..h-1 hold the bf16 hi
// parts of the 2k columns [U | eta], rows h .. their lo parts (x - hi);
// 128B-swizzled.  The point the pass evaluates, hi +
// lo, is written to Phi, so that it is exactly the point the solver holds
// (src may be Phi itself).  One thread per element of Phi (every view in
// one launch), and per element of the columns that fill up the boxes the pass
// reads, which are zero: a batch lays the image out with its own number of
// rows, so what was padding of one layout held entries of another (an infinity
// or NaN there would reach every product).  Rows beyond the 2k of a half are left
// as they are; the columns of W that they form are never used.
struct ImageArgs {
  const double* src[2];  // d x k2 row-major
  double* Phi[2];
  int d[2];
  int pad[2];            // columns of the boxes that the pass reads
  int k2;
  int h;                 // image rows per half
  uint8_t* img;
  int64_t img_view;
  const int* done;
  int* restart;          // a convergence flag to clear (the plan takes part again), or null
};
constexpr int kManyPlans = 16;  // plans of one launch of the per-plan kernels
template <int N> struct Images { ImageArgs a[N]; };

template <int N>
__global__ void __launch_bounds__(256) phi_image_kernel(const __grid_constant__ Images<N> many) {
  const ImageArgs& m = many.a[blockIdx.z];
  if (m.done != nullptr && *m.done) return;
  const int v = blockIdx.y;
  if (m.restart != nullptr && v == 0 && blockIdx.x == 0 && threadIdx.x == 0) *m.restart = 0;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;  // (data column j, Phi column q)
  if (e >= (v == 0 ? m.pad[0] : m.pad[1]) * m.k2) return;
  const int j = e / m.k2, q = e - j * m.k2;
  const bool in = j < (v == 0 ? m.d[0] : m.d[1]);
  const double x = in ? (v == 0 ? m.src[0] : m.src[1])[e] : 0.0;
  const __nv_bfloat16 hi = __double2bfloat16(x);
  const __nv_bfloat16 lo = __double2bfloat16(x - (double)__bfloat162float(hi));
  uint8_t* base = m.img + (int64_t)v * m.img_view + (int64_t)(j >> 6) * (2 * m.h * 128);
  *reinterpret_cast<__nv_bfloat16*>(base + swz(q, j & 63)) = hi;
  *reinterpret_cast<__nv_bfloat16*>(base + swz(m.h + q, j & 63)) = lo;
  if (in) (v == 0 ? m.Phi[0] : m.Phi[1])[e] = (double)__bfloat162float(hi) + (double)__bfloat162float(lo);
}

// After the data kernel: G = the sum of the clusters' partial slabs, and the
// partial sums of the Grams that need it, Phi_v^T [G_v | Phi_v], of every
// block of kPostRows rows of a view.
//
// The slabs (12.5 MB for 1024 x 40 columns and 76 clusters) sit in L2 when
// the data kernel ends, so this is a matter of loads in flight and of FP64
// rate (about two multiply-adds per clock and SM), and of launches: one pass
// over the slabs, with the Grams formed from the block's rows while they are
// in shared memory, replaces a reduction, a Gram kernel that read G back (27
// us together for 1024 x 40) and the Gram of Phi (two launches).  The FP64 work
// of a block, not the slabs, sets the time, so the blocks are as small as one
// float4 of rows: with 8 rows and all of Phi^T Phi a launch took 23 us for 128 x
// 80 columns (16 blocks) and 36 for 2048 x 80.  A slab is column-major with
// the views' rows padded to kPostRows; a CTA reads kPostRows rows of every
// column as one float4 per (column, slab), the slabs strided over the S
// threads that share an item (S = kPostThreads / items, so narrow plans split
// their slabs wider, up to kPostSplit: 42 pairs one after another instead of 16
// cost 1.2 us at six columns), kPostLoads loads in flight each.  Sums are Neumaier-compensated FP32 per
// thread, then the S pairs are added in double-float, in fixed order: the
// error is ~2^-45 of the largest partial, far below the partials' own
// rounding, and does not depend on scheduling.
constexpr int kPostThreads = 512;
constexpr int kPostSplit = 16;  // threads per item at most: their pairs are added one after another
constexpr int kPostLoads = 8;
struct PostArgs {
  const float* part;
  int64_t slab;
  const int* nparts_dev;     // batched pass: the schedule's slab count (by_pair: 16 of them)
  int nparts;
  int by_pair;               // slab counts per (view, 128-column pair): np / nparts_dev[8 view + pair]
  int np[16];
  int d[2], nv, k2;
  const double* Phi[2];
  double* G[2];              // row-major, nv k2 columns
  double* gpart;             // [block][k2 x (nv k2 + k2)]
  double* Gram;              // nv k2 x nv k2
  double* phired;            // [view][k2 x k2], or null
  const int* done;
};
template <int N> struct Posts { PostArgs a[N]; };

__device__ __forceinline__ void df_pair_add(float& S, float& C, float s2, float c2) {
  const float t = S + s2;
  const float bp = t - S;
  const float err = (S - (t - bp)) + (s2 - bp);
  S = t;
  C += err + c2;
}

template <int N>
__global__ void __launch_bounds__(kPostThreads) tc_post_kernel(const __grid_constant__ Posts<N> many) {
  const PostArgs& m = many.a[blockIdx.y];
  if (m.done != nullptr && *m.done) return;
  const int d0p = pad_rows(m.d[0]);
  const int r0 = blockIdx.x * kPostRows;  // first padded row of the block
  const int D = d0p + (m.nv > 1 ? pad_rows(m.d[1]) : 0);
  if (r0 >= D) return;
  const int v = r0 < d0p ? 0 : 1;
  const int row0 = v == 0 ? r0 : r0 - d0p;                              // row within the view
  const int nr = min(kPostRows, (v == 0 ? m.d[0] : m.d[1]) - row0);
  const int NC = m.nv * m.k2, items = NC;  // (column: one float4 of a slab)
  static_assert(kPostRows == 4, "a float4 holds a block's rows");
  __shared__ float4 red_s[kPostThreads], red_c[kPostThreads];
  __shared__ double Gs[kPostRows][4 * kMaxK], Ps[kPostRows][2 * kMaxK];
  const int t = threadIdx.x;
  const int S = min(kPostSplit, kPostThreads / items);  // items <= 80
  const int it = t % items, sl = t / items;
  for (int e = t; e < kPostRows * m.k2; e += kPostThreads) {
    const int r = e / m.k2, c = e - r * m.k2;
    Ps[r][c] = r < nr ? (v == 0 ? m.Phi[0] : m.Phi[1])[(int64_t)(row0 + r) * m.k2 + c] : 0.0;
  }
  if (sl < S) {
    const int at = m.by_pair ? 8 * v + (row0 >> 7) : 0;
    const int nparts = m.nparts_dev != nullptr ? m.nparts_dev[at] : (m.by_pair ? m.np[at] : m.nparts);
    const int64_t stride = m.slab / 4;
    const float4* src = reinterpret_cast<const float4*>(m.part + (int64_t)it * D + r0);
    float s[4] = {0.f, 0.f, 0.f, 0.f}, cp[4] = {0.f, 0.f, 0.f, 0.f};
    for (int b0 = sl; b0 < nparts; b0 += S * kPostLoads) {
      float4 x4[kPostLoads];
#pragma unroll
      for (int u = 0; u < kPostLoads; ++u)
        x4[u] = b0 + u * S < nparts ? src[(int64_t)(b0 + u * S) * stride] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < kPostLoads; ++u) {
        const float x[4] = {x4[u].x, x4[u].y, x4[u].z, x4[u].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float tt = s[i] + x[i];
          cp[i] += (fabsf(s[i]) >= fabsf(x[i])) ? ((s[i] - tt) + x[i]) : ((x[i] - tt) + s[i]);
          s[i] = tt;
        }
      }
    }
    red_s[sl * items + it] = make_float4(s[0], s[1], s[2], s[3]);
    red_c[sl * items + it] = make_float4(cp[0], cp[1], cp[2], cp[3]);
  }
  __syncthreads();
  double* G = v == 0 ? m.G[0] : m.G[1];
  const float* rs = reinterpret_cast<const float*>(red_s);
  const float* rc = reinterpret_cast<const float*>(red_c);
  for (int e = t; e < kPostRows * NC; e += kPostThreads) {
    const int r = e / NC, c = e - r * NC;
    const int o = 4 * c + r;
    float sum = 0.f, comp = 0.f;
    for (int q = 0; q < S; ++q) df_pair_add(sum, comp, rs[4 * q * items + o], rc[4 * q * items + o]);
    const double gv = widen(sum) + widen(comp);
    Gs[r][c] = gv;
    if (r < nr) G[(int64_t)(row0 + r) * NC + c] = gv;
  }
  __syncthreads();
  const int W = NC + m.k2;
  double* out = m.gpart + (int64_t)blockIdx.x * m.k2 * W;
  for (int e = t; e < m.k2 * NC; e += kPostThreads) {
    const int i = e / NC, b = e - i * NC;
    double sum = 0.0;
    for (int r = 0; r < nr; ++r) sum += Ps[r][i] * Gs[r][b];
    out[i * W + b] = sum;
  }
  // Phi^T Phi: one triangle, mirrored (products commute)
  for (int e = t; e < m.k2 * (m.k2 + 1) / 2; e += kPostThreads) {
    int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= e) ++i;
    while (i * (i + 1) / 2 > e) --i;
    const int b = e - i * (i + 1) / 2;
    double sum = 0.0;
    for (int r = 0; r < nr; ++r) sum += Ps[r][i] * Ps[r][b];
    out[i * W + NC + b] = sum;
    out[b * W + NC + i] = sum;
  }
}

// Gram = Phi_bd^T G and the views' Phi^T Phi from the blocks' partials: a CTA
// takes 32 consecutive entries (the lanes) and splits the blocks over its
// eight warps, eight loads in flight; the warps' sums are added in order.
template <int N>
__global__ void __launch_bounds__(256) gram_sum_kernel(const __grid_constant__ Posts<N> many) {
  const PostArgs& m = many.a[blockIdx.y];
  if (m.done != nullptr && *m.done) return;
  __shared__ double red[8][32];
  const int NC = m.nv * m.k2, W = NC + m.k2, per_view = m.k2 * W;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((int)blockIdx.x * 32 >= m.nv * per_view) return;
  const int e = blockIdx.x * 32 + lane;
  const int v = e < per_view ? 0 : 1, f = e - v * per_view;
  const int nb0 = pad_rows(m.d[0]) / kPostRows;
  const int first = v == 0 ? 0 : nb0, nb = v == 0 ? nb0 : pad_rows(m.d[1]) / kPostRows;
  double s = 0.0;
  if (e < m.nv * per_view) {
    const int per = (nb + 7) / 8, b1 = min(nb, (w + 1) * per);
    const double* src = m.gpart + (int64_t)first * per_view + f;
    for (int b0 = w * per; b0 < b1; b0 += 8) {
      double x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = b0 + u < b1 ? src[(int64_t)(b0 + u) * per_view] : 0.0;
#pragma unroll
      for (int u = 0; u < 8; ++u) s += x[u];
    }
  }
  red[w][lane] = s;
  __syncthreads();
  if (w != 0 || e >= m.nv * per_view) return;
#pragma unroll
  for (int q = 1; q < 8; ++q) s += red[q][lane];
  const int i = f / W, b = f - i * W;
  if (b < NC)
    m.Gram[(v * m.k2 + i) * NC + b] = s;
  else if (m.phired != nullptr)
    m.phired[((int64_t)v * m.k2 + i) * m.k2 + (b - NC)] = s;
}

}  // namespace tc

// ----------------------------------------------------------------- host side
namespace {

int make_map(CUtensorMap* map, const void* base, int64_t n, int d, int64_t ld) {
  return make_tma_map_bf16(map, base, n, d, ld, tc::kRows);
}

}  // namespace

// The tensor-core pass serves CCA plans with BF16 data (or FP32 data through
// the interleaved copy), dx, dy <= 1024, 16-byte aligned rows (ld a multiple
// of 8) and 16-byte aligned bases, and FDA plans with FP32 data and d <= 1024
// (the interleaved copy of their class-centred rows, in one-view clusters that
// split the view's column pairs over the two CTAs).  More than 24 columns of
// Phi per view, or a CCA view wider than 512 columns, take the two-sweep
// kernels of pass_two.cu.
bool tc_pass_eligible(const Plan& p) {
  if (p.kind == kLDA) return p.dtype == GBCCA_FP32 && 2 * p.k <= 2 * tc::kHalfMax && p.v[0].d <= 1024 && p.ts_ready;
  if (p.kind != kCCA || 2 * p.k > 2 * tc::kHalfMax || p.v[0].d > 1024 || p.v[1].d > 1024) return false;
  if (p.dtype == GBCCA_FP32) return p.ts_ready;  // the plan's own aligned copy
  if (p.dtype != GBCCA_BF16) return false;
  for (int v = 0; v < 2; ++v) {
    if (p.v[v].ld % 8 != 0 || (reinterpret_cast<uintptr_t>(p.v[v].Z) & 15) != 0) return false;
  }
  return true;
}

// one-view plans (FDA): clusters of two CTAs that split the view's column
// pairs
static bool tc_solo(const Plan& p) { return p.kind == kLDA; }
// Plans that take two sweeps: the one-sweep kernel's accumulators hold 24
// columns per view and its CTAs 512 columns of one.  Where both could serve (a
// view of at most 512 columns, k <= 12) one sweep reads the data once and is
// faster at every width measured (262144 x (512 + 512), k = 10: 106 against
// 185 us).
bool tc_two(const Plan& p) {
  return 2 * p.k > tc::kHalfMax || (p.kind == kCCA && std::max(p.v[0].d, p.v[1].d) > 512);
}
// rows per half of the Phi image
static int tc_h1(const Plan& p) { return tc_two(p) ? (2 * p.k + 7) / 8 * 8 : (2 * p.k <= 20 ? 20 : tc::kHalfMax); }
static int tc_nviews(const Plan& p) { return tc_solo(p) ? 1 : 2; }
// bytes between the views' images: two sweeps, every 64-column box with up
// to 40 rows per half; one-view plans, 16 K-boxes (the second CTA's pairs
// start at K-box 8 at most); else 8 K-boxes
static int64_t tc_img_view(const Plan& p) {
  if (tc_two(p)) return (int64_t)ceil_div(std::max(p.v[0].d, tc_nviews(p) > 1 ? p.v[1].d : 0), 64) * 2 * 40 * 128;
  return (tc_solo(p) ? 2 : 1) * (int64_t)tc::kPhiView;
}
int64_t tc_img_len(const Plan& p) { return tc_nviews(p) * tc_img_view(p); }
static int tc_rows(const Plan& p) { return tc::pad_rows(p.v[0].d) + (tc_nviews(p) > 1 ? tc::pad_rows(p.v[1].d) : 0); }
// floats of one partial slab: 2 x 2k columns (one view: 2k) of the views'
// padded rows; a slab per cluster (two sweeps: per CTA)
static int64_t tc_slab(const Plan& p) { return (int64_t)tc_rows(p) * tc_nviews(p) * 2 * p.k; }
static int tc_max_slabs(const Plan& p) { return tc_two(p) ? p.sm_count : p.sm_count / 2; }
// operand rows of one part of the W image (two sweeps)
static int tc_nw(const Plan& p) { return (tc_nviews(p) * 2 * p.k + 7) / 8 * 8; }
int64_t tc_wimg_bytes(const Plan& p) {
  if (!tc_two(p)) return 0;
  const int64_t rows = p.dtype == GBCCA_FP32 ? 2 * p.n : p.n;
  return (rows + 63) / 64 * (2 * (int64_t)tc_nw(p) * 128);
}

// Doubles of the partial Grams and floats of the partial slabs that a
// tensor-core plan needs.
int64_t tc_gpart_len(const Plan& p) {
  const int k2 = 2 * p.k;
  return (int64_t)(tc_rows(p) / tc::kPostRows) * k2 * (tc_nviews(p) * k2 + k2);
}
int64_t tc_part_len(const Plan& p) { return tc_max_slabs(p) * tc_slab(p); }

// Columns of a view's image: whole boxes of 64, which the one-sweep pass over two
// views reads in pairs.
static int tc_image_cols(const Plan& p, int v) {
  const int unit = tc_two(p) || tc_solo(p) ? 64 : 128;
  return ceil_div(p.v[v].d, unit) * unit;
}

// Arguments of the Phi images of a plan, h1 rows per half (0: the plan's own);
// Phi is read from the caller's blocks when `io` is given, else from the
// plan's own.
static tc::ImageArgs tc_image_args(const Plan& p, int h1, const int* done, const PassIO* io) {
  tc::ImageArgs a{};
  const int nv = tc_nviews(p);
  for (int v = 0; v < nv; ++v) {
    a.src[v] = io != nullptr ? io->Phi[v] : p.v[v].Phi;
    a.Phi[v] = p.v[v].Phi;
    a.d[v] = p.v[v].d;
    a.pad[v] = tc_image_cols(p, v);
  }
  a.k2 = 2 * p.k;
  a.h = h1 > 0 ? h1 : tc_h1(p);
  a.img = p.tc_img;
  a.img_view = tc_img_view(p);
  a.done = done;
  return a;
}
static int tc_image_blocks(const Plan& p) {
  const int cols = std::max(tc_image_cols(p, 0), tc_nviews(p) > 1 ? tc_image_cols(p, 1) : 0);
  return ceil_div(cols * 2 * p.k, 256);
}

// The Phi images of a plan; also rounds Phi to the bf16 hi + lo point the
// pass evaluates.
int tc_phi_image(Plan& p, int h1, cudaStream_t st, const int* done, const PassIO* io) {
  tc::Images<1> m{};
  m.a[0] = tc_image_args(p, h1, done, io);
  tc::phi_image_kernel<1><<<dim3(tc_image_blocks(p), tc_nviews(p), 1), 256, 0, st>>>(m);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

static tc::PostArgs tc_post_args(const Plan& p, const int* nparts, const int* nparts_dev, const int* done,
                                 const PassIO* io) {
  tc::PostArgs a{};
  const int nv = tc_nviews(p), k2 = 2 * p.k;
  a.part = p.tc_part;
  a.slab = tc_slab(p);
  a.nparts_dev = nparts_dev;
  a.by_pair = tc_two(p) ? 1 : 0;
  if (nparts != nullptr) {
    if (a.by_pair)
      std::memcpy(a.np, nparts, sizeof(a.np));
    else
      a.nparts = *nparts;
  }
  a.nv = nv;
  a.k2 = k2;
  for (int v = 0; v < nv; ++v) {
    a.d[v] = p.v[v].d;
    a.Phi[v] = p.v[v].Phi;
    a.G[v] = io != nullptr ? io->G[v] : p.G + (v == 0 ? 0 : (int64_t)p.v[0].d * nv * k2);
  }
  a.gpart = p.tc_gpart;
  a.Gram = io != nullptr ? io->Gram : p.Gram;
  a.phired = p.phired;
  a.done = done;
  return a;
}

// Sum of the partial slabs into G, then W^T W = Phi_bd^T G and the Grams of
// Phi, for `n` plans (n <= N).
template <int N>
static int tc_post_launch(const tc::Posts<N>& m, Plan* const* plans, int n, cudaStream_t st) {
  int blocks = 1, entries = 1;
  for (int i = 0; i < n; ++i) {
    const Plan& p = *plans[i];
    const int k2 = 2 * p.k, nv = tc_nviews(p);
    blocks = std::max(blocks, tc_rows(p) / tc::kPostRows);
    entries = std::max(entries, nv * k2 * (nv * k2 + k2));
  }
  tc::tc_post_kernel<N><<<dim3(blocks, n), tc::kPostThreads, 0, st>>>(m);
  GB_CHECK_LAUNCH();
  tc::gram_sum_kernel<N><<<dim3(ceil_div(entries, 32), n), 256, 0, st>>>(m);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// The streamed matrices of an eligible plan: the caller's BF16 matrices, or
// for FP32 data the plan's row-interleaved hi/lo copy (2n rows).  One-view
// plans stream view 0 (the second entry repeats it and is not read).
static void tc_sources(const Plan& p, const void* src[2], int64_t ld[2], int64_t* rows) {
  const bool fp32 = p.dtype == GBCCA_FP32;
  *rows = fp32 ? 2 * p.n : p.n;
  for (int v = 0; v < 2; ++v) {
    const int u = v < tc_nviews(p) ? v : 0;
    src[v] = fp32 ? (const void*)p.ts_copy[u] : p.v[u].Z;
    ld[v] = fp32 ? p.ts_ld[u] : p.v[u].ld;
  }
}

// A plan's pass in two sweeps (rows: of the streamed matrices).
static two::Inst tc_two_inst(const Plan& p, int64_t rows, const CUtensorMap& mx, const CUtensorMap& my,
                             const int* done) {
  two::Inst I{};
  I.map[0] = mx;
  I.map[1] = my;
  I.phi_img = p.tc_img;
  I.img_view = tc_img_view(p);
  I.wimg = static_cast<uint8_t*>(p.Wbuf);
  I.part = p.tc_part;
  I.slab = tc_slab(p);
  I.done = done;
  I.nv = tc_nviews(p);
  for (int v = 0; v < I.nv; ++v) I.d[v] = p.v[v].d;
  I.ncol = 2 * p.k;
  I.nw = tc_nw(p);
  I.pair_sum = p.dtype == GBCCA_FP32 ? 1 : 0;
  I.ntiles = ceil_div(rows, tc::kRows);
  I.wait = I.nv == 1 && p.opt.wait_cycles > 0 ? p.opt.wait_cycles : tc::kWaitCycles;
  return I;
}

int tc_pass(Plan& p, cudaStream_t st, const int* done, const PassIO* io) {
  // FP32 data: the row-interleaved hi/lo copy (2n rows) made when the data
  // was bound; BF16 data: the caller's matrices
  const bool fp32 = p.dtype == GBCCA_FP32;
  int64_t rows = 0;
  const void* src[2];
  int64_t ld[2];
  tc_sources(p, src, ld, &rows);
  const bool solo = tc_solo(p);
  const int nv = tc_nviews(p);
  for (int v = 0; v < 2; ++v) {
    if (p.tc_map_for[v] == src[v] && p.tc_map_ld[v] == ld[v]) continue;
    p.tc_map_for[v] = nullptr;
    GB_TRY(make_map(reinterpret_cast<CUtensorMap*>(p.tc_map[v]), src[v], rows, p.v[v < nv ? v : 0].d, ld[v]));
    p.tc_map_for[v] = src[v];
    p.tc_map_ld[v] = ld[v];
  }
  GB_TRY(tc_phi_image(p, 0, st, done, io));
  const CUtensorMap* mx = reinterpret_cast<const CUtensorMap*>(p.tc_map[0]);
  const CUtensorMap* my = reinterpret_cast<const CUtensorMap*>(p.tc_map[1]);
  if (p.kev0 != nullptr) GB_CUDA(record_timing_event(p.kev0, st));
  int nparts[16] = {};  // slabs written (two sweeps: per view and pair)
  if (tc_two(p)) {
    const two::Inst one = tc_two_inst(p, rows, *mx, *my, done);
    GB_TRY(two::sweep_w(one, tc_h1(p), p.flag, p.sm_count, st));
    GB_TRY(two::sweep_g(one, p.flag, p.sm_count, tc_max_slabs(p), nparts, st));
  } else {
    const int h1 = tc_h1(p);  // Phi image rows per half (GEMM 1 N = 2 h1)
    tc::Args a{};
    a.n = p.n;
    for (int v = 0; v < 2; ++v) {
      a.d[v] = v < nv ? p.v[v].d : 0;
      a.pairs[v] = ceil_div(a.d[v], 128);
    }
    a.k2 = 2 * p.k;
    a.slab = tc_slab(p);
    a.wait_limit = p.opt.wait_cycles > 0 ? p.opt.wait_cycles : tc::kWaitCycles;
    a.ntiles = ceil_div(rows, tc::kRows);
    a.pair_sum = fp32 ? 1 : 0;
    a.phi_img = p.tc_img;
    a.img_view = tc_img_view(p);
    a.partG = p.tc_part;
    a.err = p.flag;
    a.done = done;
    auto kern = solo ? (h1 == 20 ? tc::tc_pass_kernel<20, true> : tc::tc_pass_kernel<tc::kHalfMax, true>)
                     : (h1 == 20 ? tc::tc_pass_kernel<20> : tc::tc_pass_kernel<tc::kHalfMax>);
    const int smem = solo ? (h1 == 20 ? tc::Lay<20, true>::kSmemBytes : tc::Lay<tc::kHalfMax, true>::kSmemBytes)
                          : (h1 == 20 ? tc::Lay<20>::kSmemBytes : tc::Lay<tc::kHalfMax>::kSmemBytes);
    GB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(tc::kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (p.tc_clusters <= 0) {
      // persistent grid: as many clusters as can be resident at once
      cfg.gridDim = dim3(2 * (p.sm_count / 2), 1, 1);
      int nc = 0;
      GB_CUDA(cudaOccupancyMaxActiveClusters(&nc, kern, &cfg));
      p.tc_clusters = std::max(1, std::min(nc, p.sm_count / 2));
    }
    nparts[0] = std::min(p.tc_clusters, a.ntiles);
    cfg.gridDim = dim3(2 * nparts[0], 1, 1);
    GB_CUDA(cudaLaunchKernelEx(&cfg, kern, *mx, *my, a));
    GB_CHECK_LAUNCH();
  }
  if (p.kev1 != nullptr) GB_CUDA(record_timing_event(p.kev1, st));
  if (p.fork_after_pass) {
    // work that needs only Phi may start beside the reduction
    GB_CUDA(cudaEventRecord(p.pass_fork, st));
    p.pass_forked = true;
  }
  tc::Posts<1> m{};
  m.a[0] = tc_post_args(p, nparts, nullptr, done, io);
  Plan* one = &p;
  return tc_post_launch<1>(m, &one, 1, st);
}


// ------------------------------------------------------------ batched pass
// Several plans' passes in one persistent launch (same kernel, segment
// schedule).  The instance table, the segments and the per-instance slab
// counts live in device memory, so a captured graph keeps one launch while
// the schedule is rewritten between replays (finished plans drop out).
struct TcBatch {
  two::Batch* two = nullptr;   // plans that take two sweeps: their tables and schedules
  int n = 0;                   // plans
  int h1 = tc::kHalfMax;       // Phi image rows per half, common to the batch
  std::vector<int64_t> rows;   // streamed rows per plan
  std::vector<int64_t> plan_bytes;  // algorithmic bytes of one pass per plan
  tc::Inst* inst_h = nullptr;  // pinned host copies of the tables
  tc::Seg* seg_h = nullptr;
  int* off_h = nullptr;
  int* nparts_h = nullptr;
  tc::Inst* inst_d = nullptr;
  tc::Seg* seg_d = nullptr;
  int* off_d = nullptr;
  int* nparts_d = nullptr;
  int* err_d = nullptr;
  std::vector<char> sched;     // active set of the tables in device memory (empty: none yet)
  int max_clusters = 0;        // clusters the tables have room for
  int clusters = 0;            // clusters of the current schedule
  int max_segs = 0;
};

void tc_batch_destroy(TcBatch* b) {
  if (b == nullptr) return;
  two::batch_destroy(b->two);
  cudaFreeHost(b->inst_h);
  cudaFreeHost(b->seg_h);
  cudaFreeHost(b->off_h);
  cudaFreeHost(b->nparts_h);
  cudaFree(b->inst_d);
  cudaFree(b->seg_d);
  cudaFree(b->off_d);
  cudaFree(b->nparts_d);
  cudaFree(b->err_d);
  delete b;
}

// Instance table of the plans (each eligible for the tensor-core pass, with
// its data bound); copied to the device on `st`.
TcBatch* tc_batch_create(Plan* const* plans, int n, cudaStream_t st, int* rc) {
  *rc = GBCCA_OK;
  auto* b = new (std::nothrow) TcBatch();
  if (b == nullptr) {
    *rc = GBCCA_ERR_OOM;
    return nullptr;
  }
  b->n = n;
  int h1 = 0, sm = 1;
  for (int i = 0; i < n; ++i) {
    h1 = std::max(h1, tc_h1(*plans[i]));
    sm = std::max(sm, plans[i]->sm_count);
  }
  b->h1 = h1;
  b->max_clusters = std::max(1, sm / 2);
  b->rows.assign(n, 0);
  b->plan_bytes.assign(n, 0);
  if (n > 0 && tc_two(*plans[0])) {
    if (cudaMalloc(&b->err_d, sizeof(int)) != cudaSuccess || cudaMemsetAsync(b->err_d, 0, sizeof(int), st) != cudaSuccess) {
      cudaGetLastError();
      tc_batch_destroy(b);
      set_last_error("allocation of the batch schedule failed");
      *rc = GBCCA_ERR_OOM;
      return nullptr;
    }
    std::vector<two::Inst> insts;
    for (int i = 0; i < n && *rc == GBCCA_OK; ++i) {
      Plan& p = *plans[i];
      const void* src[2];
      int64_t ld[2], rows = 0;
      tc_sources(p, src, ld, &rows);
      b->rows[i] = rows;
      b->plan_bytes[i] = rows * (int64_t)(p.v[0].d + p.v[1].d) * 2;
      CUtensorMap map[2];
      for (int v = 0; v < 2 && *rc == GBCCA_OK; ++v) *rc = make_map(&map[v], src[v], rows, p.v[v].d, ld[v]);
      if (*rc == GBCCA_OK) insts.push_back(tc_two_inst(p, rows, map[0], map[1], &p.st->done));
    }
    if (*rc == GBCCA_OK) b->two = two::batch_create(insts, h1, sm, st, rc);
    if (b->two == nullptr) {
      tc_batch_destroy(b);
      return nullptr;
    }
    return b;
  }
  b->max_segs = b->max_clusters + n + 1;  // a contiguous partition has at most clusters + plans pieces
  const int n1 = std::max(n, 1);
  bool ok = cudaMallocHost(&b->inst_h, sizeof(tc::Inst) * n1) == cudaSuccess &&
            cudaMallocHost(&b->seg_h, sizeof(tc::Seg) * b->max_segs) == cudaSuccess &&
            cudaMallocHost(&b->off_h, sizeof(int) * (b->max_clusters + 1)) == cudaSuccess &&
            cudaMallocHost(&b->nparts_h, sizeof(int) * n1) == cudaSuccess &&
            cudaMalloc(&b->inst_d, sizeof(tc::Inst) * n1) == cudaSuccess &&
            cudaMalloc(&b->seg_d, sizeof(tc::Seg) * b->max_segs) == cudaSuccess &&
            cudaMalloc(&b->off_d, sizeof(int) * (b->max_clusters + 1)) == cudaSuccess &&
            cudaMalloc(&b->nparts_d, sizeof(int) * n1) == cudaSuccess &&
            cudaMalloc(&b->err_d, sizeof(int)) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    tc_batch_destroy(b);
    set_last_error("allocation of the batch schedule failed");
    *rc = GBCCA_ERR_OOM;
    return nullptr;
  }
  std::memset(b->inst_h, 0, sizeof(tc::Inst) * n1);
  for (int i = 0; i < n; ++i) {
    Plan& p = *plans[i];
    const void* src[2];
    int64_t ld[2], rows = 0;
    tc_sources(p, src, ld, &rows);
    b->plan_bytes[i] = rows * (int64_t)(p.v[0].d + p.v[1].d) * 2;
    b->rows[i] = rows;
    tc::Inst& I = b->inst_h[i];
    for (int v = 0; v < 2; ++v) {
      *rc = make_map(&I.map[v], src[v], rows, p.v[v].d, ld[v]);
      if (*rc != GBCCA_OK) {
        tc_batch_destroy(b);
        return nullptr;
      }
      I.d[v] = p.v[v].d;
      I.pairs[v] = ceil_div(p.v[v].d, 128);
    }
    I.phi_img = p.tc_img;
    I.img_view = tc_img_view(p);
    I.partG = p.tc_part;
    I.done = &p.st->done;
    I.k2 = 2 * p.k;
    I.pair_sum = p.dtype == GBCCA_FP32 ? 1 : 0;
    I.slab = tc_slab(p);
  }
  cudaError_t e = cudaMemcpyAsync(b->inst_d, b->inst_h, sizeof(tc::Inst) * n1, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(b->err_d, 0, sizeof(int), st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    set_last_error(std::string("batch table upload: ") + cudaGetErrorString(e));
    tc_batch_destroy(b);
    *rc = GBCCA_ERR_CUDA;
    return nullptr;
  }
  return b;
}

int tc_batch_h1(const TcBatch* b) { return b->h1; }
int* tc_batch_err(TcBatch* b) { return b->err_d; }
int tc_batch_max_clusters(const TcBatch* b) { return b->max_clusters; }
int tc_batch_clusters(const TcBatch* b) { return b->clusters; }
// Algorithmic bytes of one batched pass over the active plans (each plan's
// data once, also where two sweeps read it).
int64_t tc_batch_bytes(const TcBatch* b, const bool* active) {
  int64_t s = 0;
  for (int i = 0; i < b->n; ++i)
    if (active == nullptr || active[i]) s += b->plan_bytes[i];
  return s;
}

// Schedule of the active instances over `clusters` 2-CTA clusters: their
// 64-row tiles, each weighted by 2 + the pairs of its wider view (the two
// CTAs of a cluster move through a tile together, and a tile costs a fixed
// epilogue and exchange on top of its MMAs), are cut into `clusters`
// contiguous ranges of near-equal weight.  The pieces of instance i (one per
// cluster it reaches) write its slabs 0, 1, ... in order, and its reduction
// adds that many slabs.  The tables go
// to the device on `st`; the pinned host copies are rewritten only by the
// next schedule, after the caller has synchronized `st`.
int tc_batch_schedule(TcBatch* b, const bool* active, int clusters, cudaStream_t st) {
  clusters = std::max(1, std::min(clusters, b->max_clusters));
  // the same set over as many CTAs: the tables in device memory stand
  const std::vector<char> want(active, active + b->n);
  if (clusters == b->clusters && want == b->sched) return GBCCA_OK;
  b->sched.clear();
  if (b->two != nullptr) {
    GB_TRY(two::batch_schedule(b->two, active, 2 * clusters, st));
    b->clusters = clusters;
    b->sched = want;
    return GBCCA_OK;
  }
  auto cta_pairs = [&](int i) { return std::max(b->inst_h[i].pairs[0], b->inst_h[i].pairs[1]); };
  int64_t total = 0;
  for (int i = 0; i < b->n; ++i) {
    b->nparts_h[i] = 0;
    if (active[i]) total += ceil_div(b->rows[i], (int64_t)tc::kRows) * (2 + cta_pairs(i));
  }
  int c = 0, nseg = 0;
  int64_t cum = 0;
  b->off_h[0] = 0;
  auto bound = [&](int cc) { return (total * (cc + 1) + clusters - 1) / clusters; };
  for (int i = 0; i < b->n; ++i) {
    if (!active[i]) continue;
    const int64_t tiles = ceil_div(b->rows[i], (int64_t)tc::kRows);
    const int64_t w = 2 + cta_pairs(i);
    int pieces = 0;  // segments of instance i so far = its next slab
    int64_t t = 0;
    while (t < tiles) {
      int64_t take = tiles - t;
      if (c < clusters - 1) take = std::min(take, (bound(c) - cum) / w);
      if (take <= 0) {  // this cluster is full: close it
        b->off_h[++c] = nseg;
        continue;
      }
      b->seg_h[nseg++] = tc::Seg{i, (int)t, (int)take, pieces++};
      t += take;
      cum += take * w;
      if (c < clusters - 1 && cum >= bound(c)) b->off_h[++c] = nseg;
    }
    b->nparts_h[i] = pieces;
  }
  while (c < clusters) b->off_h[++c] = nseg;
  b->clusters = clusters;
  GB_CUDA(cudaMemcpyAsync(b->seg_d, b->seg_h, sizeof(tc::Seg) * std::max(nseg, 1), cudaMemcpyHostToDevice, st));
  GB_CUDA(cudaMemcpyAsync(b->off_d, b->off_h, sizeof(int) * (clusters + 1), cudaMemcpyHostToDevice, st));
  GB_CUDA(cudaMemcpyAsync(b->nparts_d, b->nparts_h, sizeof(int) * std::max(b->n, 1), cudaMemcpyHostToDevice, st));
  b->sched = want;
  return GBCCA_OK;
}

// The Phi images of a batch member (h1 of the batch); nothing once the plan
// has finished.
int tc_batch_pre(const TcBatch* b, Plan& p, cudaStream_t st) {
  return tc_phi_image(p, b->h1, st, &p.st->done, nullptr);
}

// The same for all n plans of the table, a few plans per launch, from the
// callers' blocks (two views: only CCA plans are batched); the plans' flags are
// cleared, so that the pass serves all of them.
int tc_batch_pre_all(const TcBatch* b, Plan* const* plans, int n, const PassIO* io, cudaStream_t st) {
  for (int i0 = 0; i0 < n; i0 += tc::kManyPlans) {
    const int m = std::min(tc::kManyPlans, n - i0);
    tc::Images<tc::kManyPlans> a{};
    int blocks = 1;
    for (int i = 0; i < m; ++i) {
      a.a[i] = tc_image_args(*plans[i0 + i], b->h1, nullptr, &io[i0 + i]);
      a.a[i].restart = &plans[i0 + i]->st->done;
      blocks = std::max(blocks, tc_image_blocks(*plans[i0 + i]));
    }
    tc::phi_image_kernel<tc::kManyPlans><<<dim3(blocks, 2, m), 256, 0, st>>>(a);
    GB_CHECK_LAUNCH();
  }
  return GBCCA_OK;
}

// One launch over every scheduled tile of the batch.
int tc_batch_launch(TcBatch* b, cudaStream_t st, cudaEvent_t e0, cudaEvent_t e1) {
  if (b->two != nullptr) {
    if (e0 != nullptr) GB_CUDA(record_timing_event(e0, st));
    GB_TRY(two::batch_launch(b->two, b->err_d, st));
    if (e1 != nullptr) GB_CUDA(record_timing_event(e1, st));
    return GBCCA_OK;
  }
  tc::Args a{};
  a.err = b->err_d;
  a.insts = b->inst_d;
  a.segs = b->seg_d;
  a.seg_off = b->off_d;
  auto kern = b->h1 == 20 ? tc::tc_pass_kernel<20> : tc::tc_pass_kernel<tc::kHalfMax>;
  const int smem = b->h1 == 20 ? tc::Lay<20>::kSmemBytes : tc::Lay<tc::kHalfMax>::kSmemBytes;
  GB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(tc::kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(2 * std::max(1, b->clusters), 1, 1);
  // the tensor-map parameters are unused in batch mode; any valid map will do
  const CUtensorMap* m0 = &b->inst_h[0].map[0];
  const CUtensorMap* m1 = &b->inst_h[0].map[1];
  if (e0 != nullptr) GB_CUDA(record_timing_event(e0, st));
  GB_CUDA(cudaLaunchKernelEx(&cfg, kern, *m0, *m1, a));
  GB_CHECK_LAUNCH();
  if (e1 != nullptr) GB_CUDA(record_timing_event(e1, st));
  return GBCCA_OK;
}

// Slab counts of plan i in the device tables (two sweeps: 16, per view and pair).
static const int* tc_batch_nparts(const TcBatch* b, int i) {
  return b->two != nullptr ? b->two->np_d + 16 * i : b->nparts_d + i;
}

// Sum of plan i's slabs into its G, then its Grams.
int tc_batch_post(const TcBatch* b, int i, Plan& p, cudaStream_t st, const int* done) {
  tc::Posts<1> m{};
  m.a[0] = tc_post_args(p, nullptr, tc_batch_nparts(b, i), done, nullptr);
  Plan* one = &p;
  return tc_post_launch<1>(m, &one, 1, st);
}

// The same for all n plans of the table, a few plans per launch, into the
// callers' buffers.
int tc_batch_post_all(const TcBatch* b, Plan* const* plans, int n, const PassIO* io, cudaStream_t st) {
  for (int i0 = 0; i0 < n; i0 += tc::kManyPlans) {
    const int c = std::min(tc::kManyPlans, n - i0);
    tc::Posts<tc::kManyPlans> m{};
    for (int i = 0; i < c; ++i)
      m.a[i] = tc_post_args(*plans[i0 + i], nullptr, tc_batch_nparts(b, i0 + i), nullptr, &io[i0 + i]);
    GB_TRY(tc_post_launch<tc::kManyPlans>(m, plans + i0, c, st));
  }
  return GBCCA_OK;
}

}  // namespace gbcca
