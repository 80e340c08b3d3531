// The two-sweep tensor-core pass (pass_two.cu) as pass_tc.cu drives it.
#pragma once
#include <new>
#include <vector>

#include "tc_ptx.cuh"

namespace gbcca {
namespace tc {
// Rows of a view in a partial slab: padded so that a block of kPostRows rows
// belongs to one view and starts on a 16-byte boundary.  The padding is never
// written and its sums are never used.
constexpr int kPostRows = 4;
__host__ __device__ __forceinline__ int pad_rows(int d) { return (d + kPostRows - 1) / kPostRows * kPostRows; }
}  // namespace tc

namespace two {

constexpr int kMaxPairs = 3;  // 128-column pairs of a block (TMEM: 3 x 160 columns at most)

// One plan's pass (in a batch: device memory; the tensor maps are read by the
// TMA unit from there, and carry their own alignment).
struct Inst {
  CUtensorMap map[2];      // the streamed views (boxes of 64 rows x 64 columns)
  const uint8_t* phi_img;  // [view][64-column box][2h][128 B], pre-swizzled
  int64_t img_view;
  uint8_t* wimg;           // [64-row tile][2 nw][128 B]
  float* part;             // partial slabs
  int64_t slab;            // floats of one
  const int* done;         // convergence flag: skip the instance when set
  int d[2];
  int nv;
  int ncol;                // columns of Phi per view (2k)
  int nw;                  // operand rows of one part (hi or lo): nv ncol rounded up to 8
  int pair_sum;            // rows 2i, 2i + 1 are the hi and lo parts of one data row
  int ntiles;              // 64-row tiles
  long long wait;          // cycles of one pipeline wait before the CTA gives up
};

// A contiguous range of an instance's 64-row tiles (sweep 2: of one block,
// summed into partial slab `slab`).
struct Seg {
  int inst, first, count, slab, block;
};

struct Args {
  const Inst* insts;    // null: the kernel's instance parameter
  const Seg* segs;
  const int* seg_off;   // [CTA + 1]
  int* err;
  int h;                // Phi image rows per half (sweep 1)
  int stages, stage_bytes;
  int nblk;             // over one instance: its blocks (sweep 1: one), CTAs cta0[b] .. cta0[b + 1] - 1 each
  int cta0[8];
  int nseg[8];          // and the ranges of tiles (slabs) per CTA of a block
};

// A view of P pairs is cut into ceil(P / 3) blocks of near-equal size; view
// 0's blocks come first.
__host__ __device__ __forceinline__ int block_count(const int* d, int nv) {
  int n = 0;
  for (int v = 0; v < nv; ++v) n += ((d[v] + 127) / 128 + kMaxPairs - 1) / kMaxPairs;
  return n;
}
__host__ __device__ __forceinline__ void block_of(const int* d, int nv, int b, int* view, int* pair0, int* np) {
  const int P0 = (d[0] + 127) / 128, n0 = (P0 + kMaxPairs - 1) / kMaxPairs;
  const int v = b < n0 || nv < 2 ? 0 : 1;
  const int P = v == 0 ? P0 : (d[1] + 127) / 128, n = (P + kMaxPairs - 1) / kMaxPairs, i = v == 0 ? b : b - n0;
  const int base = P / n, rem = P - base * n;
  *view = v;
  *pair0 = i * base + (i < rem ? i : rem);
  *np = base + (i < rem ? 1 : 0);
}

// One plan: W, then G; np[8 view + pair] receives the slabs written per pair
// (at most max_slabs).
int sweep_w(const Inst& one, int h, int* err, int sm_count, cudaStream_t st);
int sweep_g(const Inst& one, int* err, int sm_count, int max_slabs, int* np, cudaStream_t st);

// Several plans in the same two launches, over schedules in device memory.
struct Batch {
  int n = 0, h = 8, nw = 8, sm = 0, max_segs = 0, ctas = 1;
  Inst* inst_h = nullptr;  // pinned host copies of the tables
  Inst* inst_d = nullptr;
  Seg* seg_h[2] = {nullptr, nullptr};
  Seg* seg_d[2] = {nullptr, nullptr};
  int* off_h[2] = {nullptr, nullptr};
  int* off_d[2] = {nullptr, nullptr};
  int* np_h = nullptr;     // slabs per (instance, view, pair)
  int* np_d = nullptr;
};
Batch* batch_create(const std::vector<Inst>& insts, int h, int sm, cudaStream_t st, int* rc);
void batch_destroy(Batch* b);
int batch_schedule(Batch* b, const bool* active, int ctas, cudaStream_t st);
int batch_launch(const Batch* b, int* err, cudaStream_t st);

}  // namespace two
}  // namespace gbcca
