// Sketching transforms S Z for the preconditioner (Sec. 3, App. A).
//
// CountSketch (Sec. 3): row i of Z, times g(i) = +-1, is added into row h(i)
// of S Z.  The rows are first grouped by bucket with a stable counting sort
// (per-chunk counters, a bucket-major prefix sum, then an in-order placement
// with warp match), and each bucket is summed by one warp in row order in
// FP64, so the sketch is bitwise reproducible.
//
// SRHT (App. A, Def. A.1, scale sqrt(n/s) so that E[S^T S] = I): the
// Walsh-Hadamard transform of length n_pad = 2^m factors as
// H_{2^m} = H_{N2} (x) H_{N1}; stage 1 transforms each block of N1 consecutive
// rows in registers, stage 2 transforms the strided columns of the intermediate
// and writes only the s sampled rows.
#include "plan.h"

namespace gbcca {

// --------------------------------------------------------------- draws
__device__ __forceinline__ uint64_t feistel_even(uint64_t x, int bits, uint64_t key) {
  const int half = bits / 2;
  const uint64_t mask = (1ull << half) - 1ull;
  uint64_t L = (x >> half) & mask, R = x & mask;
  for (int r = 0; r < 4; ++r) {
    uint64_t F = sm64(key, (uint64_t)r ^ (R << 8)) & mask;
    uint64_t nL = R, nR = L ^ F;
    L = nL;
    R = nR;
  }
  return (L << half) | R;
}

__global__ void draw_countsketch_kernel(int64_t n, int64_t s, uint64_t seed, int32_t* h, int8_t* g) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t r = sm64(seed, (uint64_t)i);
    h[i] = (int32_t)(((r >> 32) * (uint64_t)s) >> 32);
    g[i] = (r & 1ull) ? (int8_t)-1 : (int8_t)1;
  }
}

__global__ void draw_srht_kernel(int64_t n_pad, int m, int64_t s, uint64_t seed, int32_t* rows, int8_t* signs,
                                 int* flag) {
  const uint64_t kd = seed ^ kSaltSigns, kr = seed ^ kSaltRows;
  const int bits = (m % 2 == 0) ? m : m + 1;
  const uint64_t lim = 1ull << m;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_pad; i += (int64_t)gridDim.x * blockDim.x) {
    signs[i] = (sm64(kd, (uint64_t)i) & 1ull) ? (int8_t)-1 : (int8_t)1;
    if (i < s) {
      uint64_t y = feistel_even((uint64_t)i, bits, kr);
      // cycle walking: the orbit of i under the permutation returns to i < 2^m,
      // so the loop ends; the bound only guards against a broken build.
      int guard = 0;
      while (y >= lim && guard < (1 << 22)) {
        y = feistel_even(y, bits, kr);
        ++guard;
      }
      if (y >= lim && flag != nullptr) atomicExch(flag, kFlagDraw);
      rows[i] = (int32_t)y;
    }
  }
}

int sketch_draws(int kind, int64_t n, int64_t s, uint64_t seed, int32_t* h, int8_t* g, cudaStream_t st) {
  if (kind == GBCCA_SKETCH_COUNTSKETCH) {
    draw_countsketch_kernel<<<std::min(ceil_div(n, 256), 8192), 256, 0, st>>>(n, s, seed, h, g);
    GB_CHECK_LAUNCH();
    return GBCCA_OK;
  }
  if (kind == GBCCA_SKETCH_SRHT) {
    int m = 0;
    while ((1ll << m) < n) ++m;
    if ((1ll << m) != n || s > n) {
      set_last_error("SRHT draws need n a power of two and s <= n");
      return GBCCA_ERR_INVALID_ARG;
    }
    draw_srht_kernel<<<std::min(ceil_div(n, 256), 8192), 256, 0, st>>>(n, m, s, seed, h, g, nullptr);
    GB_CHECK_LAUNCH();
    return GBCCA_OK;
  }
  set_last_error("unknown sketch kind");
  return GBCCA_ERR_INVALID_ARG;
}

// ---------------------------------------------------- CountSketch sort
__global__ void cs_count_kernel(const int32_t* __restrict__ h, int64_t n, int64_t rpc, int64_t s,
                                int32_t* __restrict__ tab, int* flag) {
  const int64_t r0 = blockIdx.x * rpc, r1 = min(n, r0 + rpc);
  for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
    int32_t b = h[i];
    if (b < 0 || b >= s) {
      atomicExch(flag, kFlagBucket);
      continue;
    }
    atomicAdd(&tab[(int64_t)blockIdx.x * s + b], 1);
  }
}

// per bucket: exclusive prefix over chunks (in place) and the bucket total;
// eight loads in flight (one at a time behind its own store took 48 us for
// 152 chunks of 2336 buckets)
__global__ void cs_colscan_kernel(int32_t* __restrict__ tab, int nch, int64_t s, int32_t* __restrict__ total) {
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < s; b += (int64_t)gridDim.x * blockDim.x) {
    int32_t acc = 0;
    for (int c0 = 0; c0 < nch; c0 += 8) {
      int32_t t[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) t[u] = c0 + u < nch ? tab[(int64_t)(c0 + u) * s + b] : 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (c0 + u < nch) tab[(int64_t)(c0 + u) * s + b] = acc;
        acc += t[u];
      }
    }
    total[b] = acc;
  }
}

// exclusive scan of total[0..s) into off[0..s] by one CTA of 1024 threads
__global__ void cs_scan_kernel(const int32_t* __restrict__ total, int64_t s, int32_t* __restrict__ off) {
  __shared__ int32_t buf[1024];
  __shared__ int32_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t base = 0; base < s; base += 1024) {
    int64_t i = base + threadIdx.x;
    int32_t v = i < s ? total[i] : 0;
    buf[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
      int32_t t = threadIdx.x >= o ? buf[threadIdx.x - o] : 0;
      __syncthreads();
      buf[threadIdx.x] += t;
      __syncthreads();
    }
    if (i < s) off[i] = carry + buf[threadIdx.x] - v;
    __syncthreads();
    if (threadIdx.x == 1023) carry += buf[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) off[s] = carry;
}

// in-order placement: one warp walks its chunk 32 rows at a time; rows of
// the same bucket inside a group of 32 are ranked by lane (= row) order.
// The chunk's next free place of every bucket is a shared-memory counter
// where s counters fit (kSmem), since a step depends on the counters of the
// step before it (through global memory: 44 us for 1974 rows a chunk); the
// buckets of the next kPlaceAhead groups are loaded ahead of that chain.
constexpr int kPlaceAhead = 8;
constexpr int64_t kPlaceSmem = 48 * 1024;  // counters in shared memory up to s = 12288
template <bool kSmem>
__global__ void __launch_bounds__(32) cs_place_kernel(const int32_t* __restrict__ h, int64_t n, int64_t rpc, int64_t s,
                                                      int32_t* __restrict__ tab, const int32_t* __restrict__ off,
                                                      int32_t* __restrict__ perm) {
  extern __shared__ int32_t cnt_s[];
  const int lane = threadIdx.x;
  const int64_t r0 = blockIdx.x * rpc, r1 = min(n, r0 + rpc);
  int32_t* cur = tab + (int64_t)blockIdx.x * s;
  if (kSmem) {
    for (int b = lane; b < (int)s; b += 32) cnt_s[b] = off[b] + cur[b];
    __syncwarp();
  }
  for (int64_t g0 = r0; g0 < r1; g0 += 32 * kPlaceAhead) {
    int32_t bv[kPlaceAhead];
#pragma unroll
    for (int u = 0; u < kPlaceAhead; ++u) {
      const int64_t i = g0 + 32 * u + lane;
      bv[u] = i < r1 ? h[i] : -1;
      if (bv[u] < 0 || bv[u] >= s) bv[u] = -1;  // reported by cs_count_kernel
    }
#pragma unroll
    for (int u = 0; u < kPlaceAhead; ++u) {
      const int64_t i = g0 + 32 * u + lane;
      const int32_t b = bv[u];
      const unsigned peers = __match_any_sync(0xffffffffu, b);
      const bool act = b >= 0;
      const bool last = act && (peers >> lane) == 1u;  // highest lane of its group
      if (act) {
        const int rank = __popc(peers & ((1u << lane) - 1u));
        perm[(kSmem ? cnt_s[b] : off[b] + cur[b]) + rank] = (int32_t)i;
      }
      __syncwarp();
      if (last) (kSmem ? cnt_s[b] : cur[b]) += __popc(peers);
      __syncwarp();
    }
  }
}

int countsketch_prepare(Plan& p, cudaStream_t st) {
  const int64_t rpc = (p.n + p.cs_nch - 1) / p.cs_nch;
  GB_CUDA(cudaMemsetAsync(p.cs_tab, 0, sizeof(int32_t) * (size_t)p.cs_nch * p.s, st));
  cs_count_kernel<<<p.cs_nch, 256, 0, st>>>(p.h, p.n, rpc, p.s, p.cs_tab, p.flag);
  GB_CHECK_LAUNCH();
  int32_t* total = p.perm;  // borrow perm as scratch for the bucket totals (n >= s)
  cs_colscan_kernel<<<ceil_div(p.s, 256), 256, 0, st>>>(p.cs_tab, p.cs_nch, p.s, total);
  GB_CHECK_LAUNCH();
  cs_scan_kernel<<<1, 1024, 0, st>>>(total, p.s, p.cs_off);
  GB_CHECK_LAUNCH();
  const size_t csm = sizeof(int32_t) * (size_t)p.s;
  if ((int64_t)csm <= kPlaceSmem)
    cs_place_kernel<true><<<p.cs_nch, 32, csm, st>>>(p.h, p.n, rpc, p.s, p.cs_tab, p.cs_off, p.perm);
  else
    cs_place_kernel<false><<<p.cs_nch, 32, 0, st>>>(p.h, p.n, rpc, p.s, p.cs_tab, p.cs_off, p.perm);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// x times a sign outside +-1 (a caller's own draws); out of line, so that the
// usual signs cost no FP64 instruction
static __device__ __noinline__ double scale_by(double x, int sg) { return (double)sg * x; }

// kV consecutive values of a row: one 16- or 8-byte load
template <typename Tin, int kV> struct alignas(sizeof(Tin) * kV) RowVec { Tin v[kV]; };

// One warp per (bucket, 32 kV columns): lane l owns kV consecutive columns and
// adds the bucket's rows in row order, so the sums do not depend on the grid.
// The order and signs of a bucket's rows are read 32 at a time and handed out
// by shuffles, kCsRows rows' values in flight per lane.  Bound by the FP64
// rate: one addition per element (two with class means), the sign applied to
// the bits.  A warp per bucket over all columns, one row at a time behind its
// index, with a conversion and a multiply-add per element took 1310 us for
// 300000 x 384 FP32.  kV = 1 serves rows that are not aligned for the wide load.
constexpr int kCsRows = 4;
template <typename Tin, int kV, bool kCentre>
__global__ void __launch_bounds__(256)
cs_sum_kernel(const Tin* __restrict__ Z, int64_t ld, int d, int64_t s, int ncol, const int32_t* __restrict__ off,
              const int32_t* __restrict__ perm, const int8_t* __restrict__ g, const int32_t* __restrict__ labels,
              const double* __restrict__ means, double* __restrict__ SZ) {
  const int lane = threadIdx.x & 31;
  const int64_t w = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
  const int64_t b = w / ncol;
  if (b >= s) return;
  const int c = ((int)(w - b * ncol) * 32 + lane) * kV;
  const int nv = min(kV, d - c);  // columns of this lane (none: nv <= 0)
  double acc[kV];
#pragma unroll
  for (int q = 0; q < kV; ++q) acc[q] = 0.0;
  const int32_t p1 = off[b + 1];
  for (int32_t pos = off[b]; pos < p1; pos += 32) {
    const int cnt = min(32, p1 - pos);
    const int32_t ri = lane < cnt ? perm[pos + lane] : 0;
    const int rs = lane < cnt ? (int)g[ri] : 0;
    const int rl = kCentre && lane < cnt ? labels[ri] : 0;
    for (int r0 = 0; r0 < cnt; r0 += kCsRows) {
      RowVec<Tin, kV> z[kCsRows];
      double m[kCsRows][kCentre ? kV : 1];
      int sg[kCsRows];
#pragma unroll
      for (int u = 0; u < kCsRows; ++u) {
        const int r = min(r0 + u, cnt - 1);
        const int64_t i = __shfl_sync(0xffffffffu, ri, r);
        sg[u] = __shfl_sync(0xffffffffu, rs, r);
        const Tin* row = Z + i * ld + c;
        if (nv == kV) {
          z[u] = *reinterpret_cast<const RowVec<Tin, kV>*>(row);
        } else {
#pragma unroll
          for (int q = 0; q < kV; ++q) z[u].v[q] = q < nv ? row[q] : Tin(0.0f);
        }
        if (kCentre) {
          const double* mrow = means + (int64_t)__shfl_sync(0xffffffffu, rl, r) * d + c;
#pragma unroll
          for (int q = 0; q < kV; ++q) m[u][q] = q < nv ? mrow[q] : 0.0;
        }
      }
#pragma unroll
      for (int u = 0; u < kCsRows; ++u) {
        if (r0 + u < cnt) {
#pragma unroll
          for (int q = 0; q < kV; ++q) {
            double x = widen(z[u].v[q]);
            if (kCentre) x -= m[u][q];
            if (sg[u] == 1 || sg[u] == -1)  // uniform over the warp
              x = __hiloint2double(__double2hiint(x) ^ (sg[u] & 0x80000000), __double2loint(x));
            else
              x = scale_by(x, sg[u]);
            acc[q] += x;
          }
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < kV; ++q)
    if (q < nv) SZ[b * d + c + q] = acc[q];
}

template <typename Tin, int kV>
int cs_sum_run(Plan& p, View& v, bool center, cudaStream_t st) {
  const int ncol = ceil_div(v.d, 32 * kV);
  const int grid = ceil_div(p.s * ncol, 8);
  auto kern = center ? cs_sum_kernel<Tin, kV, true> : cs_sum_kernel<Tin, kV, false>;
  kern<<<grid, 256, 0, st>>>(static_cast<const Tin*>(v.Z), v.ld, v.d, p.s, ncol, p.cs_off, p.perm, p.g,
                             center ? p.labels : nullptr, center ? p.means : nullptr, v.SZ);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

// kV columns per lane where every row starts on a kV-element boundary
template <typename Tin, int kV>
int cs_sum_any(Plan& p, View& v, bool center, cudaStream_t st) {
  const bool vec = v.ld % kV == 0 && reinterpret_cast<uintptr_t>(v.Z) % (sizeof(Tin) * kV) == 0;
  return vec ? cs_sum_run<Tin, kV>(p, v, center, st) : cs_sum_run<Tin, 1>(p, v, center, st);
}

int countsketch_apply(Plan& p, int view, bool center, cudaStream_t st) {
  View& v = p.v[view];
  switch (p.dtype) {
    case GBCCA_FP64: return cs_sum_any<double, 2>(p, v, center, st);
    case GBCCA_FP32: return cs_sum_any<float, 4>(p, v, center, st);
    default: return cs_sum_any<__nv_bfloat16, 4>(p, v, center, st);
  }
}

// ---------------------------------------------------------------- SRHT
// Transform of length N < 64 (tiny n): one thread per column
template <typename T>
__device__ __forceinline__ void fwht_thread_col(T* col, int stride, int N) {
  for (int h = 1; h < N; h <<= 1)
    for (int i = 0; i < N; ++i)
      if ((i & h) == 0) {
        const T a = col[i * stride], b = col[(i + h) * stride];
        col[i * stride] = a + b;
        col[(i + h) * stride] = a - b;
      }
}

// The intermediate between the stages is stored as tiles of 32 columns,
// [residue a1][column block][row block][32], so that stage 2 reads one
// contiguous tile and stage 1's 128-byte rows of neighbouring row blocks lie
// side by side.

// Walsh-Hadamard transform of N = 32 NW rows (NW = 2 .. 32 warps) of 32 columns,
// lane = column: warp w holds rows 32 w .. 32 w + 31 in registers (spans 1 ..
// 16), the tile is exchanged once through shared memory, and the same warp
// then holds the residues w (32 / NW) .. of the row index modulo 32, NW rows
// each (spans 32 .. N / 2): about nine additions and two shared-memory
// accesses per element.  (A column per warp with shuffles for the first five
// levels and two passes over shared memory was bound by its instructions:
// 437 us a view for 262144 x 512 BF16, 1.8 TB/s.)  buf: N x kC, scratch; out(r,
// x) receives row r of the lane's column (each warp its own rows).  kC: columns
// of the tile; with 16 a half-warp takes the part of a warp.
template <typename T, int NW, int kC = 32, typename F>
__device__ __forceinline__ void fwht_tile(T (&v)[32], T* buf, F out) {
  const int lane = threadIdx.x % kC, w = threadIdx.x / kC;
#pragma unroll
  for (int h = 1; h < 32; h <<= 1) {
#pragma unroll
    for (int t = 0; t < 32; ++t)
      if ((t & h) == 0) {
        const T a = v[t], b = v[t + h];
        v[t] = a + b;
        v[t + h] = a - b;
      }
  }
#pragma unroll
  for (int t = 0; t < 32; ++t) buf[(32 * w + t) * kC + lane] = v[t];
  __syncthreads();
  constexpr int NJ = 32 / NW;  // residues of this warp: j = w NJ + q, rows j + 32 m
#pragma unroll
  for (int q = 0; q < NJ; ++q) {
    T u[NW];
#pragma unroll
    for (int m = 0; m < NW; ++m) u[m] = buf[(w * NJ + q + 32 * m) * kC + lane];
#pragma unroll
    for (int h = 1; h < NW; h <<= 1) {
#pragma unroll
      for (int m = 0; m < NW; ++m)
        if ((m & h) == 0) {
          const T a = u[m], b = u[m + h];
          u[m] = a + b;
          u[m + h] = a - b;
        }
    }
#pragma unroll
    for (int m = 0; m < NW; ++m) out(w * NJ + q + 32 * m, u[m]);
  }
}

// One element of D Z (signs, and the class means for LDA) in the working type.
template <typename Tin, typename T>
__device__ __forceinline__ T signed_value(Tin z, int g, const int32_t* labels, const double* means, int64_t row, int d,
                                          int col) {
  if (labels != nullptr) {
    const double x = to_f64(z) - means[(int64_t)labels[row] * d + col];
    return (T)(g < 0 ? -x : x);
  }
  const T x = to_work<T>(z);
  return g < 0 ? -x : x;
}

// Stage 1: per block of N1 = 32 NW consecutive rows and 32 columns, D Z then
// the N1-point transform along the rows.  All 32 loads of a thread are in
// flight together; a thread takes at most 64 registers (FP32 work), so that
// the loads of one CTA run under the transform and the stores of another (one
// CTA per SM: 323 us a view for 262144 x 512 BF16; two: 267 us, 3.0 TB/s).
template <typename Tin, typename T, int NW>
__global__ void __launch_bounds__(32 * NW, sizeof(T) == 4 ? 32 / NW : 16 / NW)
srht_stage1_kernel(const Tin* __restrict__ Z, int64_t ld, int64_t n, int d, const int8_t* __restrict__ sg,
                   const int32_t* __restrict__ labels, const double* __restrict__ means, T* __restrict__ Tmid) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf = reinterpret_cast<T*>(smem_raw);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t i2 = blockIdx.y, N2 = gridDim.y;
  const int cb = blockIdx.x, ncb = gridDim.x, col = 32 * cb + lane;
  const int64_t row0 = i2 * 32 * NW + 32 * w;
  // the signs of this warp's 32 rows (a zero drops the row)
  const int g = row0 + lane < n ? (int)sg[row0 + lane] : 0;
  const unsigned neg = __ballot_sync(0xffffffffu, g < 0), use = __ballot_sync(0xffffffffu, g != 0);
  Tin z[32];
  const Tin* src = Z + row0 * ld + col;
#pragma unroll
  for (int t = 0; t < 32; ++t) z[t] = (use >> t & 1) && col < d ? src[(int64_t)t * ld] : Tin(0.0f);
  T v[32];
#pragma unroll
  for (int t = 0; t < 32; ++t)
    v[t] = (use >> t & 1) && col < d
               ? signed_value<Tin, T>(z[t], (neg >> t & 1) ? -1 : 1, labels, means, row0 + t, d, col)
               : T(0);
  // row r of the block is residue a1 = r: straight from registers, 128 bytes a
  // warp (back through shared memory first: 267 us a view, 255 now)
  fwht_tile<T, NW>(v, buf, [&](int r, T x) { Tmid[(((int64_t)r * ncb + cb) * N2 + i2) * 32 + lane] = x; });
}

// The same for short blocks (N1 < 64): one thread per column.
template <typename Tin, typename T>
__global__ void srht_stage1_small_kernel(const Tin* __restrict__ Z, int64_t ld, int64_t n, int d, int N1,
                                         const int8_t* __restrict__ sg, const int32_t* __restrict__ labels,
                                         const double* __restrict__ means, T* __restrict__ Tmid) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf = reinterpret_cast<T*>(smem_raw);
  const int lane = threadIdx.x;
  const int64_t i2 = blockIdx.y, N2 = gridDim.y;
  const int cb = blockIdx.x, ncb = gridDim.x, col = 32 * cb + lane;
  for (int r = 0; r < N1; ++r) {
    const int64_t row = i2 * N1 + r;
    const int g = row < n ? (int)sg[row] : 0;
    buf[r * 32 + lane] =
        g != 0 && col < d ? signed_value<Tin, T>(Z[row * ld + col], g, labels, means, row, d, col) : T(0);
  }
  fwht_thread_col<T>(buf + lane, 32, N1);
  for (int r = 0; r < N1; ++r) Tmid[(((int64_t)r * ncb + cb) * N2 + i2) * 32 + lane] = buf[r * 32 + lane];
}

// Sampled rows of the transform of residue a1, columns c0 .. c0 + kC - 1: SZ[j] =
// scale * row (rows[j] >> m1).
template <typename T, int kC = 32>
__device__ __forceinline__ void srht_pick(const T* buf, int d, int c0, int a1, int nsel, int m1, const int32_t* off1,
                                          const int32_t* list, const int32_t* rows, double scale, double* SZ) {
  for (int e = threadIdx.x; e < nsel * kC; e += blockDim.x) {
    const int q = e / kC, c = c0 + e % kC;
    const int j = list[off1[a1] + q];
    if (c < d) SZ[(int64_t)j * d + c] = scale * (double)buf[(rows[j] >> m1) * kC + e % kC];
  }
}

// Columns of a CTA of stage 2: a whole tile of the intermediate, or half of one
// where 32 columns do not fit shared memory (FP64 of 1024 rows: 262144 bytes of
// the 232448).
template <typename T, int NW> constexpr int kStage2Cols = sizeof(T) * 32 * NW * 32 > 232448 ? 16 : 32;

// Stage 2: for one residue a1 of the low m1 row bits, the N2-point transform
// across the row blocks of each column, kept only at the sampled rows and
// scaled by sqrt(n'/s) / sqrt(n') = 1 / sqrt(s) (App. A).
template <typename T, int NW>
__global__ void __launch_bounds__(kStage2Cols<T, NW> * NW)
srht_stage2_kernel(const T* __restrict__ Tmid, int d, int m1, const int32_t* __restrict__ off1,
                   const int32_t* __restrict__ list, const int32_t* __restrict__ rows, double scale,
                   double* __restrict__ SZ) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf = reinterpret_cast<T*>(smem_raw);
  constexpr int kC = kStage2Cols<T, NW>, kPer = 32 / kC;  // CTAs of a tile
  const int a1 = blockIdx.y, cb = blockIdx.x / kPer, ncb = gridDim.x / kPer, first = kC * (blockIdx.x % kPer);
  const int nsel = off1[a1 + 1] - off1[a1];
  if (nsel == 0) return;
  const int lane = threadIdx.x % kC, w = threadIdx.x / kC;
  const T* src = Tmid + ((int64_t)a1 * ncb + cb) * (32 * NW) * 32 + first;
  T v[32];
#pragma unroll
  for (int t = 0; t < 32; ++t) v[t] = src[(32 * w + t) * 32 + lane];
  fwht_tile<T, NW, kC>(v, buf, [&](int r, T x) { buf[r * kC + lane] = x; });
  __syncthreads();
  srht_pick<T, kC>(buf, d, 32 * cb + first, a1, nsel, m1, off1, list, rows, scale, SZ);
}

template <typename T>
__global__ void srht_stage2_small_kernel(const T* __restrict__ Tmid, int d, int N2, int m1,
                                         const int32_t* __restrict__ off1, const int32_t* __restrict__ list,
                                         const int32_t* __restrict__ rows, double scale, double* __restrict__ SZ) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf = reinterpret_cast<T*>(smem_raw);
  const int a1 = blockIdx.y, cb = blockIdx.x, ncb = gridDim.x;
  const int nsel = off1[a1 + 1] - off1[a1];
  if (nsel == 0) return;
  const T* src = Tmid + ((int64_t)a1 * ncb + cb) * N2 * 32;
  for (int r = 0; r < N2; ++r) buf[r * 32 + threadIdx.x] = src[r * 32 + threadIdx.x];
  fwht_thread_col<T>(buf + threadIdx.x, 32, N2);
  __syncwarp();
  srht_pick(buf, d, 32 * cb, a1, nsel, m1, off1, list, rows, scale, SZ);
}

// group the sampled rows by their low m1 bits (order within a group is free:
// every sampled row writes its own output row)
__global__ void srht_group_kernel(const int32_t* __restrict__ rows, int64_t s, int N1, int32_t* __restrict__ cnt,
                                  int32_t* __restrict__ off1, int32_t* __restrict__ list, int phase) {
  if (phase == 0) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < s; j += (int64_t)gridDim.x * blockDim.x)
      atomicAdd(&cnt[rows[j] & (N1 - 1)], 1);
  } else if (phase == 1) {
    // exclusive scan of the N1 counts by one warp: lane l sums a contiguous
    // run of the counts, the lanes' totals are scanned by shuffles, then
    // each lane writes its run's offsets (and clears its counts)
    if (blockIdx.x == 0 && threadIdx.x < 32) {
      const int lane = threadIdx.x;
      const int per = (N1 + 31) / 32;
      const int a0 = min(N1, lane * per), a1 = min(N1, a0 + per);
      int32_t tot = 0;
      for (int a = a0; a < a1; ++a) tot += cnt[a];
      int32_t inc = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      int32_t acc = inc - tot;
      for (int a = a0; a < a1; ++a) {
        off1[a] = acc;
        acc += cnt[a];
        cnt[a] = 0;
      }
      if (lane == 31) off1[N1] = inc;
    }
  } else {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < s; j += (int64_t)gridDim.x * blockDim.x) {
      int a = rows[j] & (N1 - 1);
      int pos = atomicAdd(&cnt[a], 1);
      list[off1[a] + pos] = (int32_t)j;
    }
  }
}

template <typename Tin, typename T, int NW>
int srht_stage1(const View& v, const Plan& p, int N2, const int32_t* lab, T* Tmid, cudaStream_t st) {
  const size_t sm = sizeof(T) * 32 * NW * 32;
  auto k1 = srht_stage1_kernel<Tin, T, NW>;
  GB_CUDA(cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  k1<<<dim3(ceil_div(v.d, 32), N2), 32 * NW, sm, st>>>((const Tin*)v.Z, v.ld, p.n, v.d, p.g, lab, p.means, Tmid);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

template <typename T, int NW>
int srht_stage2(const View& v, const Plan& p, int N1, int m1, const int32_t* off1, const int32_t* list, const T* Tmid,
                cudaStream_t st) {
  constexpr int kC = kStage2Cols<T, NW>;
  const size_t sm = sizeof(T) * 32 * NW * kC;
  auto k2 = srht_stage2_kernel<T, NW>;
  GB_CUDA(cudaFuncSetAttribute(k2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  k2<<<dim3(32 / kC * ceil_div(v.d, 32), N1), kC * NW, sm, st>>>(Tmid, v.d, m1, off1, list, p.h, 1.0 / sqrt((double)p.s), v.SZ);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

template <typename Tin, typename T>
int srht_run(Plan& p, View& v, cudaStream_t st) {
  int m = 0;
  while ((1ll << m) < p.n_pad) ++m;
  const int m1 = std::min(m, 9), m2 = m - m1;
  const int N1 = 1 << m1, N2 = 1 << m2;
  if (N2 > 1024) {
    set_last_error("SRHT supports n <= 2^19");
    return GBCCA_ERR_UNSUPPORTED;
  }
  T* Tmid = reinterpret_cast<T*>(p.srht_T);
  const int32_t* lab = p.kind == kLDA ? p.labels : nullptr;
  switch (N1) {
    case 64: GB_TRY((srht_stage1<Tin, T, 2>(v, p, N2, lab, Tmid, st))); break;
    case 128: GB_TRY((srht_stage1<Tin, T, 4>(v, p, N2, lab, Tmid, st))); break;
    case 256: GB_TRY((srht_stage1<Tin, T, 8>(v, p, N2, lab, Tmid, st))); break;
    case 512: GB_TRY((srht_stage1<Tin, T, 16>(v, p, N2, lab, Tmid, st))); break;
    default:
      srht_stage1_small_kernel<Tin, T><<<dim3(ceil_div(v.d, 32), N2), 32, sizeof(T) * 32 * N1, st>>>(
          (const Tin*)v.Z, v.ld, p.n, v.d, N1, p.g, lab, p.means, Tmid);
      GB_CHECK_LAUNCH();
  }
  int32_t* cnt = p.cs_tab;
  int32_t* off1 = p.cs_off;
  int32_t* list = p.perm;
  GB_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int32_t) * N1, st));
  srht_group_kernel<<<ceil_div(p.s, 256), 256, 0, st>>>(p.h, p.s, N1, cnt, off1, list, 0);
  GB_CHECK_LAUNCH();
  srht_group_kernel<<<1, 32, 0, st>>>(p.h, p.s, N1, cnt, off1, list, 1);
  GB_CHECK_LAUNCH();
  srht_group_kernel<<<ceil_div(p.s, 256), 256, 0, st>>>(p.h, p.s, N1, cnt, off1, list, 2);
  GB_CHECK_LAUNCH();
  switch (N2) {
    case 64: return srht_stage2<T, 2>(v, p, N1, m1, off1, list, Tmid, st);
    case 128: return srht_stage2<T, 4>(v, p, N1, m1, off1, list, Tmid, st);
    case 256: return srht_stage2<T, 8>(v, p, N1, m1, off1, list, Tmid, st);
    case 512: return srht_stage2<T, 16>(v, p, N1, m1, off1, list, Tmid, st);
    case 1024: return srht_stage2<T, 32>(v, p, N1, m1, off1, list, Tmid, st);
  }
  srht_stage2_small_kernel<T><<<dim3(ceil_div(v.d, 32), N1), 32, sizeof(T) * 32 * N2, st>>>(
      Tmid, v.d, N2, m1, off1, list, p.h, 1.0 / sqrt((double)p.s), v.SZ);
  GB_CHECK_LAUNCH();
  return GBCCA_OK;
}

int srht_apply(Plan& p, int view, cudaStream_t st) {
  View& v = p.v[view];
  switch (p.dtype) {
    case GBCCA_FP64: return srht_run<double, double>(p, v, st);
    case GBCCA_FP32: return srht_run<float, float>(p, v, st);
    default: return srht_run<__nv_bfloat16, float>(p, v, st);
  }
}

}  // namespace gbcca
