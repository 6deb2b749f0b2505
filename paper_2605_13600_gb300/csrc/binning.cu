// binning.cu -- tile binning of one view's projected Gaussians.
//
// Every visible Gaussian is listed in the 16x16 tiles of its rectangle (the
// 3DGS rule: membership is tile-granular).  The rectangles here are the 3DGS
// rectangles cut to the bounding box of each Gaussian's alpha >= 1/255
// ellipse (by the projection): a dropped tile holds no pixel that passes the
// alpha test, so the composite is unchanged.  There is a list per block of
// 2 x 2 tiles (TileList, scoup_internal.cuh); lists are left unordered here and
// ordered front to back (depth, then index) inside the tile kernels.
//
// The Gaussians arrive in spatial (Morton) order, so one CTA's group covers a
// compact set of blocks; of the group (512 or 1024 Gaussians) it takes those
// whose kept bit is set: all listed ones, or those in front of the depth cut
// (a tenth of a 1M-Gaussian scene).  Counting is privatised per CTA in
// shared memory over the group's bounding box in blocks; the counting pass
// reserves the CTA's run in each list right away (one global atomic per (CTA,
// list)) and keeps the run's offset, so the filling pass expands the items
// only once and writes each CTA's keys of a list into one contiguous run.
// Rectangles larger than kBigRect blocks go to separate global counters and are
// placed after the reserved runs.
//
// Every kernel takes a chunk of views (blockIdx.y).  The second pass of a view
// lists only into the blocks with a tile recorded as open; a rectangle's other
// blocks are skipped.
#include "scoup_internal.cuh"

namespace scoup {
namespace {

constexpr int kBinThreads = 256;
constexpr int kGroupMax = 1024;  // most Gaussians of one CTA (bin_group)
constexpr int kLocalMax = 4096;  // blocks of the per-CTA bounding box kept in shared memory
constexpr int kBigRect = 256;
constexpr unsigned kFull = 0xffffffffu;

// The rectangle of blocks that a rectangle of tiles meets.
__device__ __forceinline__ ushort4 block_rect(const ushort4& r, int shift) {
  return make_ushort4(r.x >> shift, r.y >> shift, (r.z + shift) >> shift, (r.w + shift) >> shift);
}

// Blocks that a pass does not list into: none in the first, those without an open tile in the second.
struct BlockSkip {
  const uint32_t* bits;  // null: no tile is skipped
  int ow;
  __device__ __forceinline__ bool operator()(int tx, int ty) const {
    return bits && !((bits[ty * ow + (tx >> 5)] >> (tx & 31)) & 1u);
  }
};

// Positions (in the group) of the kept Gaussians of group [base, base + group),
// ascending, into list; returns their number.  Block-wide.
__device__ int kept_list(const ViewJob& v, int64_t base, uint16_t* list) {
  __shared__ int s_total;
  if (threadIdx.x < 32) {
    // one word of 32 kept bits per lane covers the largest group
    const int lane = threadIdx.x;
    uint32_t w = (lane < v.group >> 5 && base + 32 * lane < v.n) ? v.keep[(base >> 5) + lane] : 0u;
    const int c = __popc(w);
    int incl = c;
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, off);
      if (lane >= off) incl += y;
    }
    int at = incl - c;
    for (; w != 0u; w &= w - 1u) list[at++] = (uint16_t)(32 * lane + __ffs(w) - 1);
    if (lane == 31) s_total = incl;
  }
  __syncthreads();
  return s_total;
}

struct LocalBox {
  int x0, y0, w, h;
  bool ok;
  __device__ __forceinline__ int idx(int tx, int ty) const { return (ty - y0) * w + (tx - x0); }
};

__device__ __forceinline__ bool big(const ushort4& r) { return (r.z - r.x) * (r.w - r.y) > kBigRect; }

// Warp-cooperative expansion of the (Gaussian, list) items of the 32 Gaussians
// held by the lanes (lane l holds rectangle r, in blocks of tiles where the
// lists are blocks'): the items are
// numbered by an exclusive scan of the rectangle areas and dealt out 32 at a
// time, one per lane, so every lane works on one item per round whatever the
// rectangle sizes.  f(src_lane, tx, ty) is called for each item.
// q = local / w for 0 <= local < 2^22, 1 <= w: (local + 0.5) / w lies at
// least 0.5 / w away from an integer, far more than the error of the
// approximate quotient, so truncation gives the exact integer quotient.
__device__ __forceinline__ int div_small(int local, int w) {
  return local < (1 << 22) ? (int)__fdividef((float)local + 0.5f, (float)w) : local / w;
}

template <typename F>
__device__ __forceinline__ void expand_items(const ushort4& r, F&& f) {
  const int lane = threadIdx.x & 31;
  const int w = r.z > r.x ? r.z - r.x : 0, h = r.w > r.y ? r.w - r.y : 0;
  const int c = w * h;
  int incl = c;
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(kFull, incl, off);
    if (lane >= off) incl += y;
  }
  const int total = __shfl_sync(kFull, incl, 31);
  const int excl = incl - c;
  const int packed = (int)r.x | ((int)r.y << 16);
  for (int k0 = 0; k0 < total; k0 += 32) {
    const int item = k0 + lane;
    int src = 0;  // largest lane whose first item is <= item (it owns the item)
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
      const int e = __shfl_sync(kFull, excl, src + step);
      if (e <= item) src += step;
    }
    const int e_src = __shfl_sync(kFull, excl, src);
    const int w_src = __shfl_sync(kFull, w, src);
    const int p_src = __shfl_sync(kFull, packed, src);
    if (item < total) {
      const int local = item - e_src;
      const int yy = div_small(local, w_src);
      f(src, (p_src & 0xffff) + (local - yy * w_src), (p_src >> 16) + yy);
    }
  }
}

// Block-wide bounding box of the group's kept, non-big rectangles.
__device__ LocalBox group_box(const ushort4* __restrict__ rects, const uint16_t* list, int m, int shift) {
  __shared__ int s_box[4];
  if (threadIdx.x == 0) { s_box[0] = 1 << 30; s_box[1] = 1 << 30; s_box[2] = 0; s_box[3] = 0; }
  __syncthreads();
  int x0 = 1 << 30, y0 = 1 << 30, x1 = 0, y1 = 0;
  for (int k = threadIdx.x; k < m; k += kBinThreads) {
    const ushort4 r = block_rect(rects[list[k]], shift);
    if (!big(r)) { x0 = min(x0, (int)r.x); y0 = min(y0, (int)r.y); x1 = max(x1, (int)r.z); y1 = max(y1, (int)r.w); }
  }
  x0 = __reduce_min_sync(kFull, x0);
  y0 = __reduce_min_sync(kFull, y0);
  x1 = __reduce_max_sync(kFull, x1);
  y1 = __reduce_max_sync(kFull, y1);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&s_box[0], x0); atomicMin(&s_box[1], y0); atomicMax(&s_box[2], x1); atomicMax(&s_box[3], y1);
  }
  __syncthreads();
  LocalBox b;
  b.x0 = s_box[0];
  b.y0 = s_box[1];
  b.w = max(0, s_box[2] - s_box[0]);
  b.h = max(0, s_box[3] - s_box[1]);
  b.ok = (b.w + 1) * (b.h + 1) <= kLocalMax;  // the counting pass's difference array has one more row and column
  return b;
}

template <int N, bool kSecond>
__global__ void __launch_bounds__(kBinThreads) count_kernel(const __grid_constant__ ViewArgs<N> args) {
  const ViewJob& v = args.v[N == 1 ? 0 : blockIdx.y];
  __shared__ uint32_t s_cnt[kLocalMax];
  __shared__ uint16_t s_list[kGroupMax];
  if (kSecond && v.hdr->open_tiles == 0u) return;
  const int gx = list_dim(v.cam.gx, v.shift);  // blocks
  const BlockSkip skip{kSecond ? v.open_bits : nullptr, open_words(v.cam.gx)};
  const int64_t lo = (int64_t)blockIdx.x * v.group;
  if (lo >= v.n) return;
  const int m = kept_list(v, lo, s_list);
  if (m == 0) return;
  const ushort4* rects = v.rect + lo;
  const LocalBox box = group_box(rects, s_list, m, v.shift);
  const int area = box.w * box.h;
  // Per-block counts of the group's box from a 2D difference array: each
  // rectangle adds +1 / -1 / -1 / +1 at its four corners of a (w + 1) x
  // (h + 1) grid, and prefix sums along x then y give, at every block, the
  // number of rectangles covering it (items in skipped blocks are counted here
  // but neither reserved nor filled).  Big rectangles, and every rectangle
  // of a group whose box is too large, count item by item in global memory.
  const int pw = box.w + 1;
  if (box.ok)
    for (int t = threadIdx.x; t < pw * (box.h + 1); t += kBinThreads) s_cnt[t] = 0u;
  __syncthreads();
  for (int k0 = threadIdx.x & ~31; k0 < m; k0 += kBinThreads) {  // whole warps (expand_items)
    const int k = k0 + (threadIdx.x & 31);
    const ushort4 r = k < m ? block_rect(rects[s_list[k]], v.shift) : make_ushort4(0, 0, 0, 0);
    const bool local = box.ok && k < m && !big(r);
    if (local) {
      const int x0 = r.x - box.x0, x1 = r.z - box.x0, y0 = r.y - box.y0, y1 = r.w - box.y0;
      atomicAdd(&s_cnt[y0 * pw + x0], 1u);
      atomicAdd(&s_cnt[y0 * pw + x1], 0xffffffffu);
      atomicAdd(&s_cnt[y1 * pw + x0], 0xffffffffu);
      atomicAdd(&s_cnt[y1 * pw + x1], 1u);
    }
    expand_items(local ? make_ushort4(0, 0, 0, 0) : r, [&](int, int tx, int ty) {
      if (!skip(tx, ty)) atomicAdd(&v.tile_glob[ty * gx + tx], 1u);
    });
  }
  __syncthreads();
  if (!box.ok) return;
  for (int y = threadIdx.x; y < box.h; y += kBinThreads) {  // along x, one row per thread
    uint32_t run = 0u;
    for (int x = 0; x < box.w; ++x) { run += s_cnt[y * pw + x]; s_cnt[y * pw + x] = run; }
  }
  __syncthreads();
  for (int x = threadIdx.x; x < box.w; x += kBinThreads) {  // along y, one column per thread
    uint32_t run = 0u;
    for (int y = 0; y < box.h; ++y) { run += s_cnt[y * pw + x]; s_cnt[y * pw + x] = run; }
  }
  __syncthreads();
  // reserve this CTA's run in every tile of its box (offset inside the tile's list)
  uint32_t* base = v.run_base + (int64_t)blockIdx.x * kLocalMax;
  for (int t = threadIdx.x; t < area; t += kBinThreads) {
    const int ty = t / box.w, tx = t - ty * box.w;
    const uint32_t c = s_cnt[ty * pw + tx];
    base[t] = (c && !skip(box.x0 + tx, box.y0 + ty)) ? atomicAdd(&v.tile_count[(box.y0 + ty) * gx + box.x0 + tx], c)
                                                      : 0u;
  }
}

// Exclusive scan of the tile counts (reserved runs + big-rectangle items; one
// CTA per view, four tiles per thread and round); the fill cursor of a tile
// starts after its reserved runs; the counters are reset for the next pass.
// First pass: capacity check on the view's whole number of listed pairs (what
// the depth cut leaves out included), and the record of open tiles is cleared.
template <int N, bool kSecond>
__global__ void __launch_bounds__(1024) scan_kernel(const __grid_constant__ ViewArgs<N> args, uint32_t* ctr) {
  const ViewJob& v = args.v[N == 1 ? 0 : blockIdx.y];
  if (ctr && blockIdx.y == 0 && threadIdx.x == 0) *ctr = 0u;
  if (kSecond && v.hdr->open_tiles == 0u) return;
  __shared__ uint32_t s_warp[32];
  const int ntiles = list_dim(v.cam.gx, v.shift) * list_dim(v.cam.gy, v.shift);  // lists
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long carry = 0ull;
  for (int base = 0; base < ntiles; base += 4096) {
    const int t = base + 4 * threadIdx.x;
    uint32_t local[4], c[4], sum = 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      local[q] = t + q < ntiles ? v.tile_count[t + q] : 0u;
      c[q] = t + q < ntiles ? local[q] + v.tile_glob[t + q] : 0u;
      sum += c[q];
    }
    uint32_t x = sum;
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, x, off);
      if (lane >= off) x += y;
    }
    __syncthreads();  // the previous round has read s_warp
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    const uint32_t w = s_warp[lane];
    uint32_t run = x - sum + __reduce_add_sync(kFull, lane < warp ? w : 0u);
    const uint32_t total = __reduce_add_sync(kFull, w);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (t + q < ntiles) {
        v.tile_start[t + q] = (uint32_t)(carry + run);
        v.tile_count[t + q] = 0u;
        v.tile_glob[t + q] = 0u;
        v.tile_fill[t + q] = local[q];
        run += c[q];
      }
    carry += total;
  }
  if (!kSecond && v.open_bits)
    for (int t = threadIdx.x; t < cut_blocks(v.cam.gy) * open_words(v.cam.gx); t += 1024) v.open_bits[t] = 0u;
  if (threadIdx.x == 0) {
    v.tile_start[ntiles] = (uint32_t)carry;
    if (!kSecond) {
      const unsigned long long listed = v.hdr->listed;
      if ((long long)listed > v.capacity || listed > 0xffffffffull) atomicOr(&v.hdr->status, kStatCapacity);
      atomicMax(&v.hdr->max_dups_view, (int)min(listed, 0x7fffffffull));
      v.hdr->open_tiles = 0u;
    }
  }
}

// Writes the keys.  The (Gaussian, block) items of the whole group are numbered
// by a scan of the rectangle areas and cut into one contiguous share per
// thread: near Gaussians meet a hundred tiles and lie together in space, and
// dealing each warp the items of its own 32 left single warps with most of a
// launch's work (one view of 300k Gaussians, 640x480: 56 us so, 16.6 now).
template <int N, bool kSecond>
__global__ void __launch_bounds__(kBinThreads) fill_kernel(const __grid_constant__ ViewArgs<N> args) {
  const ViewJob& v = args.v[N == 1 ? 0 : blockIdx.y];
  __shared__ uint32_t s_next[kLocalMax];  // next free position of each box tile's run
  __shared__ uint16_t s_list[kGroupMax];
  __shared__ ushort4 s_rect[kGroupMax];
  __shared__ unsigned long long s_key[kGroupMax];
  __shared__ uint32_t s_first[kGroupMax];  // first item of each Gaussian
  __shared__ uint32_t s_warp[kBinThreads / 32];
  if (v.hdr->status & kStatCapacity) return;
  if (kSecond && v.hdr->open_tiles == 0u) return;
  const int gx = list_dim(v.cam.gx, v.shift), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const BlockSkip skip{kSecond ? v.open_bits : nullptr, open_words(v.cam.gx)};
  const int64_t lo = (int64_t)blockIdx.x * v.group;
  if (lo >= v.n) return;
  const int m = kept_list(v, lo, s_list);
  if (m == 0) return;
  constexpr int kPer = kGroupMax / kBinThreads;
  uint32_t c[kPer], sum = 0u;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int k = tid * kPer + q;
    c[q] = 0u;
    if (k < m) {
      const int i = s_list[k];
      const ushort4 r = v.rect[lo + i];
      s_rect[k] = r;
      s_key[k] = ((unsigned long long)v.depth[lo + i] << 32) | ((uint32_t)v.orig[lo + i] << (4 * v.shift));
      const ushort4 b = block_rect(r, v.shift);
      c[q] = (uint32_t)(b.z - b.x) * (uint32_t)(b.w - b.y);
    }
    sum += c[q];
  }
  uint32_t incl = sum;
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, incl, off);
    if (lane >= off) incl += y;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  uint32_t run = incl - sum, total = 0u;
#pragma unroll
  for (int w = 0; w < kBinThreads / 32; ++w) {
    if (w < warp) run += s_warp[w];
    total += s_warp[w];
  }
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int k = tid * kPer + q;
    if (k < m) s_first[k] = run;
    run += c[q];
  }
  const LocalBox box = group_box(v.rect + lo, s_list, m, v.shift);
  if (box.ok) {
    // the runs reserved by the counting pass (same group, same box)
    const uint32_t* base = v.run_base + (int64_t)blockIdx.x * kLocalMax;
    const int area = box.w * box.h;
    for (int t = tid; t < area; t += kBinThreads)
      s_next[t] = v.tile_start[(box.y0 + t / box.w) * gx + box.x0 + t % box.w] + base[t];
  }
  __syncthreads();
  unsigned long long* __restrict__ keys = v.keys;
  const uint32_t share = (total + kBinThreads - 1) / kBinThreads;
  uint32_t item = share * tid;
  const uint32_t end = min(item + share, total);
  if (item >= end) return;
  int k = 0;
  for (int step = kGroupMax / 2; step >= 1; step >>= 1)  // last Gaussian whose first item is at or before `item`
    if (k + step < m && s_first[k + step] <= item) k += step;
  while (item < end) {
    const ushort4 t = s_rect[k], r = block_rect(t, v.shift);
    const unsigned long long key = s_key[k];
    const bool local = box.ok && !big(r);
    const int w = r.z - r.x, h = r.w - r.y;
    const int at = (int)(item - s_first[k]);
    int y = at / w, x = at - y * w;
    for (; y < h && item < end; ++item) {
      const int bx = r.x + x, by = r.y + y;
      if (!skip(bx, by)) {
        uint32_t tiles = 0u;  // the block's tiles inside the rectangle
        if (v.shift) {
          const uint32_t xm = (2 * bx >= t.x ? 1u : 0u) | (2 * bx + 1 < t.z ? 2u : 0u);
          tiles = (2 * by >= t.y ? xm : 0u) | (2 * by + 1 < t.w ? xm << 2 : 0u);
        }
        const uint32_t pos = local ? atomicAdd(&s_next[box.idx(bx, by)], 1u)
                                   : v.tile_start[by * gx + bx] + atomicAdd(&v.tile_fill[by * gx + bx], 1u);
        keys[pos] = key | tiles;
      }
      if (++x == w) { x = 0; ++y; }
    }
    ++k;
  }
}

template <int N, bool kSecond>
cudaError_t launch_n(const ViewJob* v, int nv, uint32_t* ctr, cudaStream_t st) {
  ViewArgs<N> a;
  int groups = 0;
  for (int k = 0; k < N; ++k) {
    a.v[k] = v[k < nv ? k : 0];
    const int g = (int)(((int64_t)a.v[k].n + a.v[k].group - 1) / a.v[k].group);
    groups = g > groups ? g : groups;
  }
  const dim3 grid(groups, nv);
  if (groups > 0) count_kernel<N, kSecond><<<grid, kBinThreads, 0, st>>>(a);
  scan_kernel<N, kSecond><<<dim3(1, nv), 1024, 0, st>>>(a, ctr);
  if (groups > 0) fill_kernel<N, kSecond><<<grid, kBinThreads, 0, st>>>(a);
  g_launches += groups > 0 ? 3 : 1;
  return cudaGetLastError();
}

template <bool kSecond>
cudaError_t launch_pass(const ViewJob* v, int nv, uint32_t* ctr, cudaStream_t st) {
  if (nv == 1) return launch_n<1, kSecond>(v, nv, ctr, st);
  if (nv <= 8) return launch_n<8, kSecond>(v, nv, ctr, st);
  return launch_n<kMaxDrainJobs, kSecond>(v, nv, ctr, st);
}

}  // namespace

cudaError_t launch_binning(const ViewJob* v, int nv, bool second, uint32_t* ctr, cudaStream_t st) {
  if (nv <= 0) return cudaSuccess;
  if (nv > kMaxDrainJobs) return cudaErrorInvalidValue;
  return second ? launch_pass<true>(v, nv, ctr, st) : launch_pass<false>(v, nv, ctr, st);
}

}  // namespace scoup
