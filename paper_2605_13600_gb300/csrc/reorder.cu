// reorder.cu -- one-time spatial reordering of the scene for binning locality.
//
// Gaussians are grouped by the 3D Morton code of a 32^3 grid over the
// bounding box of their means (a counting sort), and the scene arrays are
// gathered into that order in the workspace.  Gaussians that are close in 3D
// project close together in every view, so a binning CTA's chunk of
// consecutive Gaussians covers a compact set of tiles and writes long
// contiguous runs of keys.  The original index travels with every Gaussian:
// keys, records and accumulator rows stay addressed by it, so no result
// depends on this order.  What of the projection does not depend on the view
// -- the 3D covariance Sigma3 and the alpha-threshold exponent tau -- is
// computed here once per call instead of once per view.
//
// This translation unit is compiled with --fmad=false like preprocess.cu:
// Sigma3 is part of the binary32 projection, each operation rounded in order.
#include <math.h>
#include <stddef.h>

#include "scoup_internal.cuh"

namespace scoup {
namespace {

constexpr int kCells = 1 << 15;  // 32^3 Morton cells

__device__ __forceinline__ uint32_t ordered_bits(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float from_ordered(uint32_t u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

__device__ __forceinline__ uint32_t spread3(uint32_t v) {  // 5 bits -> every third bit
  v &= 0x1fu;
  v = (v | (v << 8)) & 0x0100f00fu;
  v = (v | (v << 4)) & 0x010c30c3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

// Bounding box of the means: reduced per CTA first, so that the six header
// words receive one atomic per CTA (per warp they serialise: 22.6 us for 1M
// Gaussians against 6.4).
__global__ void __launch_bounds__(256) bbox_kernel(const float* __restrict__ means, int64_t n,
                                                   WsHeader* __restrict__ hdr) {
  __shared__ uint32_t s_lo[8][3], s_hi[8][3];
  uint32_t lo[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, hi[3] = {0u, 0u, 0u};
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const uint32_t u = ordered_bits(means[3 * i + a]);
      lo[a] = min(lo[a], u);
      hi[a] = max(hi[a], u);
    }
  }
  const int warp = threadIdx.x >> 5;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = __reduce_min_sync(0xffffffffu, lo[a]);
    hi[a] = __reduce_max_sync(0xffffffffu, hi[a]);
    if ((threadIdx.x & 31) == 0) { s_lo[warp][a] = lo[a]; s_hi[warp][a] = hi[a]; }
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    const int a = threadIdx.x;
    for (int w = 1; w < 8; ++w) { s_lo[0][a] = min(s_lo[0][a], s_lo[w][a]); s_hi[0][a] = max(s_hi[0][a], s_hi[w][a]); }
    atomicMin(&hdr->bbox[a][0], s_lo[0][a]);
    atomicMax(&hdr->bbox[a][1], s_hi[0][a]);
  }
}

// Cell of every Gaussian and its rank among the Gaussians of the cell (the
// count before it), packed: kCellBits of cell, the rest of rank.  Ranks that
// do not fit saturate; the gather gives those their place with a cursor.
constexpr int kCellBits = 15;
constexpr uint32_t kRankMax = (1u << (32 - kCellBits)) - 1u;

__global__ void __launch_bounds__(256) cell_kernel(const float* __restrict__ means, int64_t n,
                                                   const WsHeader* __restrict__ hdr, uint32_t* __restrict__ cell,
                                                   uint32_t* __restrict__ cnt) {
  float lo[3], scale[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = from_ordered(hdr->bbox[a][0]);
    const float ext = from_ordered(hdr->bbox[a][1]) - lo[a];
    scale[a] = ext > 0.0f ? 32.0f / ext : 0.0f;
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    uint32_t q[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float f = (means[3 * i + a] - lo[a]) * scale[a];
      q[a] = f > 0.0f ? (uint32_t)min(f, 31.0f) : 0u;
    }
    const uint32_t c = spread3(q[0]) | (spread3(q[1]) << 1) | (spread3(q[2]) << 2);
    cell[i] = c | (min(atomicAdd(&cnt[c], 1u), kRankMax) << kCellBits);
  }
}

// Exclusive scan of the cell counts into start[], overflow cursors zeroed.
// One CTA per 1024 cells: it sums the counts in front of its own (at most
// 128 KB, read coalesced from L2) instead of waiting for the CTA before it.
// (One CTA scanning all cells, 32 consecutive ones per thread, took 51 us, this form 7.8.)
__global__ void __launch_bounds__(1024) cell_scan_kernel(const uint32_t* __restrict__ cnt,
                                                         uint32_t* __restrict__ start,
                                                         uint32_t* __restrict__ cur) {
  __shared__ uint32_t s_warp[32], s_base[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = blockIdx.x * 1024 + tid;
  uint32_t before = 0u;
#pragma unroll 8
  for (int k = tid; k < (int)blockIdx.x * 1024; k += 1024) before += cnt[k];
  const uint32_t v = cnt[c];
  before = __reduce_add_sync(0xffffffffu, before);
  uint32_t incl = v;
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += y;
  }
  if (lane == 31) s_warp[warp] = incl;
  if (lane == 0) s_base[warp] = before;
  __syncthreads();
  uint32_t run = __reduce_add_sync(0xffffffffu, s_base[lane]);
  run += __reduce_add_sync(0xffffffffu, lane < warp ? s_warp[lane] : 0u);
  start[c] = run + incl - v;
  cur[c] = 0u;
}

__device__ __noinline__ float tau_fp64(float o) {
  const double t = -log(255.0 * (double)o);
  float th = (float)t;
  if ((double)th < t) th = nextafterf(th, INFINITY);
  return th;
}

// The alpha-threshold exponent of opacity o: the smallest binary32 tau with
// o * exp(tau) >= 1/255, i.e. -log(255 o) rounded up.  FP64 runs at 1/64 of
// the FP32 rate here, and its logarithm alone took 50 of the gather's 75 us
// for 1M Gaussians; instead 255 o = 2^e m (m in [sqrt(1/2), sqrt(2))) goes
// through log m = 2 atanh(s), s = (m - 1) / (m + 1), with s and its cubic term
// as unevaluated sums of two floats (the terms from s^5 on in one float).
// The result t = th + tl carries an error below `eps`; only where |tl| does
// not decide the rounding (0.1% of the opacities) the FP64 form runs.  Equal
// to it for every binary32 o in [2^-31, 32] (checked one by one).
__device__ __forceinline__ float alpha_threshold(float o) {
  if (!(o > 0.0f)) return INFINITY;
  if (o < 1e-30f || o > 1e30f) return tau_fp64(o);
  const float xh = 255.0f * o, xl = fmaf(255.0f, o, -xh);
  const uint32_t b = __float_as_uint(xh);
  const int e = (int)(b - 0x3f3504f3u) >> 23;
  const float mh = __uint_as_float(b - ((uint32_t)e << 23)), ml = xl * __uint_as_float((uint32_t)(127 - e) << 23);
  const float dh = mh + 1.0f, dl = (mh - (dh - 1.0f)) + ml, nh = mh - 1.0f;
  const float sh = __fdiv_rn(nh + ml, dh);
  const float sl = __fdividef(fmaf(-sh, dh, nh) + fmaf(-sh, dl, ml), dh);
  const float zh = sh * sh, zl = fmaf(sh, sh, -zh) + 2.0f * sh * sl;
  const float ch = zh * sh, cl = fmaf(zh, sh, -ch) + fmaf(zl, sh, zh * sl);
  constexpr float kThird2 = (float)(2.0 / 3.0), kThird2Lo = (float)(2.0 / 3.0 - (double)kThird2);
  const float ph = ch * kThird2, pl = fmaf(ch, kThird2, -ph) + fmaf(ch, kThird2Lo, cl * kThird2);
  float q = fmaf(zh, 2.0f / 15, 2.0f / 13);
  q = fmaf(zh, q, 2.0f / 11);
  q = fmaf(zh, q, 2.0f / 9);
  q = fmaf(zh, q, 2.0f / 7);
  q = zh * ch * fmaf(zh, q, 0.4f);
  // ln 2 in a 16-bit part (its product with e is exact) and the rest
  const float kh = (float)e * 0.693145751953125f, kl = (float)e * 1.42860682030941723e-6f;
  const float s1 = kh + 2.0f * sh, v1 = s1 - kh, e1 = (kh - (s1 - v1)) + (2.0f * sh - v1);
  const float s2 = s1 + ph, v2 = s2 - s1, e2 = (s1 - (s2 - v2)) + (ph - v2);
  const float rest = (((q + pl) + 2.0f * sl) + kl) + (e1 + e2);
  const float sum = s2 + rest, v3 = sum - s2;
  const float th = -sum, tl = -((s2 - (sum - v3)) + (rest - v3));
  const float eps = fabsf(th) * 3.0e-11f + fabsf(q) * 4.8e-6f + fabsf(kl) * 2.4e-7f;
  if (!(fabsf(tl) > eps)) return tau_fp64(o);
  return tl > 0.0f ? nextafterf(th, INFINITY) : th;
}

// Scene records in spatial order.  A record's 48 bytes go out as three
// 16-byte stores to one place (the arrays one by one scattered 7 sectors per
// Gaussian: 97.5 us for 1M Gaussians against 74.8, and 38.5 with the FP32 tau).
__global__ void __launch_bounds__(256) gather_kernel(const float* __restrict__ means, const float* __restrict__ scales,
                                                     const float* __restrict__ quats,
                                                     const float* __restrict__ opacity, int64_t n,
                                                     const uint32_t* __restrict__ cell,
                                                     const uint32_t* __restrict__ start, uint32_t* __restrict__ cur,
                                                     SceneP sp) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t cr = cell[i], c = cr & ((1u << kCellBits) - 1u);
    uint32_t rank = cr >> kCellBits;
    if (rank == kRankMax) rank += atomicAdd(&cur[c], 1u);
    const int64_t p = (int64_t)start[c] + rank;
    const float o = opacity[i];
    SceneRec r;
    r.mean_op = make_float4(means[3 * i], means[3 * i + 1], means[3 * i + 2], o);
    const float4 q = *reinterpret_cast<const float4*>(quats + 4 * i);
    const float s0 = scales[3 * i], s1 = scales[3 * i + 1], s2 = scales[3 * i + 2];
    // Sigma3 = (R S)(R S)^T from the normalised quaternion and scales
    const float qn = q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w;
    const float inv = 1.0f / sqrtf(qn);
    const float w = q.x * inv, x = q.y * inv, y = q.z * inv, z = q.w * inv;
    const float R00 = 1.0f - 2.0f * (y * y + z * z);
    const float R01 = 2.0f * (x * y - w * z);
    const float R02 = 2.0f * (x * z + w * y);
    const float R10 = 2.0f * (x * y + w * z);
    const float R11 = 1.0f - 2.0f * (x * x + z * z);
    const float R12 = 2.0f * (y * z - w * x);
    const float R20 = 2.0f * (x * z - w * y);
    const float R21 = 2.0f * (y * z + w * x);
    const float R22 = 1.0f - 2.0f * (x * x + y * y);
    const float M00 = R00 * s0, M01 = R01 * s1, M02 = R02 * s2;
    const float M10 = R10 * s0, M11 = R11 * s1, M12 = R12 * s2;
    const float M20 = R20 * s0, M21 = R21 * s1, M22 = R22 * s2;
    r.cov_a = make_float4(M00 * M00 + M01 * M01 + M02 * M02, M00 * M10 + M01 * M11 + M02 * M12,
                          M00 * M20 + M01 * M21 + M02 * M22, M10 * M10 + M11 * M11 + M12 * M12);
    r.cov_b = make_float4(M10 * M20 + M11 * M21 + M12 * M22, M20 * M20 + M21 * M21 + M22 * M22, alpha_threshold(o),
                          __int_as_float((int32_t)i));
    sp.rec[p] = r;
    sp.orig[p] = (int32_t)i;
  }
}

__global__ void __launch_bounds__(256) threshold_kernel(const float* __restrict__ o, int64_t n, float* __restrict__ tau) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    tau[i] = alpha_threshold(o[i]);
}

// Everything a call starts from, in one launch: the header (zero but for the
// empty depth range and bounding box), the cell counts, and the binning
// counters of a render's view.
struct BeginArgs {
  WsHeader* hdr;
  uint32_t* cnt;
  uint32_t* zero[2];  // arrays of max_tiles + 1 words (null: none)
  int max_tiles;
};

__global__ void __launch_bounds__(256) begin_kernel(const __grid_constant__ BeginArgs a) {
  const int t0 = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  static_assert(offsetof(WsHeader, drange) == 8 && offsetof(WsHeader, bbox) == 16, "words below");
  if (t0 < (int)(sizeof(WsHeader) / 4))
    reinterpret_cast<uint32_t*>(a.hdr)[t0] = (t0 >= 2 && t0 < 10 && !(t0 & 1)) ? 0xffffffffu : 0u;
  for (int t = t0; t < kCells; t += stride) a.cnt[t] = 0u;
#pragma unroll
  for (int q = 0; q < 2; ++q)
    if (a.zero[q])
      for (int t = t0; t <= a.max_tiles; t += stride) a.zero[q][t] = 0u;
}

int grid_for(int64_t n, int per_sm) {
  int64_t b = (n + 255) / 256;
  if (b > num_sms() * per_sm) b = num_sms() * per_sm;
  return (int)(b > 0 ? b : 1);
}

}  // namespace

size_t reorder_scratch_bytes() { return sizeof(uint32_t) * (size_t)(3 * kCells); }

cudaError_t launch_alpha_thresholds(const float* opacity, int64_t n, float* tau, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  threshold_kernel<<<grid_for(n, 8), 256, 0, st>>>(opacity, n, tau);
  g_launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_begin(const UpliftWs& ws, bool view, int max_tiles, cudaStream_t st) {
  BeginArgs a = {};
  a.hdr = ws.hdr;
  a.cnt = ws.cells_scratch;
  a.max_tiles = max_tiles;
  if (view) {
    a.zero[0] = ws.tile_count;
    a.zero[1] = ws.tile_glob;
  }
  begin_kernel<<<32, 256, 0, st>>>(a);
  g_launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_reorder(const scoup_scene& sc, const UpliftWs& ws, cudaStream_t st) {
  if (sc.n <= 0) return cudaSuccess;
  uint32_t* cnt = ws.cells_scratch;
  uint32_t* start = cnt + kCells;
  uint32_t* cur = start + kCells;
  bbox_kernel<<<grid_for(sc.n, 4), 256, 0, st>>>(sc.means, sc.n, ws.hdr);
  cell_kernel<<<grid_for(sc.n, 8), 256, 0, st>>>(sc.means, sc.n, ws.hdr, ws.cell, cnt);
  cell_scan_kernel<<<kCells / 1024, 1024, 0, st>>>(cnt, start, cur);
  gather_kernel<<<grid_for(sc.n, 8), 256, 0, st>>>(sc.means, sc.scales, sc.quats, sc.opacity, sc.n,
                                                   ws.cell, start, cur, ws.sp);
  g_launches += 4;
  return cudaGetLastError();
}

}  // namespace scoup
