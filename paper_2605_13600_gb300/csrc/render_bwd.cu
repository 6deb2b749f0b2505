// render_bwd.cu -- gradient of a loss through the sparse-code rendering
// (Eq. 7 with the compositing of Eq. 2) with respect to the Top-K values and
// the opacities.  For one pixel with contributions i = 1..m (front to back),
// g = dL/dWhat(p), gw_i = g . w^_i and S = sum_i e_i gw_i:
//   dL/dval_ik  += e_i g[idx_ik]
//   dL/dalpha_i  = T_i gw_i - (S - sum_{j<=i} e_j gw_j) / (1 - alpha_i)
//   dL/do_i     += dalpha_i/do_i dL/dalpha_i,   dalpha/do = G while o G < 0.99, else 0.
// Top-K indices, the alpha >= 1/255 test and the transmittance stop are held
// fixed (piecewise-constant decisions).
//
// Transmittance is recomputed, not stored: the tile's list is walked twice
// (window by window, same order as the forward), the first walk giving S per
// pixel, the second the gradients.  Per window, gradients of the window's
// Gaussians are summed over the tile's pixels in shared memory (entry-major,
// so a warp's lanes hit consecutive words) and flushed with one global atomic
// per (Gaussian, entry).  The window's Top-K codes are staged in shared
// memory with the records whenever they fit.
//
// Two kernels.  Codes of up to 16 entries take render_bwd_block_kernel: a warp
// owns an 8 x 4 block of the tile's pixels and walks the window entries that
// may reach it 32 at a time, one Gaussian per lane, over all its open pixels
// before the next 32.  The Gaussian's record, code and gradient sums then stay
// in the lane's registers: a (pixel, Gaussian) pair costs the exponent, its
// share of two warp scans and one gather of K words of the pixel's gradient
// row, without a shared atomic.  Longer codes take render_bwd_kernel (a warp
// per pixel, every window entry).  Up to 16 entries the block kernel is the
// faster one at every width, though its gradient rows leave one CTA per SM at C =
// 1024 (its time over the other's, K = 4 / 8 / 16, 500k Gaussians, 800 x 600: C =
// 256 0.62 / 0.54 / 0.48, 512 0.61 / 0.50 / 0.40, 1024 0.73 / 0.56 / 0.57; 10k,
// 160 x 120: 0.27 / 0.23 / 0.22, 0.27 / 0.24 / 0.23, 0.26 / 0.25 / 0.24).
#include <math.h>

#include "tile_order.cuh"

namespace scoup {
namespace {

constexpr int kBThreads = 256;
constexpr int kBWarps = kBThreads / 32;
using BOrder = OrderSmem<256, 10>;
constexpr size_t kBStageMaxBytes = 48 * 1024;

struct BwdSmem {
  BOrder ord;
  float4 rec_a[BOrder::kWin];
  float4 rec_b[BOrder::kWin];
  float T[kTilePixels];
  float S[kTilePixels];      // pass 1: running sum of e gw; pass 2: total
  float Sb[kTilePixels];     // pass 2: sum of e gw in front of the current position
  int done[kTilePixels];
  int next_pixel;
  // dynamic: g rows [kBWarps][C], dval [K][kWin], dop [kWin], staged codes
  // (values [K][kWin], atom ids [K][kWin] as int16)
};

struct BwdDyn {
  float* g;
  float* dval;
  float* dop;
  float* cval;
  short* cidx;
};

__device__ __forceinline__ BwdDyn bwd_dyn(BwdSmem& sm, int C, int K) {
  float* base = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(&sm) + sizeof(BwdSmem));
  BwdDyn d;
  d.g = base;
  d.dval = base + kBWarps * C;
  d.dop = d.dval + BOrder::kWin * K;
  d.cval = d.dop + BOrder::kWin;
  d.cidx = reinterpret_cast<short*>(d.cval + BOrder::kWin * K);
  return d;
}

// One pass of pixel (fpx, fpy) over window win[0..m).  pass 1 accumulates S;
// pass 2 accumulates the gradients of the window's Gaussians.
template <int kPass, bool kStaged>
__device__ __forceinline__ bool walk_bwd(BwdSmem& sm, const BwdDyn& dy, const float* gw_row, int m,
                                         float fpx, float fpy, float& T, float& S, float& Sb, float Stot,
                                         const int32_t* __restrict__ topk_idx, const float* __restrict__ topk_val,
                                         int K, int C) {
  const int lane = threadIdx.x & 31;
  for (int w0 = 0; w0 < m; w0 += 32) {
    const int j = w0 + lane;
    const bool live = j < m;
    const int jj = live ? j : 0;
    const float4 a = sm.rec_a[jj];
    const float4 b = sm.rec_b[jj];
    const float dx = a.x - fpx, dyy = a.y - fpy;
    const float power = fmaf(dx, fmaf(a.z, dx, __fmul_rn(a.w, dyy)), __fmul_rn(__fmul_rn(b.x, dyy), dyy));
    const bool accept = live && power <= 0.0f && power >= b.z;
    const float G = __expf(power);
    const float alpha = accept ? fminf(0.99f, b.y * G) : 0.0f;
    float P = 1.0f - alpha;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float y = __shfl_up_sync(0xffffffffu, P, off);
      if (lane >= off) P *= y;
    }
    float Pex = __shfl_up_sync(0xffffffffu, P, 1);
    if (lane == 0) Pex = 1.0f;
    const float Tl = T * Pex;
    const float test = T * P;
    const unsigned stopmask = __ballot_sync(0xffffffffu, accept && test < 1e-4f);
    const int first = stopmask ? __ffs(stopmask) - 1 : 32;
    const bool take = accept && lane < first;
    const float e = take ? alpha * Tl : 0.0f;
    const int gidx = (int)(sm.ord.win[jj] & 0xffffffffull);
    float gw = 0.0f;
    if (take) {
      if constexpr (kStaged) {
        for (int k = 0; k < K; ++k) {
          const int atom = dy.cidx[k * BOrder::kWin + j];
          if (atom >= 0) gw += dy.cval[k * BOrder::kWin + j] * gw_row[atom];
        }
      } else {
        const int32_t* ci = topk_idx + (int64_t)gidx * K;
        const float* cv = topk_val + (int64_t)gidx * K;
        for (int k = 0; k < K; ++k) {
          const int atom = ci[k];
          if (atom >= 0 && atom < C) gw += cv[k] * gw_row[atom];
        }
      }
    }
    const float eg = e * gw;
    // inclusive sum scan of e * gw over the lanes
    float incl = eg;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float y = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += y;
    }
    if (kPass == 2 && take) {
      const float S_after = Stot - (Sb + incl);
      const float dLda = Tl * gw - S_after / (1.0f - alpha);
      const float dado = (b.y * G < 0.99f) ? G : 0.0f;
      atomicAdd(&dy.dop[j], dado * dLda);
      for (int k = 0; k < K; ++k) {
        int atom;
        if constexpr (kStaged) {
          atom = dy.cidx[k * BOrder::kWin + j];
        } else {
          atom = topk_idx[(int64_t)gidx * K + k];
          if (atom >= C) atom = -1;
        }
        if (atom >= 0) atomicAdd(&dy.dval[k * BOrder::kWin + j], e * gw_row[atom]);
      }
    }
    const float round_sum = __shfl_sync(0xffffffffu, incl, 31);
    if (kPass == 1) S += round_sum;
    else Sb += round_sum;
    if (stopmask) {
      T = __shfl_sync(0xffffffffu, Tl, first);
      return true;
    }
    T = __shfl_sync(0xffffffffu, test, 31);
  }
  return false;
}

// Codes of more than 16 entries: their gradient sums and staged codes take the
// shared memory of two or three CTAs per SM, so the launch bound is two, which
// leaves the walk's registers alone (at four, 64 registers, the walk is 3 to 6 %
// slower and spills; 500k Gaussians, 800x600, ms at four / two: C = 64, K = 17
// 3.9 / 3.7, C = 256, K = 24 6.3 / 5.8, C = 512, K = 32 13.7 / 12.3; C = 256,
// K = 33, codes not staged, 17.3 / 11.6).
template <bool kStaged>
__global__ void __launch_bounds__(kBThreads, 2) render_bwd_kernel(
    const __grid_constant__ ViewJob view, const int32_t* __restrict__ topk_idx,
    const float* __restrict__ topk_val, int K, int C, const float* __restrict__ dL_dcodes,
    float* __restrict__ d_val, float* __restrict__ d_opacity) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BwdSmem& sm = *reinterpret_cast<BwdSmem*>(smem_raw);
  const CamArgs& cam = view.cam;
  WsHeader* __restrict__ const hdr = view.hdr;
  const ProjRec* __restrict__ const proj = view.proj;
  const int tile = (int)blockIdx.x;
  const TileList list = tile_list(view.keys, view.tile_start, nullptr, view.shift, cam.gx, tile);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tx = tile % cam.gx, ty = tile / cam.gx;
  const int n = list.n;
  if (n == 0) return;
  if (hdr->status & kStatCapacity) return;
  const BwdDyn dy = bwd_dyn(sm, C, K);
  float* grow = dy.g + warp * C;
  const OrderBuckets bk = order_buckets<BOrder>(hdr);
  order_init(sm.ord, list, bk);

  for (int pass = 1; pass <= 2; ++pass) {
    for (int p = tid; p < kTilePixels; p += kBThreads) {
      const int px = tx * kTile + (p & (kTile - 1)), py = ty * kTile + (p >> 4);
      sm.T[p] = 1.0f;
      sm.Sb[p] = 0.0f;
      if (pass == 1) sm.S[p] = 0.0f;
      sm.done[p] = !(px < cam.width && py < cam.height);
    }
    __syncthreads();
    OrderState st;
    while (true) {
      const int m = order_next_window(sm.ord, list, bk, st, hdr);
      if (m <= 0) break;
      for (int j = tid; j < m; j += kBThreads) {
        const ProjRec pr = proj[(int)(sm.ord.win[j] & 0xffffffffull)];
        sm.rec_a[j] = pr.a;
        sm.rec_b[j] = pr.b;
        if (pass == 2) {
          for (int k = 0; k < K; ++k) dy.dval[k * BOrder::kWin + j] = 0.0f;
          dy.dop[j] = 0.0f;
        }
      }
      if constexpr (kStaged) {
        for (int t = tid; t < m * K; t += kBThreads) {
          const int j = t / K, k = t - j * K;
          const int64_t g = (int64_t)(sm.ord.win[j] & 0xffffffffull);
          const int atom = topk_idx[g * K + k];
          dy.cidx[k * BOrder::kWin + j] = (short)(atom >= 0 && atom < C ? atom : -1);
          dy.cval[k * BOrder::kWin + j] = topk_val[g * K + k];
        }
      }
      if (tid == 0) sm.next_pixel = 0;
      __syncthreads();
      while (true) {
        int p = 0;
        if (lane == 0) p = atomicAdd(&sm.next_pixel, 1);
        p = __shfl_sync(0xffffffffu, p, 0);
        if (p >= kTilePixels) break;
        if (sm.done[p]) continue;
        const int px = tx * kTile + (p & (kTile - 1)), py = ty * kTile + (p >> 4);
        const float* g = dL_dcodes + ((int64_t)py * cam.width + px) * C;
        for (int c = lane; c < C; c += 32) grow[c] = g[c];
        __syncwarp();
        float T = sm.T[p], S = sm.S[p], Sb = sm.Sb[p];
        const bool fin = pass == 1
            ? walk_bwd<1, kStaged>(sm, dy, grow, m, (float)px, (float)py, T, S, Sb, 0.0f, topk_idx, topk_val, K, C)
            : walk_bwd<2, kStaged>(sm, dy, grow, m, (float)px, (float)py, T, S, Sb, sm.S[p], topk_idx, topk_val,
                                   K, C);
        if (lane == 0) {
          sm.T[p] = T;
          if (pass == 1) sm.S[p] = S;
          sm.Sb[p] = Sb;
          sm.done[p] = fin;
        }
        __syncwarp();
      }
      __syncthreads();
      if (pass == 2) {
        // flush the window's per-Gaussian gradient sums
        for (int j = tid; j < m; j += kBThreads) {
          const int64_t gi = (int64_t)(sm.ord.win[j] & 0xffffffffull);
          const float dop = dy.dop[j];
          if (dop != 0.0f) atomicAdd(&d_opacity[gi], dop);
          for (int k = 0; k < K; ++k) {
            const float v = dy.dval[k * BOrder::kWin + j];
            if (v != 0.0f) atomicAdd(&d_val[gi * K + k], v);
          }
        }
        __syncthreads();
      }
      int open = 0;
      for (int p = tid; p < kTilePixels; p += kBThreads) open |= !sm.done[p];
      if (!__syncthreads_or(open)) break;
    }
    __syncthreads();
  }
}

// ---- codes of up to 16 entries ---------------------------------------------

struct BwdBlockSmem {
  BOrder ord;
  float4 rec_a[BOrder::kWin];
  float4 rec_b[BOrder::kWin];
  uint16_t list[kBWarps][BOrder::kWin];  // per warp: window entries that may reach its block
  uint8_t mask[BOrder::kWin];            // per window entry: the blocks it may reach
  // dynamic: gradient rows [kBWarps][2][kNP][row_words(C)], dval [K][kWin], dop [kWin]
};

// A staged gradient row: C words, then a zero that padding entries read, in 16-byte units.
__host__ __device__ inline int row_words(int C) { return (C + 4) & ~3; }

__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Starts the copy of one pixel's gradient row.
template <bool kVec>
__device__ __forceinline__ void stage_row(float* dst, const float* src, int C, int lane) {
  if constexpr (kVec) {
    for (int c = 4 * lane; c < C; c += 128) cp_async16(dst + c, src + c);
  } else {
    for (int c = lane; c < C; c += 32) cp_async4(dst + c, src + c);
  }
}

// State of a pixel, uniform over the warp.
struct BwdPixel {
  float x, y;
  float T, S, Sb;  // S: sum of e gw, complete in pass 2; Sb: its part in front
  bool on, stopped;
};

// kNP pixels over the chunk, interleaved (their scans are dependent chains of
// shuffles).  kPass 1: S += sum of e gw over the chunk; kPass 2: the gradient
// sums of the lane's Gaussian.
template <int kPass, int KR, int kNP>
__device__ __forceinline__ void walk_pixels(const float4& a, const float4& b, bool live, const uint32_t (&ids)[KR / 2],
                                            const float (&vals)[KR], const float* const (&row)[kNP],
                                            BwdPixel (&px)[kNP], float (&acc)[KR], float& dop) {
  const int lane = threadIdx.x & 31;
  float G[kNP], alpha[kNP], P[kNP];
  bool accept[kNP], any = false;
#pragma unroll
  for (int u = 0; u < kNP; ++u) {
    const float dx = a.x - px[u].x, dy = a.y - px[u].y;
    const float power = fmaf(dx, fmaf(a.z, dx, __fmul_rn(a.w, dy)), __fmul_rn(__fmul_rn(b.x, dy), dy));
    accept[u] = live && px[u].on && power <= 0.0f && power >= b.z;
    any = any || accept[u];
    G[u] = __expf(power);
    alpha[u] = accept[u] ? fminf(0.99f, b.y * G[u]) : 0.0f;
    P[u] = 1.0f - alpha[u];
    px[u].stopped = false;
  }
  if (!__any_sync(0xffffffffu, any)) return;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1)
#pragma unroll
    for (int u = 0; u < kNP; ++u) {
      const float y = __shfl_up_sync(0xffffffffu, P[u], off);
      if (lane >= off) P[u] *= y;
    }
  float Tl[kNP], e[kNP], gw[kNP], g[kNP][KR];
  int src[kNP];
#pragma unroll
  for (int u = 0; u < kNP; ++u) {
    float Pex = __shfl_up_sync(0xffffffffu, P[u], 1);
    if (lane == 0) Pex = 1.0f;
    Tl[u] = px[u].T * Pex;
    const float test = px[u].T * P[u];
    const unsigned stopmask = __ballot_sync(0xffffffffu, accept[u] && test < 1e-4f);
    const int first = stopmask ? __ffs(stopmask) - 1 : 32;
    accept[u] = accept[u] && lane < first;  // takes part
    e[u] = accept[u] ? alpha[u] * Tl[u] : 0.0f;
    px[u].stopped = stopmask != 0u;
    src[u] = stopmask ? first : 31;
    P[u] = stopmask ? Tl[u] : test;
    gw[u] = 0.0f;
    if (accept[u]) {
#pragma unroll
      for (int k = 0; k < KR; ++k) g[u][k] = row[u][(ids[k / 2] >> (16 * (k & 1))) & 0xffffu];
#pragma unroll
      for (int k = 0; k < KR; ++k) gw[u] = fmaf(vals[k], g[u][k], gw[u]);
    }
  }
  float incl[kNP];
#pragma unroll
  for (int u = 0; u < kNP; ++u) incl[u] = e[u] * gw[u];
  if constexpr (kPass == 1) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
      for (int u = 0; u < kNP; ++u) incl[u] += __shfl_xor_sync(0xffffffffu, incl[u], off);
#pragma unroll
    for (int u = 0; u < kNP; ++u) px[u].S += incl[u];
  } else {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1)
#pragma unroll
      for (int u = 0; u < kNP; ++u) {
        const float y = __shfl_up_sync(0xffffffffu, incl[u], off);
        if (lane >= off) incl[u] += y;
      }
#pragma unroll
    for (int u = 0; u < kNP; ++u) {
      if (accept[u]) {
        const float S_after = px[u].S - (px[u].Sb + incl[u]);
        const float dLda = Tl[u] * gw[u] - S_after / (1.0f - alpha[u]);
        dop += (b.y * G[u] < 0.99f) ? G[u] * dLda : 0.0f;
#pragma unroll
        for (int k = 0; k < KR; ++k) acc[k] = fmaf(e[u], g[u][k], acc[k]);
      }
      px[u].Sb += __shfl_sync(0xffffffffu, incl[u], 31);
    }
  }
#pragma unroll
  for (int u = 0; u < kNP; ++u) px[u].T = __shfl_sync(0xffffffffu, P[u], src[u]);
}

// Two pixels in flight and two CTAs per SM (127 registers).  The backward of an
// 800 x 600 view of 500k Gaussians, C = 256, K = 8: 2145 us in the warp-per-pixel
// kernel; here 2516 us with one pixel and four CTAs (232 B of spills), 1440 and
// 1388 with three and two CTAs, 1195 with two pixels and two CTAs.  Bound by
// the latency of the scans (49% of the issue rate, 4 warps per scheduler).
template <int KR, int kNP, bool kVec>
__global__ void __launch_bounds__(kBThreads, 2) render_bwd_block_kernel(
    const __grid_constant__ ViewJob view, const int32_t* __restrict__ topk_idx,
    const float* __restrict__ topk_val, int K, int C, const float* __restrict__ dL_dcodes,
    float* __restrict__ d_val, float* __restrict__ d_opacity) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BwdBlockSmem& sm = *reinterpret_cast<BwdBlockSmem*>(smem_raw);
  const CamArgs& cam = view.cam;
  WsHeader* __restrict__ const hdr = view.hdr;
  const int tile = (int)blockIdx.x;
  const TileList list = tile_list(view.keys, view.tile_start, nullptr, view.shift, cam.gx, tile);
  if (list.n == 0) return;
  if (hdr->status & kStatCapacity) return;
  constexpr int kW = BOrder::kWin;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tx = tile % cam.gx, ty = tile / cam.gx;
  const int bx = tx * kTile + (warp & 1) * 8, by = ty * kTile + (warp >> 1) * 4;
  const bool inside = bx + (lane & 7) < cam.width && by + (lane >> 3) < cam.height;
  const int rw = row_words(C);
  float* const rows = reinterpret_cast<float*>(smem_raw + ((sizeof(BwdBlockSmem) + 15) & ~(size_t)15)) + warp * 2 * kNP * rw;
  float* const dval = reinterpret_cast<float*>(smem_raw + ((sizeof(BwdBlockSmem) + 15) & ~(size_t)15)) + kBWarps * 2 * kNP * rw;
  float* const dop_sum = dval + K * kW;
  const float* const gblock = dL_dcodes + ((int64_t)by * cam.width + bx) * C;
  if (lane < 2 * kNP) rows[lane * rw + C] = 0.0f;
  const OrderBuckets bk = order_buckets<BOrder>(hdr);
  order_init(sm.ord, list, bk);

  float S = 0.0f;  // lane p: sum of e gw of the block's pixel p (pass 1)
  for (int pass = 1; pass <= 2; ++pass) {
    float T = 1.0f, Sb = 0.0f;  // of the lane's pixel
    bool open = inside;
    OrderState st;
    while (true) {
      const int m = order_next_window(sm.ord, list, bk, st, hdr);
      if (m <= 0) break;
      for (int j = tid; j < m; j += kBThreads) {
        const ProjRec pr = view.proj[(int)(sm.ord.win[j] & 0xffffffffull)];
        sm.rec_a[j] = pr.a;
        sm.rec_b[j] = pr.b;
        sm.mask[j] = (uint8_t)box_grid_mask<2, 4>(pr, (float)(tx * kTile), (float)(ty * kTile), 8.0f, 4.0f);
      }
      if (pass == 2)
        for (int t = tid; t < (K + 1) * kW; t += kBThreads) dval[t] = 0.0f;
      __syncthreads();
      int cnt = 0;
      if (__any_sync(0xffffffffu, open)) {
        for (int j0 = 0; j0 < m; j0 += 32) {
          const bool rel = j0 + lane < m && ((sm.mask[j0 + lane] >> warp) & 1u);
          const unsigned rm = __ballot_sync(0xffffffffu, rel);
          if (rel) sm.list[warp][cnt + __popc(rm & ((1u << lane) - 1u))] = (uint16_t)(j0 + lane);
          cnt += __popc(rm);
        }
        __syncwarp();
      }
      for (int c0 = 0; c0 < cnt; c0 += 32) {
        unsigned todo = __ballot_sync(0xffffffffu, open);
        if (todo == 0u) break;
        // the lane's Gaussian: record, code, gradient sums
        const bool live = c0 + lane < cnt;
        const int j = live ? sm.list[warp][c0 + lane] : 0;
        const float4 a = sm.rec_a[j], b = sm.rec_b[j];
        const int64_t gi = (int64_t)(sm.ord.win[j] & 0xffffffffull);
        uint32_t ids[KR / 2];
        float vals[KR], acc[KR], dop = 0.0f;
#pragma unroll
        for (int k = 0; k < KR; ++k) {
          int atom = -1;
          float v = 0.0f;
          if (live && k < K) {
            atom = topk_idx[gi * K + k];
            v = topk_val[gi * K + k];
          }
          const bool ok = atom >= 0 && atom < C;
          const uint32_t id = ok ? (uint32_t)atom : (uint32_t)C;  // the row's zero word
          if (k & 1) ids[k / 2] |= id << 16;
          else ids[k / 2] = id;
          vals[k] = ok ? v : 0.0f;
          acc[k] = 0.0f;
        }
        // the open pixels in steps of kNP, the next step's rows on their way
        // into the other half of the warp's buffer
        int next[kNP];
        auto advance = [&](int half) {
#pragma unroll
          for (int u = 0; u < kNP; ++u) {
            next[u] = todo ? __ffs(todo) - 1 : -1;
            todo &= todo - 1u;  // 0 stays 0
            if (next[u] >= 0)
              stage_row<kVec>(rows + (half * kNP + u) * rw,
                              gblock + ((int64_t)(next[u] >> 3) * cam.width + (next[u] & 7)) * C, C, lane);
          }
          asm volatile("cp.async.commit_group;" ::: "memory");
        };
        advance(0);
        for (int half = 0; next[0] >= 0; half ^= 1) {
          BwdPixel px[kNP];
          const float* row[kNP];
          int cur[kNP];
#pragma unroll
          for (int u = 0; u < kNP; ++u) {
            const int p = cur[u] = next[u];
            px[u].on = p >= 0;
            px[u].x = (float)(bx + (p & 7));
            px[u].y = (float)(by + ((p & 31) >> 3));
            px[u].T = __shfl_sync(0xffffffffu, T, p & 31);
            px[u].S = __shfl_sync(0xffffffffu, S, p & 31);
            px[u].Sb = __shfl_sync(0xffffffffu, Sb, p & 31);
            row[u] = rows + (half * kNP + u) * rw;
          }
          advance(half ^ 1);
          asm volatile("cp.async.wait_group 1;" ::: "memory");
          __syncwarp();
          if (pass == 1) walk_pixels<1, KR, kNP>(a, b, live, ids, vals, row, px, acc, dop);
          else walk_pixels<2, KR, kNP>(a, b, live, ids, vals, row, px, acc, dop);
#pragma unroll
          for (int u = 0; u < kNP; ++u)
            if (lane == cur[u]) { T = px[u].T; S = px[u].S; Sb = px[u].Sb; open = !px[u].stopped; }
          __syncwarp();  // these rows are overwritten by the copies after the next
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (pass == 2 && live) {
#pragma unroll
          for (int k = 0; k < KR; ++k)
            if (k < K && acc[k] != 0.0f) atomicAdd(&dval[k * kW + j], acc[k]);
          if (dop != 0.0f) atomicAdd(&dop_sum[j], dop);
        }
      }
      __syncthreads();
      if (pass == 2) {
        // the window's gradient sums over the tile
        for (int t = tid; t < m * K; t += kBThreads) {
          const int j = t / K, k = t - j * K;
          const float v = dval[k * kW + j];
          if (v != 0.0f) atomicAdd(&d_val[(int64_t)(sm.ord.win[j] & 0xffffffffull) * K + k], v);
        }
        for (int j = tid; j < m; j += kBThreads)
          if (dop_sum[j] != 0.0f) atomicAdd(&d_opacity[sm.ord.win[j] & 0xffffffffull], dop_sum[j]);
      }
      if (!__syncthreads_or(open)) break;
    }
    __syncthreads();
  }
}

}  // namespace

// The block kernel's largest K, and the shared memory it takes.
constexpr int kBlockK = 16;
constexpr int kBlockPixels = 2;  // most pixels of a warp in flight (K <= 8; one beyond, by registers)
size_t bwd_block_smem(int C, int K) {
  return ((sizeof(BwdBlockSmem) + 15) & ~(size_t)15) +
         sizeof(float) * ((size_t)kBWarps * 2 * kBlockPixels * row_words(C) + (size_t)BOrder::kWin * (K + 1));
}

bool bwd_stages(int K) { return (size_t)K * BOrder::kWin * (sizeof(float) + sizeof(short)) <= kBStageMaxBytes; }

size_t render_bwd_smem_bytes(int C, int K) {
  return sizeof(BwdSmem) + sizeof(float) * ((size_t)kBWarps * C + (size_t)BOrder::kWin * (K + 1)) +
         (bwd_stages(K) ? (size_t)K * BOrder::kWin * (sizeof(float) + sizeof(short)) : 0);
}

cudaError_t launch_render_bwd(const ViewJob& v, const int32_t* topk_idx,
                              const float* topk_val, int K, int C, const float* dL_dcodes, float* d_val,
                              float* d_opacity, cudaStream_t st) {
  const int ntiles = v.cam.gx * v.cam.gy;
  if (ntiles <= 0) return cudaSuccess;
  if (K <= kBlockK) {
    const bool vec = C % 4 == 0 && ((uintptr_t)dL_dcodes & 15u) == 0;
    auto bk = vec ? (K <= 4   ? render_bwd_block_kernel<4, kBlockPixels, true>
                     : K <= 8 ? render_bwd_block_kernel<8, kBlockPixels, true>
                              : render_bwd_block_kernel<16, 1, true>)
                  : (K <= 4   ? render_bwd_block_kernel<4, kBlockPixels, false>
                     : K <= 8 ? render_bwd_block_kernel<8, kBlockPixels, false>
                              : render_bwd_block_kernel<16, 1, false>);
    const size_t bytes = bwd_block_smem(C, K);
    cudaError_t be = cudaFuncSetAttribute(bk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (be != cudaSuccess) return be;
    bk<<<ntiles, kBThreads, bytes, st>>>(v, topk_idx, topk_val, K, C, dL_dcodes, d_val, d_opacity);
    g_launches += 1;
    return cudaGetLastError();
  }
  const size_t smem = render_bwd_smem_bytes(C, K);
  auto kern = bwd_stages(K) ? render_bwd_kernel<true> : render_bwd_kernel<false>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  kern<<<ntiles, kBThreads, smem, st>>>(v, topk_idx, topk_val, K, C, dL_dcodes, d_val, d_opacity);
  g_launches += 1;
  return cudaGetLastError();
}

}  // namespace scoup
