// render_mma.cu -- sparse coefficient rendering (Sec. 4.3, Eq. 7) as a
// tensor-core contraction.
//
// For one 16x16 tile, What(p) = sum_i e_i(p) w^_i over the tile's
// front-to-back list.  Cut the list into chunks of 32 Gaussians: the weights
// of a chunk form a 256 x 32 matrix E (pixels x Gaussians, e_i(p) or 0) and
// its K-sparse codes a dense 32 x C matrix W, so the tile's code rows are
// the sum over chunks of E W.  The kernel keeps that sum in tensor memory
// (two 128-pixel halves x C FP32 columns) and adds every chunk with
// tcgen05.mma; the rows leave the SM once, at the end of the tile.
//
// One CTA of 256 threads per tile, two CTAs per SM.  A CTA orders its list
// window by window as in the uplift (tile_order.cuh).  Per chunk every thread
// walks its pixel front to back over the chunk's Gaussians (the binary32
// exponent, alpha test and T-stop rule of the uplift) and writes its row of E,
// the threads expand the chunk's codes into W, and warp 0 issues the chunk's
// MMAs and commits them to the completion barrier, on which the next chunk's
// writes wait.  The bf16 operands are split, e = e_hi +
// e_lo and w = w_hi + w_lo (each part rounded to bf16), and three MMAs add
// E_hi W_hi + E_hi W_lo + E_lo W_hi.  With u = 2^-8 (bf16 unit roundoff)
// each split leaves u^2 of its value and the dropped E_lo W_lo is below u^2
// of the product: at most about 3 u^2 = 3 * 2^-16 (4.6e-5) relative per
// product before FP32 accumulation.  A chunk in which a pixel half has no
// weight issues no MMA for that half.
//
// What bounds it is latency: ordering, staging, walk and epilogue of a tile
// follow each other (at 1080p, 1M Gaussians, C = 256, cycles: order 12k, stage
// 7k, walk 24k, expansion and barriers 7k, epilogue 11k of 63k), and with one
// CTA per SM the issue slots are 35 % used.  At C = 256 a tile takes all 512
// TMEM columns, so two CTAs cannot both hold an accumulator: it is allocated
// only in front of the first MMA, and the SM's other CTA orders, stages and
// walks its first chunk until this one frees it.  One chunk buffer in place of
// two and the MMAs issued by a walker warp make room for the second CTA (64 KB
// less shared memory, 128 registers a thread).  1080p with query, 1M
// Gaussians, C = 256: 2.56 -> 2.13 ms; forward and backward at 800 x 600 1.93
// -> 1.87 ms; a grid that does not fill the SMs once (161 x 119, C = 64) waits
// for its single buffer, 129 -> 134 us.
//
// The work per chunk is kept down: a warp walks only the Gaussians that may
// reach its 8 x 4 block and scatters their weights into E (all 32 of a chunk
// in 16 x 2 blocks before: 161 x 119 146 -> 129 us, 800 x 600 1.96 -> 1.93 ms,
// 1080p 2.59 -> 2.56 ms); codes are merged and split into their bf16 parts
// once per window and not per chunk, the warps a Gaussian may reach are a byte
// staged with it, the walk multiplies the transmittance down without a test
// per step and masks the weights behind the stop, and E and W are cleared only
// where they were written (155 -> 146 us, 2.04 -> 2.02 ms and 2.87 -> 2.83 ms
// for the same three).  Half-tile CTAs (128 pixels) take 1.84 ms where whole
// tiles with one CTA per SM take 1.61 ms (1080p): every half orders and stages
// the tile's list again.
//
// Every wait on a completion is bounded; a wait that gives up sets the timeout
// status and the tile ends; TMEM is freed on every path (the allocation itself
// waits for the SM's other CTA, which never waits for this one).  The rows are
// written at the end through the chunk buffer, in coalesced 256-byte pieces.
#include <cuda_bf16.h>
#include <math.h>

#include "sm100_ptx.cuh"
#include "tile_order.cuh"

namespace scoup {
namespace {

constexpr int kMThreads = 256;  // one thread per pixel of the 16 x 16 tile
constexpr int kMWarps = kMThreads / 32;
constexpr int kChunk = 32;      // Gaussians per chunk (contraction depth of one round of MMAs)
constexpr int kMaxN = 256;      // widest code row: two 128-lane halves of N FP32 TMEM columns
constexpr int kMaxK = 16;       // largest Top-K staged per window
constexpr uint32_t kWaitIters = 1u << 22;
using MOrder = OrderSmem<256, 10>;

// Operand tiles are K-major without swizzle, built from 8-row x 16-byte core
// matrices: the 4 core matrices of an 8-row group (32 bf16 along K) are
// adjacent (LBO = 128 bytes) and the 8-row groups follow each other (SBO =
// 512 bytes).  A K = 16 slice starts 2 core matrices (256 bytes) further.
constexpr uint32_t kLBO = 128, kSBO = 512;
constexpr int kEBytes = 128 * kChunk * 2;    // one 128-pixel E tile: 8 KB
constexpr int kWBytes = kMaxN * kChunk * 2;  // one W tile: 16 KB

__device__ __forceinline__ int core_off(int row, int k) {
  return (row >> 3) * (int)kSBO + (k >> 3) * (int)kLBO + (row & 7) * 16 + (k & 7) * 2;
}

struct alignas(128) ChunkBuf {
  unsigned char e[2][2][kEBytes];  // [hi, lo][pixel half]
  unsigned char w[2][kWBytes];     // [hi, lo]
};

template <int KT>
struct RenderMmaSmem {
  ChunkBuf buf;
  MOrder ord;
  float4 rec_a[MOrder::kWin + 1];  // one more: a record that no pixel accepts
  float4 rec_b[MOrder::kWin + 1];
  uint32_t code_val[KT * MOrder::kWin];  // [k][window position]: the value's bf16 parts, hi | lo << 16
  short code_idx[KT * MOrder::kWin];     // atom; -1: no entry, or added to an earlier entry of the atom
  uint8_t rows[MOrder::kWin];            // bit w: the Gaussian may reach warp w's 8 x 4 block
  uint64_t mma_done;  // the MMAs that read the chunk buffer have completed
  uint32_t tmem;
  int any_e[kMWarps];
  int abort;  // a wait gave up
  unsigned long long cnt[2];
};

constexpr int kPieceBytes = 256;  // of a row, per epilogue store
static_assert(sizeof(ChunkBuf) >= kMWarps * 32 * kPieceBytes, "the epilogue stages a piece per row in the buffer");
static_assert(sizeof(RenderMmaSmem<kMaxK>) + 128 <= 113 * 1024, "two CTAs per SM");

// TMEM columns: a power of two holding two halves of Np columns, each half a
// multiple of 32 columns (the width of one tcgen05.ld).
__host__ __device__ inline uint32_t mma_tmem_cols(int Np) {
  uint32_t c = 64;
  while (c < 2u * (uint32_t)Np) c <<= 1;
  return c;
}

__device__ __forceinline__ void split_bf16x2(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  const float2 hf = __bfloat1622float2(h);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x - hf.x, y - hf.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// Walks the thread's pixel over window positions j0 .. j0 + 31 and writes its
// row of E (hi and lo parts, zero where a Gaussian does not contribute);
// returns whether any weight of the row is nonzero.  T below the cutoff: the
// pixel has stopped, and Tout holds its transmittance.
// Only the Gaussians that may pass the alpha test at some pixel of the warp's
// 8 x 4 block (sm.rows) are walked, eight at a time in list order, and their
// weights scattered to their columns.  `held`: the columns of the buffer's row
// groups that may hold weights of an earlier chunk (bit per column, uniform
// over the warp), cleared here eight columns at a time.
template <int KT>
__device__ __forceinline__ bool walk_chunk(const RenderMmaSmem<KT>& sm, int j0, int m, int wbase, float fpx, float fpy,
                                           float& T, float& Tout, int& last, unsigned& n_eval, unsigned& n_contrib,
                                           unsigned& held, unsigned char* e_hi, unsigned char* e_lo) {
  unsigned rel = 0u;
  if (!__all_sync(0xffffffffu, T < 1e-4f)) {
    const int jl = j0 + (int)(threadIdx.x & 31);
    rel = __ballot_sync(0xffffffffu, jl < m && ((sm.rows[jl] >> (threadIdx.x >> 5)) & 1u));
  }
#pragma unroll
  for (int g = 0; g < kChunk / 8; ++g)
    if (((held | rel) >> (8 * g)) & 0xffu) {  // warp-uniform
      *reinterpret_cast<uint4*>(e_hi + g * (int)kLBO) = make_uint4(0u, 0u, 0u, 0u);
      *reinterpret_cast<uint4*>(e_lo + g * (int)kLBO) = make_uint4(0u, 0u, 0u, 0u);
    }
  held = rel;
  uint32_t any = 0u;
  while (rel != 0u && !__all_sync(0xffffffffu, T < 1e-4f)) {
    // the next eight (past the last: a record that never passes, tau = +inf).
    // Independent per Gaussian: exponent, alpha test and alpha (8 chains in
    // flight).
    int jj[8];
    float al[8], om[8];
    unsigned pass = 0u;
    const int cnt = min(8, __popc(rel));
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      jj[u] = __ffs(rel) - 1;  // -1: none
      rel &= rel - 1u;
      const int j = jj[u] >= 0 ? j0 + jj[u] : MOrder::kWin;
      const float4 a = sm.rec_a[j];
      const float4 b = sm.rec_b[j];
      const float dx = a.x - fpx, dy = a.y - fpy;
      const float power = fmaf(dx, fmaf(a.z, dx, __fmul_rn(a.w, dy)), __fmul_rn(__fmul_rn(b.x, dy), dy));
      const bool ok = power <= 0.0f && power >= b.z;
      al[u] = ok ? fminf(0.99f, b.y * __expf(power)) : 0.0f;
      om[u] = 1.0f - al[u];
      if (ok) pass |= 1u << u;
    }
    // front to back: T only falls, so once a product is below the cutoff all
    // later ones are, and the running product needs no test of its own: the
    // weights from the stop on are masked afterwards
    float ev[8];
    const float T0 = T;
    unsigned n_ok = 0u;  // Gaussians in front of the stop
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float test = __fmul_rn(T, om[u]);
      const bool ok = test >= 1e-4f;
      ev[u] = ok ? al[u] * T : 0.0f;
      n_ok += ok ? 1u : 0u;
      T = test;
    }
    if (T0 >= 1e-4f) {  // the pixel was open
      pass &= (1u << n_ok) - 1u;
      n_contrib += __popc(pass);
      // examined: up to and including the stop
      n_eval += min(cnt, (int)n_ok + 1);
      Tout = T;
      if (n_ok < 8u) {
        Tout = T0;  // the transmittance in front of the stop
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (u < (int)n_ok) Tout = __fmul_rn(Tout, om[u]);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if ((pass >> u) & 1u) last = wbase + j0 + jj[u] + 1;
    }
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      uint32_t hi, lo;
      split_bf16x2(ev[u], ev[u + 1], hi, lo);
      any |= hi;
      if (jj[u] >= 0) {  // uniform
        const int o = (jj[u] >> 3) * (int)kLBO + (jj[u] & 7) * 2;
        *reinterpret_cast<uint16_t*>(e_hi + o) = (uint16_t)hi;
        *reinterpret_cast<uint16_t*>(e_lo + o) = (uint16_t)lo;
      }
      if (jj[u + 1] >= 0) {
        const int o = (jj[u + 1] >> 3) * (int)kLBO + (jj[u + 1] & 7) * 2;
        *reinterpret_cast<uint16_t*>(e_hi + o) = (uint16_t)(hi >> 16);
        *reinterpret_cast<uint16_t*>(e_lo + o) = (uint16_t)(lo >> 16);
      }
    }
  }
  return any != 0u;
}

__device__ __forceinline__ uint32_t pack2_bf16(float x, float y) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// 32 columns c0 .. c0 + 31 of the pixel's row (fewer at the end of the row).
__device__ __forceinline__ void store_cols(void* __restrict__ out, int64_t pix, int C, int c0, bool bf16,
                                           const float (&v)[32]) {
  const int nc = min(32, C - c0);
  if (bf16) {
    __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(out) + pix * C + c0;
    if (nc == 32 && (C & 7) == 0) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        reinterpret_cast<uint4*>(o)[q] = make_uint4(pack2_bf16(v[8 * q], v[8 * q + 1]), pack2_bf16(v[8 * q + 2], v[8 * q + 3]),
                                                    pack2_bf16(v[8 * q + 4], v[8 * q + 5]),
                                                    pack2_bf16(v[8 * q + 6], v[8 * q + 7]));
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (i < nc) o[i] = __float2bfloat16_rn(v[i]);
    }
  } else {
    float* o = reinterpret_cast<float*>(out) + pix * C + c0;
    if (nc == 32 && (C & 3) == 0) {
#pragma unroll
      for (int q = 0; q < 8; ++q)
        reinterpret_cast<float4*>(o)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (i < nc) o[i] = v[i];
    }
  }
}

// One CTA per tile, two CTAs per SM.
template <int KT>
__global__ void __launch_bounds__(kMThreads, 2) render_mma_kernel(
    const __grid_constant__ ViewJob view, const int32_t* __restrict__ topk_idx,
    const float* __restrict__ topk_val, int K, int C, void* __restrict__ out, int out_bf16,
    float* __restrict__ out_T, int32_t* __restrict__ out_last) {
  extern __shared__ __align__(128) unsigned char msm_raw[];
  unsigned char* base = msm_raw + ((128u - (ptx::smem_u32(msm_raw) & 127u)) & 127u);
  RenderMmaSmem<KT>& sm = *reinterpret_cast<RenderMmaSmem<KT>*>(base);
  const CamArgs& cam = view.cam;
  WsHeader* __restrict__ const hdr = view.hdr;
  const ProjRec* __restrict__ const proj = view.proj;
  if (hdr->status & kStatCapacity) return;  // set by the binning before this launch: uniform
  const int tile = (int)blockIdx.x;
  const TileList list = tile_list(view.keys, view.tile_start, nullptr, view.shift, cam.gx, tile);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tx = tile % cam.gx, ty = tile / cam.gx;
  const int n = list.n;
  const int Np = (C + 15) & ~15;  // MMA N: C rounded up to a multiple of 16
  const uint32_t cols = mma_tmem_cols(Np), half_cols = cols / 2;

  if (tid == 0) {
    ptx::mbar_init(&sm.mma_done, 1);
    ptx::fence_mbar_init();
    sm.cnt[0] = sm.cnt[1] = 0ull;
    sm.abort = 0;
  }
  // a warp's pixels are an 8 x 4 block, its rows of E in that order
  const int wx = tx * kTile + (warp & 1) * 8, wy = ty * kTile + (warp >> 1) * 4;
  const int px = wx + (lane & 7), py = wy + (lane >> 3);
  const bool inside = px < cam.width && py < cam.height;
  const int half = tid >> 7, row = tid & 127;  // E row and TMEM lane of this pixel
  float T = inside ? 1.0f : 0.0f, Tout = T;
  int last = 0;
  // W starts cleared; each thread clears what it wrote for the last chunk
  for (int i = tid; i < 2 * kWBytes / 16; i += kMThreads)
    reinterpret_cast<uint4*>(sm.buf.w[0])[i] = make_uint4(0u, 0u, 0u, 0u);
  constexpr int kPer = (kChunk * KT + kMThreads - 1) / kMThreads;  // W entries of a thread per chunk
  constexpr int kNone = 0xffff;
  int wrote[kPer];  // offsets written for the last chunk
#pragma unroll
  for (int q = 0; q < kPer; ++q) wrote[q] = kNone;
  unsigned held = 0xffffffffu;
  if (tid == 0) {
    sm.rec_a[MOrder::kWin] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    sm.rec_b[MOrder::kWin] = make_float4(0.0f, 0.0f, INFINITY, 0.0f);
  }
  // code rows by 16-byte loads (K = 4, 8, ..; the arrays may start anywhere)
  const bool vec =
      (K & 3) == 0 && ((reinterpret_cast<uintptr_t>(topk_idx) | reinterpret_cast<uintptr_t>(topk_val)) & 15) == 0;
  const OrderBuckets bk = order_buckets<MOrder>(hdr);
  order_init<MOrder, 16>(sm.ord, list, bk);

  unsigned n_eval = 0, n_contrib = 0;
  unsigned acc_init = 0u;  // bit h: pixel half h has received an MMA
  bool aborted = false, all_done = false;
  int wbase = 0, issued = 0;  // list positions in front of the window; chunks with MMAs
  OrderState ost;
  while (!all_done && !aborted) {
    const int m = n > 0 ? order_next_window<MOrder, 16>(sm.ord, list, bk, ost, hdr) : 0;
    if (m <= 0) break;  // list exhausted, or an inconsistency (status already set)
    // the window's records, which warps' blocks they may reach, and their code
    // rows (one thread per Gaussian, all loads in flight together)
    for (int j = tid; j < m; j += kMThreads) {
      const int64_t g = (int64_t)(sm.ord.win[j] & 0xffffffffull);
      const ProjRec pr = proj[g];
      int32_t ai[KT];
      float av[KT];
      if (vec) {
#pragma unroll
        for (int k4 = 0; k4 < KT / 4; ++k4)
          if (4 * k4 < K) {
            const int4 a = reinterpret_cast<const int4*>(topk_idx + g * K)[k4];
            const float4 v = reinterpret_cast<const float4*>(topk_val + g * K)[k4];
            ai[4 * k4] = a.x; ai[4 * k4 + 1] = a.y; ai[4 * k4 + 2] = a.z; ai[4 * k4 + 3] = a.w;
            av[4 * k4] = v.x; av[4 * k4 + 1] = v.y; av[4 * k4 + 2] = v.z; av[4 * k4 + 3] = v.w;
          }
      } else {
#pragma unroll
        for (int k = 0; k < KT; ++k)
          if (k < K) {
            ai[k] = topk_idx[g * K + k];
            av[k] = topk_val[g * K + k];
          }
      }
      sm.rec_a[j] = pr.a;
      sm.rec_b[j] = pr.b;
      sm.rows[j] = (uint8_t)box_grid_mask<2, 4>(pr, (float)(tx * kTile), (float)(ty * kTile), 8.0f, 4.0f);
      // repeated atoms of one code add up in the first of them
#pragma unroll
      for (int k = 0; k < KT; ++k) {
        int atom = -1;
        if (k < K) {
          if (!(ai[k] >= 0 && ai[k] < C)) ai[k] = -1;
#pragma unroll
          for (int k2 = k + 1; k2 < KT; ++k2)
            if (k2 < K && ai[k] >= 0 && ai[k2] == ai[k]) { av[k] += av[k2]; ai[k2] = -1; }
          atom = ai[k];
          const __nv_bfloat16 h = __float2bfloat16_rn(av[k]);
          const __nv_bfloat16 l = __float2bfloat16_rn(av[k] - __bfloat162float(h));
          sm.code_val[k * MOrder::kWin + j] =
              (uint32_t)__bfloat16_as_ushort(h) | ((uint32_t)__bfloat16_as_ushort(l) << 16);
        }
        sm.code_idx[k * MOrder::kWin + j] = (short)atom;
      }
    }
    __syncthreads();
    for (int j0 = 0; j0 < m; j0 += kChunk) {
      ChunkBuf& cb = sm.buf;
      // the MMAs that last read the buffer have completed (every thread waits)
      if (issued > 0 && !ptx::mbar_wait_bounded(&sm.mma_done, (uint32_t)(issued - 1) & 1u, kWaitIters)) {
        atomicOr(&hdr->status, kStatTimeout);
        *(volatile int*)&sm.abort = 1;
      }
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        if (wrote[q] != kNone) {
          *reinterpret_cast<uint16_t*>(cb.w[0] + wrote[q]) = 0;
          *reinterpret_cast<uint16_t*>(cb.w[1] + wrote[q]) = 0;
        }
        wrote[q] = kNone;
      }
      const bool any = walk_chunk<KT>(sm, j0, m, wbase, (float)px, (float)py, T, Tout, last, n_eval, n_contrib, held,
                                      cb.e[0][half] + core_off(row, 0), cb.e[1][half] + core_off(row, 0));
      const unsigned wany = __ballot_sync(0xffffffffu, any);
      if (lane == 0) sm.any_e[warp] = wany != 0u;
      __syncthreads();
      if (*(volatile int*)&sm.abort) {  // set before the barrier
        aborted = true;
        break;
      }
      const bool any0 = (sm.any_e[0] | sm.any_e[1] | sm.any_e[2] | sm.any_e[3]) != 0;
      const bool any1 = (sm.any_e[4] | sm.any_e[5] | sm.any_e[6] | sm.any_e[7]) != 0;
      if (any0 || any1) {
        // the accumulator: allocated late, so that the SM's other CTA orders,
        // stages and walks while this one holds all of tensor memory
        if (acc_init == 0u && warp == 0) {
          ptx::tmem_alloc(&sm.tmem, cols);
          ptx::tmem_relinquish();
          ptx::tc_fence_before();
        }
        // W (hi, lo): entry (atom, Gaussian)
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
          const int t = tid + q * kMThreads, jc = t & (kChunk - 1), k = t / kChunk, j = j0 + jc;
          if (k >= K || j >= m) continue;
          const int atom = sm.code_idx[k * MOrder::kWin + j];
          if (atom < 0) continue;
          const uint32_t v = sm.code_val[k * MOrder::kWin + j];
          const int o = core_off(atom, jc);
          *reinterpret_cast<uint16_t*>(cb.w[0] + o) = (uint16_t)v;
          *reinterpret_cast<uint16_t*>(cb.w[1] + o) = (uint16_t)(v >> 16);
          wrote[q] = o;
        }
      }
      ptx::fence_async_shared();  // E and W are read by the tensor core (async proxy)
      const bool open = __syncthreads_or(T >= 1e-4f);
      if (any0 || any1) {
        if (warp == 0) {
          // the warp builds the descriptors together (uniform registers), lane 0 issues
          ptx::tc_fence_after();
          const uint32_t idesc = ptx::idesc_bf16_f32(128, Np), tmem = *(volatile uint32_t*)&sm.tmem;
          const uint64_t eb = ptx::smem_desc_kmajor_none(ptx::smem_u32(cb.e[0][0]), kLBO, kSBO);
          const uint64_t wb = ptx::smem_desc_kmajor_none(ptx::smem_u32(cb.w[0]), kLBO, kSBO);
          if (lane == 0) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              if (!(h ? any1 : any0)) continue;
              const uint32_t d = tmem + (uint32_t)h * half_cols;
#pragma unroll
              for (int pass = 0; pass < 3; ++pass)
#pragma unroll
                for (int ks = 0; ks < kChunk / 16; ++ks)
                  ptx::mma_f16(d, eb + ((((pass == 2 ? 2 : 0) + h) * kEBytes + ks * 2 * (int)kLBO) >> 4),
                               wb + (((pass == 1 ? kWBytes : 0) + ks * 2 * (int)kLBO) >> 4), idesc,
                               (((acc_init >> h) & 1u) || pass > 0 || ks > 0) ? 1u : 0u);
            }
            ptx::mma_commit(&sm.mma_done);
          }
          __syncwarp();
        }
        acc_init |= (any0 ? 1u : 0u) | (any1 ? 2u : 0u);
        ++issued;
      }
      if (!open) {
        all_done = true;
        break;
      }
    }
    wbase += m;
  }

  // every MMA has completed before the accumulator is read and TMEM freed
  bool fin_ok = true;
  if (tid == 0 && issued > 0) {
    fin_ok = ptx::mbar_wait_bounded(&sm.mma_done, (uint32_t)(issued - 1) & 1u, kWaitIters);
    if (!fin_ok) atomicOr(&hdr->status, kStatTimeout);
  }
  const bool bad = __syncthreads_or(!fin_ok) || aborted;
  const uint32_t tmem = *(volatile uint32_t*)&sm.tmem;  // with acc_init only
  ptx::tc_fence_after();

  // epilogue: each thread reads its own pixel's row (TMEM lane)
  const int q = warp & 3;
  const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)half * half_cols;
  const int64_t pix = (int64_t)py * cam.width + px;
  const bool have = ((acc_init >> half) & 1u) && !bad;  // uniform over the warp
  // Rows that split into 256-byte pieces (bf16 with C a multiple of 128, FP32
  // with C a multiple of 64) go through shared memory: the warp stages one
  // piece of each of its 32 pixel rows (16-byte chunks XOR-swizzled by row,
  // so neither the staging stores nor the reads conflict) in the chunk
  // buffer, free once the last MMA has completed, and writes two rows'
  // pieces with each coalesced warp store; other rows are stored per thread.
  const int esz = out_bf16 ? 2 : 4;
  const int piece_cols = kPieceBytes / esz;
  if (!bad && C == Np && C % piece_cols == 0 && ((uintptr_t)out & 15u) == 0) {
    unsigned char* stg = reinterpret_cast<unsigned char*>(&sm.buf) + warp * 32 * kPieceBytes;
    for (int p0 = 0; p0 < Np; p0 += piece_cols) {
      for (int c0 = p0; c0 < p0 + piece_cols; c0 += 32) {
        float v[32];
        if (have) {
          ptx::tmem_ld32(tb + (uint32_t)c0, v);
        } else {
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = 0.0f;
        }
        const int k0 = (c0 - p0) * esz / 16;  // first 16-byte chunk of these columns in the piece
        if (out_bf16) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            *reinterpret_cast<uint4*>(stg + lane * kPieceBytes + (((k0 + j) ^ lane) & 15) * 16) =
                make_uint4(pack2_bf16(v[8 * j], v[8 * j + 1]), pack2_bf16(v[8 * j + 2], v[8 * j + 3]),
                           pack2_bf16(v[8 * j + 4], v[8 * j + 5]), pack2_bf16(v[8 * j + 6], v[8 * j + 7]));
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            *reinterpret_cast<float4*>(stg + lane * kPieceBytes + (((k0 + j) ^ lane) & 15) * 16) =
                make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        }
      }
      __syncwarp();
#pragma unroll 4
      for (int r0 = 0; r0 < 32; r0 += 2) {
        const int r = r0 + (lane >> 4), ch = lane & 15;
        const uint4 val = *reinterpret_cast<const uint4*>(stg + r * kPieceBytes + ((ch ^ r) & 15) * 16);
        const int rx = wx + (r & 7), ry = wy + (r >> 3);
        if (rx < cam.width && ry < cam.height)
          *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(out) +
                                    ((int64_t)ry * cam.width + rx) * (int64_t)C * esz + p0 * esz + ch * 16) = val;
      }
      __syncwarp();
    }
  } else {
    for (int c0 = 0; c0 < Np; c0 += 32) {
      float v[32];
      if (have) {
        ptx::tmem_ld32(tb + (uint32_t)c0, v);
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = 0.0f;
      }
      if (inside && !bad) store_cols(out, pix, C, c0, out_bf16 != 0, v);
    }
  }
  if (inside) {
    if (out_T) out_T[pix] = Tout;
    if (out_last) out_last[pix] = last;
  }
  const unsigned we = __reduce_add_sync(0xffffffffu, n_eval);
  const unsigned wc = __reduce_add_sync(0xffffffffu, n_contrib);
  if (lane == 0) {
    atomicAdd(&sm.cnt[0], (unsigned long long)we);
    atomicAdd(&sm.cnt[1], (unsigned long long)wc);
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0 && acc_init != 0u) ptx::tmem_dealloc(tmem, cols);
  if (tid == 0) {
    atomicAdd(&hdr->evaluated, sm.cnt[0]);
    atomicAdd(&hdr->contributions, sm.cnt[1]);
  }
}

}  // namespace

bool render_mma_supported(int C, int K) { return C >= 1 && C <= kMaxN && K >= 1 && K <= kMaxK; }

size_t render_mma_smem_bytes(int K) {
  return (K <= 4 ? sizeof(RenderMmaSmem<4>) : K <= 8 ? sizeof(RenderMmaSmem<8>) : sizeof(RenderMmaSmem<16>)) + 128;
}

cudaError_t launch_render_mma(const ViewJob& v, const int32_t* topk_idx,
                              const float* topk_val, int K, int C, void* out, int out_bf16, float* out_T,
                              int32_t* out_last, cudaStream_t st) {
  const int ntiles = v.cam.gx * v.cam.gy;
  if (ntiles <= 0) return cudaSuccess;
  const size_t smem = render_mma_smem_bytes(K);
  const auto kernel = K <= 4 ? render_mma_kernel<4> : K <= 8 ? render_mma_kernel<8> : render_mma_kernel<16>;
  cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  kernel<<<ntiles, kMThreads, smem, st>>>(v, topk_idx, topk_val, K, C, out, out_bf16, out_T,
                                            out_last);
  g_launches += 1;
  return cudaGetLastError();
}

}  // namespace scoup
