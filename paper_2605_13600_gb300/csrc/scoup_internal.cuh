// scoup_internal.cuh -- shared definitions of the CUDA translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/scoup.h"
#include "../../include/scoup_selftest.h"

#include <atomic>

namespace scoup {

// Kernel launches issued by the library (every launcher adds its count).
extern std::atomic<long long> g_launches;

// Streaming multiprocessors of the current device (queried once per device);
// grid sizes of the grid-stride kernels are multiples of it.
int num_sms();

constexpr int kTile = 16;            // 16x16 pixel tiles define binning membership (3DGS)
constexpr int kTilePixels = kTile * kTile;

// Device status bits (workspace header).
constexpr int kStatCapacity = 1;
constexpr int kStatDeviceCheck = 2;
constexpr int kStatTimeout = 4;

// Workspace header: status word, depth range of the view's visible Gaussians,
// scene bounding box and counters, 256 bytes.  A scene has one (its status and
// the counters of the whole call); every view part of an uplift has its own,
// whose counters are merged into the scene's after each chunk of views.
struct WsHeader {
  int32_t status;
  int32_t max_dups_view;
  uint32_t drange[2];     // {min, max} float bits of visible depths
  uint32_t bbox[3][2];    // order-preserving bits of the means' bounding box
  unsigned long long visible;
  unsigned long long duplicates;
  unsigned long long evaluated;
  unsigned long long contributions;
  unsigned long long flushes;
  unsigned long long atomics;
  unsigned long long listed;
  unsigned long long split_windows;  // windows cut out of a depth bucket holding more than a window
  unsigned long long resumed_tiles;  // scene header: tiles that a second pass took up behind the depth cut
  uint32_t open_tiles;               // tiles still open behind the depth cut (length of open_list)
  uint32_t drain_ctr[2][2];          // scene header: item counters of each chunk lane's two drains
  uint32_t reserved[31];
};
static_assert(sizeof(WsHeader) == 256, "header size");

// Projected Gaussian of one view, 32 bytes:
//   a = (mx, my, qa, qb), b = (qc, opacity, tau, log2(opacity))
// power(dx, dy) = dx*(qa*dx + qb*dy) + (qc*dy)*dy and the Gaussian is
// accepted at a pixel iff tau <= power <= 0  (tau: smallest float with
// o*exp(tau) >= 1/255).
struct __align__(16) ProjRec {
  float4 a;
  float4 b;
};

// Conservative test of a whole grid of boxes at once: bit r * kCols + c is
// set when box (c, r) -- pixels x0 + c w .. x0 + c w + w - 1 by
// y0 + r h .. y0 + r h + h - 1 -- may hold a pixel centre with power >= tau.
// In offsets (u, v) = (x - mx, y - my) the accepted set is the ellipse
// E = {qa u^2 + qb u v + qc v^2 >= lvl}, with the level lvl a margin below
// tau that covers the binary32 rounding of the per-pixel exponent (the terms
// of the exponent reach |tau| times the ellipse's aspect ratio, so the margin
// grows with it).  For each row of boxes (a strip va <= v <= vb) the x-extent
// of E inside the strip is found in closed form: the right end of E's chord
// at height v is a concave function of v whose maximum is E's rightmost point
// (u_e, v_e), so over the strip it peaks at v = clamp(v_e, va, vb); the left
// end, by symmetry, at clamp(-v_e, va, vb).  A strip that misses E has no
// chord there (negative discriminant).  The extent is widened by 0.01 px.
template <int kCols, int kRows>
__device__ __forceinline__ uint32_t box_grid_mask(const ProjRec& r, float x0, float y0, float w, float h) {
  constexpr uint32_t kAll = kCols * kRows >= 32 ? 0xffffffffu : ((1u << (kCols * kRows)) - 1u);
  const float mx = r.a.x, my = r.a.y, qa = r.a.z, qb = r.a.w, qc = r.b.x, tau = r.b.z;
  const float det = 4.0f * qa * qc - qb * qb;  // > 0 for a negative-definite exponent
  if (!(qa < 0.0f && qc < 0.0f && det > 0.0f && tau < 0.0f)) return kAll;
  const float aspect = 4.0f * (qa + qc) * (qa + qc) / det;  // >= the ratio of the ellipse's axes squared
  const float lvl = tau - (0.02f + 2e-3f * fabsf(tau) + 1e-5f * fabsf(tau) * aspect);
  const float c4 = 4.0f * qa * lvl;                           // > 0
  const float ue = sqrtf(4.0f * qc * lvl / det);              // rightmost point of E
  const float ve = -qb * ue / (2.0f * qc);
  const float inv2a = 0.5f / qa;                              // < 0
  uint32_t mask = 0u;
#pragma unroll
  for (int row = 0; row < kRows; ++row) {
    const float va = y0 + (float)row * h - my - 0.01f, vb = va + (h - 1.0f) + 0.02f;
    const float vr = fminf(fmaxf(ve, va), vb), vl = fminf(fmaxf(-ve, va), vb);
    const float dr = fmaf(-det, vr * vr, c4), dl = fmaf(-det, vl * vl, c4);
    if (dr < 0.0f && dl < 0.0f) continue;
    // chord roots (-qb v -/+ sqrt(D)) / (2 qa): the right end takes -sqrt(D)
    const float xr = mx + (-qb * vr - sqrtf(fmaxf(dr, 0.0f))) * inv2a + 0.01f;
    const float xl = mx + (-qb * vl + sqrtf(fmaxf(dl, 0.0f))) * inv2a - 0.01f;
#pragma unroll
    for (int col = 0; col < kCols; ++col) {
      const float bx0 = x0 + (float)col * w;
      if (xr >= bx0 && xl <= bx0 + (w - 1.0f)) mask |= 1u << (row * kCols + col);
    }
  }
  return mask;
}

// One relevancy term of App. B, Eq. 9: e^{a s_q} / (e^{a s_q} + e^{a s_k}) =
// 1 / (1 + e^{a (s_k - s_q)}), with s_k the largest canonical similarity (the
// term decreases in s_k, so it is the minimum over the canonical phrases).
// The exponential is the SFU's base-2 one and the quotient the fast
// reciprocal (about 2^-21 relative together); both relevancy paths use this
// one function, so they agree bit for bit.
__device__ __forceinline__ float relevancy_term(float alpha, float s_canon_max, float s_query) {
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(alpha * 1.4426950408889634f * (s_canon_max - s_query)));
  return fminf(1.0f, __fdividef(1.0f, 1.0f + e));
}

// Region maps and code tables of one view, one per semantic level (a single
// level for scoup_uplift; up to three for scoup_uplift_levels).
constexpr int kMaxLevels = 3;
struct LevelCodes {
  const int32_t* rmap[kMaxLevels];  // this view's region map of each level
  const int32_t* ci[kMaxLevels];    // code tables [R, s] of each level
  const float* cv[kMaxLevels];
  int s[kMaxLevels];
  int R[kMaxLevels];
  int L;      // number of levels
  int s_tot;  // sum of s over the levels (entries of a combined region code)
};

struct CamArgs {
  float vm[12];
  float fx, fy, cx, cy;
  int width, height;
  int gx, gy;  // tile grid
};

// One view of a chunk, as the drain kernel takes it.
struct TileJob {
  CamArgs cam;
  LevelCodes lc;
  const ProjRec* proj;
  const unsigned long long* keys;
  const uint32_t* tile_start;
  const uint32_t* zcut;        // depth cut per tile block, or null (DepthCut below)
  uint32_t* open_bits;
  uint32_t* open_list;
  float* pix_state;
  float* accum;
  float* comp;                 // compensation array (compensated form) or null
  WsHeader* hdr;        // the view's own header: depth range, counters, status
  WsHeader* scene_hdr;  // the scene's header, into which the view's counters are merged
  int C, Crow;          // accumulator rows hold Crow = levels x C floats
  int shift;            // of the view's tile lists (TileList)
  int tiles;
};

// Scene copy in spatial (Morton) order: one 48-byte record per Gaussian, with
// what of the projection does not depend on the view; orig[p] is the caller's
// index.
struct __align__(16) SceneRec {
  float4 mean_op;  // mean, opacity
  float4 cov_a;    // Sigma3: S00, S01, S02, S11
  float4 cov_b;    // S12, S22, alpha-threshold exponent tau, the caller's index (int bits)
};
struct SceneP {
  SceneRec* rec;   // [n]
  int32_t* orig;   // [n]
};

// Depth cut.  A tile's pixels are opaque long before its list ends (of 4500
// listed Gaussians per tile of a 1M-Gaussian view about 280 are composited),
// so each block of 2 x 2 tiles gets a depth zcut, estimated from a sample of
// the scene's optical depth, and a Gaussian is listed only if it lies in
// front of the cut of some block that its rectangle meets.  A tile's list is
// then complete up to its cut, and keys behind it are left out.  A tile that
// is still open at its cut is recorded, with its pixels' state, and a second
// pass lists what lies behind the cut for the recorded tiles alone.  The
// estimate decides speed only: every tile sees its whole list, in order.
// Taken by the uplift's chunks of views of large scenes (use_depth_cut).
constexpr int kCutBins = 512;                // 64 per octave of depth, from 0.2 up
constexpr uint32_t kCutBase = 0x3E4CCCCDu;   // bits of 0.2f
constexpr int kCutShift = 17;
constexpr uint32_t kNoCut = 0xffffffffu;
__host__ __device__ inline int cut_blocks(int g) { return (g + 1) >> 1; }
__host__ __device__ inline int open_words(int gx) { return (cut_blocks(gx) + 31) >> 5; }  // per row of blocks

// Tile lists.  A list belongs to a block of 2 x 2 tiles: a Gaussian meets
// several neighbouring tiles, so a view has less than half as many (Gaussian,
// block) items as (Gaussian, tile) ones to count, place and write, and a tile
// takes its own out of the block's list in the pass over it that it makes
// anyway.  Key: depth bits << 32 | index << 4 | the block's tiles that the
// rectangle meets (bit (ty & 1) * 2 + (tx & 1)).  Views less than 4 tiles wide
// or high, where blocks save nothing, and scenes of 2^28 Gaussians, whose
// index leaves no room for the bits, have one list per tile and no bits
// (shift 0), and so have images dense in Gaussians (list_shift).
struct TileList {
  const unsigned long long* keys;
  int n;             // keys of the list; those of the tile are among them
  uint32_t bit;      // the tile's bit (0: every key is the tile's)
  int id_shift;      // of the index in the key's low word
  uint32_t cut;      // the tile's depth cut
  __device__ __forceinline__ bool mine(unsigned long long k) const { return ((uint32_t)k & bit) == bit; }
  // the key without tile bits: depth bits << 32 | index
  __device__ __forceinline__ unsigned long long plain(unsigned long long k) const {
    return (k & 0xffffffff00000000ull) | ((uint32_t)k >> id_shift);
  }
  // the largest key of a list that stands for the plain key k
  __device__ __forceinline__ unsigned long long last_as_listed(unsigned long long k) const {
    return (k & 0xffffffff00000000ull) | ((uint32_t)k << id_shift) | ((1u << id_shift) - 1u);
  }
};
//
// A block's list serves the binning (a quarter of the lists to count and fill)
// and costs every tile the keys of its three neighbours, read once per window.
// With many Gaussians to a tile the windows' passes decide: uplift of 12 views
// (ms, blocks / tiles; Gaussians per tile of the image): 526 2.66 / 2.86, 631
// 0.90 / 0.87, 2105 1.99 / 1.79, 2560 0.79 / 0.71, 8550 3.68 / 2.49; one
// render the same way around (526 0.745 / 0.754, 2105 0.73 / 0.68, 8550 1.69 /
// 1.61).  Behind the depth cut of a large scene a block's list is short up to
// a later point (24 views in chunks, cut block lists / tile lists: 1M Gaussians
// 833 3.15 / 3.85 in blobs and 4.25 / 4.33 uniform, 2105 2.52 / 2.83 and 4.08 /
// 3.54; 300k Gaussians 631 1.67 / 1.58 and 1.88 / 1.61).
constexpr int64_t kDensePerTile = 560, kDenseCut = 1400;
constexpr int64_t kDenseCutFrom = 1 << 19;  // Gaussians
inline int64_t dense_limit(int64_t n, bool cut) { return cut && n >= kDenseCutFrom ? kDenseCut : kDensePerTile; }
inline int list_shift(int64_t n, int gx, int gy, int64_t dense) {
  return n < (1ll << 28) && gx >= 4 && gy >= 4 && n <= dense * gx * gy ? 1 : 0;
}
__host__ __device__ inline int list_dim(int g, int shift) { return (g + shift) >> shift; }

__device__ __forceinline__ TileList tile_list(const unsigned long long* keys, const uint32_t* list_start,
                                              const uint32_t* zcut, int shift, int gx, int tile) {
  const int tx = tile % gx, ty = tile / gx;
  const int b = (ty >> shift) * list_dim(gx, shift) + (tx >> shift);
  const uint32_t begin = list_start[b];
  TileList l;
  l.keys = keys + begin;
  l.n = (int)(list_start[b + 1] - begin);
  l.bit = shift ? 1u << ((ty & 1) * 2 + (tx & 1)) : 0u;
  l.id_shift = shift ? 4 : 0;
  l.cut = zcut ? zcut[b] : kNoCut;  // a cut goes with shift 1: one per block
  return l;
}
// Records a tile as open (one thread per tile).
__device__ __forceinline__ void record_open(WsHeader* hdr, uint32_t* open_bits, uint32_t* open_list, int gx, int tile) {
  const int bx = (tile % gx) >> 1, by = (tile / gx) >> 1;
  atomicOr(&open_bits[by * open_words(gx) + (bx >> 5)], 1u << (bx & 31));
  open_list[atomicAdd(&hdr->open_tiles, 1u)] = (uint32_t)tile;
}

// Workspace carve-up for one uplift call.
struct UpliftWs {
  WsHeader* hdr;
  SceneP sp;
  uint32_t* cell;           // [n] Morton cell of each Gaussian and its rank in the cell (reorder)
  uint32_t* cells_scratch;  // counting-sort scratch (reorder_scratch_bytes())
  WsHeader* vhdr;           // the view part's own header
  ProjRec* proj;            // [n] by original index
  uint32_t* depth;          // [n] float bits of camera depth, spatial order
  ushort4* rect;            // [n] listed tiles (x_lo, y_lo, x_hi, y_hi), spatial order: the 3DGS
                            //     rectangle cut to the alpha >= 1/255 ellipse's box; empty if culled
  uint32_t* keep;           // [ceil(n / 32)] bit i: Gaussian i (spatial order) is listed in this pass
  uint32_t* tile_count;     // [max_tiles + 1] runs reserved per list (binning)
  uint32_t* tile_glob;      // [max_tiles + 1] big-rectangle items per list (binning)
  uint32_t* run_base;       // [groups x box blocks] offset of each binning CTA's run in a list
  uint32_t* tile_start;     // [max_tiles + 1] first key of each list (TileList)
  uint32_t* tile_fill;      // [max_tiles]
  float* pix_state;         // [max_tiles * 256] per pixel of an open tile: T (< 1e-4: stopped); holds
                            //     the depth cut's histogram while the view is projected
  uint32_t* zcut;           // [blocks] depth cut per block of 2 x 2 tiles (null: the part has no room)
  uint32_t* open_bits;      // [blocks high x open_words(gx)] bit per block with a tile recorded as open
  uint32_t* open_list;      // [max_tiles] the recorded tiles
  unsigned long long* keys; // [dup_capacity] (TileList)
  int64_t dup_capacity;
  int max_tiles;
};

// One view as the projection and binning kernels take it.
struct ViewJob {
  CamArgs cam;
  const float* means;    // the caller's arrays, in the caller's order (depth-cut sample)
  const float* scales;
  const float* opacity;
  const SceneRec* rec;
  const int32_t* orig;
  ProjRec* proj;
  uint32_t* depth;
  ushort4* rect;
  uint32_t* keep;
  uint32_t* tile_count;
  uint32_t* tile_glob;
  uint32_t* run_base;
  uint32_t* tile_start;
  uint32_t* tile_fill;
  unsigned long long* keys;
  long long capacity;
  WsHeader* hdr;
  uint32_t* hist;        // depth cut: [blocks][kCutBins] optical mass; null = no cut for this view
  uint32_t* zcut;
  uint32_t* open_bits;
  uint32_t* open_list;
  float* pix_state;
  int n;
  int group;             // Gaussians per binning CTA (bin_group(n))
  int shift;             // 1: one list per block of 2 x 2 tiles, 0: per tile (TileList)
};
constexpr int kMaxDrainJobs = 64;
template <int N>
struct ViewArgs {
  ViewJob v[N];
};
static_assert(sizeof(ViewArgs<kMaxDrainJobs>) <= 32000, "kernel parameter space");
ViewJob view_job(const scoup_scene& sc, const CamArgs& cam, const UpliftWs& ws, WsHeader* hdr, bool cut);
// Whether views of this size get a depth cut (given room in the view part).
// views: how many views a launch of the view's chunk takes.
bool use_depth_cut(int64_t n, const CamArgs& cam, const UpliftWs& ws, int views);
// Gaussians per binning CTA; larger groups for scenes above kSmallScene, of which
// the depth cut leaves a fraction, and whose kept bits have room beside the runs.
// The kept bits of a smaller scene lie behind the view part's header (kAuxBytes).
constexpr int64_t kSmallScene = 63488;
constexpr size_t kAuxBytes = 8192;
static_assert(sizeof(WsHeader) + (kSmallScene + 31) / 32 * 4 <= kAuxBytes, "kept bits of the largest small scene");
inline int bin_group(int64_t n) { return n <= kSmallScene ? 512 : 1024; }

// Records msg as the calling thread's last error and returns code.
int set_error(int code, const char* msg);

// Arguments of one uplift call (the scoup_uplift parameters).
struct UpliftCall {
  const scoup_scene* scene;
  const scoup_camera* cams;
  int32_t V;
  const int32_t* region_maps;
  const int64_t* map_offsets;
  int32_t R_total;
  const int32_t* code_idx;
  const float* code_val;
  int32_t s, C, K;
  float* accum;
  int32_t accum_mode;
  int32_t* topk_idx;
  float* topk_val;
  int32_t L = 0;                        // > 0: semantic levels in `levels` replace the
  const scoup_level* levels = nullptr;  // single-level region map and code fields above
  // region_maps in HOST memory (single level): each view's map is copied into
  // a device ring of slots of map_stage_cap entries, on a library copy
  // stream, just ahead of the drain of the view's chunk
  bool maps_on_host = false;
  int32_t* map_stage = nullptr;
  int64_t map_stage_cap = 0;
};
constexpr int kMapStageSlots = 4;

// Validates and enqueues one uplift on `st` without synchronising; warp_w is
// the tile kernel's warp pixel-block width (8, 16 or 4).  *hdr_out receives
// the workspace header that holds the call's status and counters.
// view_lanes = 2 runs even and odd views in two pipelines (a second stream)
// when the workspace holds both; lane_views > 1 runs them in chunks of that
// many (the workspace then holds view_lanes x lane_views view parts).
int uplift_call(const UpliftCall& c, void* workspace, size_t ws_bytes, int warp_w, const struct WsHeader** hdr_out,
                cudaStream_t st, int view_lanes = 1, int lane_views = 1);
size_t uplift_required_bytes(int64_t n, const scoup_camera* cams, int32_t V, int32_t s, int32_t K, int32_t R_total,
                             int64_t dup_capacity, int parts = 1);
int uplift_stats(const struct WsHeader* dev_hdr, scoup_stats* stats, cudaStream_t st);
// Parts of an uplift workspace (api.cu): the scene part (header, Morton-ordered
// scene copy, codes filtered to K entries) and one view part (records, depth,
// rectangles, tile counters, state of open tiles); the carve functions lay a part out
// from a 256-byte aligned base and return its size.
size_t uplift_scene_part_bytes(int64_t n, int64_t code_rows_k);
size_t uplift_view_part_bytes(int64_t n, int max_tiles);
size_t carve_scene_part(void* base, int64_t n, int64_t code_rows_k, UpliftWs* w, int32_t** codes_i,
                        float** codes_v);
size_t carve_view_part(void* base, int64_t n, int max_tiles, UpliftWs* w);
CamArgs camera_args(const scoup_camera& c);
int check_scene_views(const scoup_scene* scene, const scoup_camera* cams, int32_t V, int* max_tiles);
void header_stats(const struct WsHeader& h, scoup_stats* stats);

// Launchers (each defined in its own translation unit).
// Self-test: the alpha-threshold exponents that the reorder gives n opacities.
cudaError_t launch_alpha_thresholds(const float* opacity, int64_t n, float* tau, cudaStream_t st);
size_t reorder_scratch_bytes();
// First launch of a call: sets up the scene header, the reorder's cell counts
// and (view: a render, whose view uses the scene's header) the binning counters.
cudaError_t launch_begin(const UpliftWs& ws, bool view, int max_tiles, cudaStream_t st);
cudaError_t launch_reorder(const scoup_scene& sc, const UpliftWs& ws, cudaStream_t st);
// Chunk of nv <= kMaxDrainJobs views (HOST array, copied into the launches'
// parameters): depth cut (for the views that have one), projection, tile lists.
cudaError_t launch_depth_cut(const ViewJob* v, int nv, cudaStream_t st);
cudaError_t launch_project(const ViewJob* v, int nv, cudaStream_t st);
// Second pass, for the tiles recorded as open: keeps the Gaussians that reach
// one of them behind its cut, with their records.
cudaError_t launch_recover(const ViewJob* v, int nv, cudaStream_t st);
// Tile lists of the kept Gaussians; second: only of the open tiles.  The lane's
// drain counter of the pass (ctr, may be null) is cleared on the way.
cudaError_t launch_binning(const ViewJob* v, int nv, bool second, uint32_t* ctr, cudaStream_t st);
// One persistent launch composites every tile of njobs <= kMaxDrainJobs views
// (HOST jobs[njobs], copied into the launch's parameters); second: their open
// tiles, resumed from pix_state.  CTAs take items from *ctr (DEVICE, zero
// before the launch).  All jobs have the same number of levels.
cudaError_t launch_uplift_drain(const TileJob* jobs, int njobs, bool second, uint32_t* ctr, bool compensated,
                                int warp_w, cudaStream_t st);
size_t render_smem_bytes(int C, int K);
bool render_uses_mma(int C, int K);
bool render_mma_supported(int C, int K);
size_t render_mma_smem_bytes(int K);
cudaError_t launch_render_mma(const ViewJob& v, const int32_t* topk_idx,
                              const float* topk_val, int K, int C, void* out, int out_bf16, float* out_T,
                              int32_t* out_last, cudaStream_t st);
cudaError_t launch_render_tiles(const ViewJob& v, const int32_t* topk_idx,
                                const float* topk_val, int K, int C, void* out, int out_bf16, float* out_T,
                                int32_t* out_last, cudaStream_t st);
size_t render_bwd_smem_bytes(int C, int K);
cudaError_t launch_render_bwd(const ViewJob& v, const int32_t* topk_idx,
                              const float* topk_val, int K, int C, const float* dL_dcodes, float* d_val,
                              float* d_opacity, cudaStream_t st);
constexpr int kOutBF16 = 0, kOutF32 = 1, kOutCos = 2, kOutRel = 3;
struct GemmEpi {
  int M, N, K;
  int mode;              // kOutBF16 / kOutF32 / kOutCos / kOutRel
  void* out;             // kOutRel: the relevancy [M, N - n_canon] (ldo = N - n_canon, a multiple of 4)
  int64_t ldo;           // elements
  float* rownorm2;       // kOutBF16: accumulated squared row norms (may be null); kOutCos, kOutRel: input
  const float* colnorm;  // kOutCos, kOutRel: column norms
  int n_canon = 0;       // kOutRel (N <= 32): the first n_canon columns are the canonical phrases
  float alpha = 0.0f;    // kOutRel: softmax temperature of Eq. 9
  int* status;
  int stall_loads = 0;   // self-test only: the producer issues no loads, so the bounded waits run out
  // Fused query (mode kOutBF16): every CTA takes whole row blocks and, after
  // a block's N columns, one more unit of sim_n (16 or 32) columns against
  // the operand Gt (bf16 [sim_n, K]); that unit's epilogue writes, with the
  // row's squared norm summed over the block's rounded features, the cosine
  // (sim_mode kOutCos, colnorm = the sim_n column norms) or the relevancy
  // (kOutRel, with n_canon and alpha) to sim_out [M, sim_ldo] (f32).
  int sim_n = 0;
  int sim_mode = 0;
  void* sim_out = nullptr;
  int64_t sim_ldo = 0;
  int a_f32 = 0;  // A holds FP32 values, rounded to bf16 on the way in (only where gemm_takes_f32())
  int store = 1;  // 0: the kOutBF16 rows are not written (their norms and the fused unit still are)
};
cudaError_t launch_gemm_bf16(const void* A, const void* Bt, const GemmEpi& ep, cudaStream_t st);
// Whether a launch of these sizes (kOutBF16, kOutF32 or a fused query) takes
// FP32 rows of A (ep.a_f32).
bool gemm_takes_f32(int64_t M, int N, int K);
// launch_gemm_bf16 with the fused query unit (ep.sim_n > 0; Gt bf16 [sim_n, K]).
cudaError_t launch_gemm_bf16_query(const void* A, const void* Bt, const void* Gt, const GemmEpi& ep,
                                   cudaStream_t st);
// Before a decode's GEMM: *hdr cleared, Bt [D, C] = bf16 of the transposed
// codebook [C, D], and either (Q > 0) Gt[q][c] = bf16(sum_d text[q][d]
// codebook[c][d]) (FP32 sums) with tnorm[q] = |text_q| (FP32), or (rownorm2)
// rows cleared row norms.
struct GemmPrep {
  WsHeader* hdr;
  const float* codebook;
  void* Bt;
  int C, D;
  const float* text = nullptr;
  int Q = 0;
  void* Gt = nullptr;
  float* tnorm = nullptr;
  float* rownorm2 = nullptr;
  int64_t rows = 0;
};
cudaError_t launch_decode_prep(const GemmPrep& p, cudaStream_t st);
// Before a similarity's GEMM: *hdr cleared, tb = bf16 of text [Q, D], tnorm = the norms of its rows.
cudaError_t launch_text_prep(WsHeader* hdr, const float* text, int Q, int D, void* tb, float* tnorm, cudaStream_t st);
// hdr: cleared by the same launch (null: none).
cudaError_t launch_f32_to_bf16(const float* x, void* y, int64_t n, cudaStream_t st, WsHeader* hdr = nullptr);
cudaError_t launch_row_norm_bf16(const void* X, int64_t R, int D, float* out, int squared, cudaStream_t st);
bool gemm_tma_available();
int gemm_timeout_selftest(void* workspace, size_t ws_bytes, cudaStream_t st);
cudaError_t launch_sgemm(const float* A, const float* B, bool b_transposed, float* out, int64_t M, int N, int K,
                         const float* rownorm2, const float* colnorm2, cudaStream_t st);
cudaError_t launch_row_norm2_f32(const float* X, int64_t R, int D, float* out, cudaStream_t st);
// ld: row stride of accum / comp in floats (C for a plain [n, C] accumulator).
cudaError_t launch_topk(const float* accum, const float* comp, int64_t n, int C, int K, int32_t* idx, float* val,
                        float* entropy, cudaStream_t st, int64_t ld = 0);
size_t entropy_filter_state_bytes();
int entropy_filter_run(const float* H, int64_t n, int64_t keep, int K, int32_t* idx, float* val, uint8_t* mask,
                       void* workspace, cudaStream_t st);
cudaError_t launch_region_targets(const int32_t* ci, const float* cv, int R, int s, const float* codebook, int C,
                                  int D, float* target, int* status, cudaStream_t st);
cudaError_t launch_l2_grad(const void* F, int F_bf16, int64_t P, int D, const int32_t* rmap, int R,
                           const float* target, void* dF, int dF_bf16, double* loss, int* status, cudaStream_t st);
cudaError_t launch_relevancy(const float* sim, int64_t P, int ncols, int n_canon, float alpha, float* R,
                             cudaStream_t st);
cudaError_t launch_code_topk(const int32_t* ci, const float* cv, int64_t R, int s, int K,
                             int32_t* ci_out, float* cv_out, cudaStream_t st);

}  // namespace scoup
