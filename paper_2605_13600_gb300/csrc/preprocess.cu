// preprocess.cu -- per-view projection of the Gaussians (paper Sec. 3) and the
// depth cut of the tile lists.
//
// Standard 3DGS projection: camera-space mean, near-plane cull at z <= 0.2,
// EWA 2D covariance T Sigma3 T^T + 0.3 I with T = J Rv and the Jacobian J taken at
// the tangent clamped to 1.3x the half field of view, inverse covariance,
// radius ceil(3 sqrt(lambda_max)) with the 0.1 eigenvalue floor, and the
// 16x16 tile rectangle.
//
// This translation unit is compiled with --fmad=false: every expression is
// evaluated left to right in IEEE binary32 with each operation rounded, in the
// operation order written here, so the discrete outcomes (cull, radius,
// rectangle, depth) are reproducible on any IEEE binary32 machine.
//
// Every kernel here takes a chunk of views (blockIdx.y), so that a chunk's
// launches fill the chip whatever the size of one view.
//
// The depth cut (scoup_internal.cuh) is estimated before the projection: the
// optical mass of a sample of the Gaussians (a fixed stride in the caller's
// order, so that it does not change from run to run; integer sums) is
// histogrammed by depth for every block of 2 x 2 tiles, and the block's cut
// is the depth at which its mean optical depth reaches kCutOptical.
#include <math.h>

#include "scoup_internal.cuh"

namespace scoup {
namespace {

__device__ __forceinline__ int tile_clamp(float v, int g) {
  if (!(v > 0.0f)) return 0;
  if (v > (float)g) return g;
  return (int)v;
}

struct Projected {
  ProjRec rec;
  ushort4 listed;  // tiles of the rectangle that meet the alpha >= 1/255 ellipse's box
  int area;        // tiles of the 3DGS rectangle
  float z;
};

// Projects one Gaussian; returns whether it survives culling.  Every operation
// is rounded on its own, in this order; Sigma3 comes with the record (reorder.cu).
__device__ __forceinline__ bool project_gaussian(const SceneRec& g, const CamArgs& cam, Projected& out) {
  const float m0 = g.mean_op.x, m1 = g.mean_op.y, m2 = g.mean_op.z;
  const float tau_i = g.cov_b.z;
  const float* W = cam.vm;
  float t0 = W[0] * m0 + W[1] * m1 + W[2] * m2 + W[3];
  float t1 = W[4] * m0 + W[5] * m1 + W[6] * m2 + W[7];
  float t2 = W[8] * m0 + W[9] * m1 + W[10] * m2 + W[11];
  out.z = t2;
  out.listed = make_ushort4(0, 0, 0, 0);
  if (!(t2 > 0.2f)) return false;
  const float S00 = g.cov_a.x, S01 = g.cov_a.y, S02 = g.cov_a.z, S11 = g.cov_a.w, S12 = g.cov_b.x, S22 = g.cov_b.y;
  // S10 = S01, S20 = S02, S21 = S12 (each is the same rounded expression)

  float limx = 1.3f * (0.5f * (float)cam.width / cam.fx);
  float limy = 1.3f * (0.5f * (float)cam.height / cam.fy);
  float txz = t0 / t2, tyz = t1 / t2;
  float txc = fminf(limx, fmaxf(-limx, txz)) * t2;
  float tyc = fminf(limy, fmaxf(-limy, tyz)) * t2;
  float tz2 = t2 * t2;
  float j00 = cam.fx / t2;
  float j02 = -(cam.fx * txc) / tz2;
  float j11 = cam.fy / t2;
  float j12 = -(cam.fy * tyc) / tz2;
  float T00 = j00 * W[0] + j02 * W[8];
  float T01 = j00 * W[1] + j02 * W[9];
  float T02 = j00 * W[2] + j02 * W[10];
  float T10 = j11 * W[4] + j12 * W[8];
  float T11 = j11 * W[5] + j12 * W[9];
  float T12 = j11 * W[6] + j12 * W[10];
  float U00 = T00 * S00 + T01 * S01 + T02 * S02;
  float U01 = T00 * S01 + T01 * S11 + T02 * S12;
  float U02 = T00 * S02 + T01 * S12 + T02 * S22;
  float U10 = T10 * S00 + T11 * S01 + T12 * S02;
  float U11 = T10 * S01 + T11 * S11 + T12 * S12;
  float U12 = T10 * S02 + T11 * S12 + T12 * S22;
  float ca2 = U00 * T00 + U01 * T01 + U02 * T02 + 0.3f;
  float cb2 = U00 * T10 + U01 * T11 + U02 * T12;
  float cc2 = U10 * T10 + U11 * T11 + U12 * T12 + 0.3f;
  float det = ca2 * cc2 - cb2 * cb2;
  if (!(det > 0.0f)) return false;
  float idet = 1.0f / det;
  float con_a = cc2 * idet, con_b = -cb2 * idet, con_c = ca2 * idet;
  float mid = 0.5f * (ca2 + cc2);
  float lam = mid + sqrtf(fmaxf(0.1f, mid * mid - det));
  float r = ceilf(3.0f * sqrtf(lam));
  float mx = cam.fx * txz + cam.cx - 0.5f;
  float my = cam.fy * tyz + cam.cy - 0.5f;
  int xlo = tile_clamp(floorf((mx - r) / 16.0f), cam.gx);
  int xhi = tile_clamp(floorf((mx + r + 15.0f) / 16.0f), cam.gx);
  int ylo = tile_clamp(floorf((my - r) / 16.0f), cam.gy);
  int yhi = tile_clamp(floorf((my + r + 15.0f) / 16.0f), cam.gy);
  if (!(xhi > xlo && yhi > ylo)) return false;
  out.rec.a = make_float4(mx, my, -0.5f * con_a, -con_b);
  out.rec.b = make_float4(-0.5f * con_c, g.mean_op.w, tau_i, 0.0f);
  out.area = (xhi - xlo) * (yhi - ylo);
  // Binning lists only the tiles of the rectangle that also meet the
  // bounding box of the alpha >= 1/255 ellipse {d : power(d) >= tau}:
  // half-widths sqrt(-2 tau (A^-1)_xx), sqrt(-2 tau (A^-1)_yy) with
  // A = [[-2qa, -qb], [-qb, -2qc]], widened by 0.1% + 0.5 px so no
  // pixel centre that passes the alpha test is left out.
  if (tau_i < 0.0f) {
    const float A00 = con_a, A11 = con_c, A01 = con_b;  // = -2qa, -2qc, -qb
    const float detA = A00 * A11 - A01 * A01;
    const float ex = sqrtf(-2.0f * tau_i * A11 / detA) * 1.001f + 0.5f;
    const float ey = sqrtf(-2.0f * tau_i * A00 / detA) * 1.001f + 0.5f;
    const int lx0 = max(xlo, tile_clamp(floorf((mx - ex) / 16.0f), cam.gx));
    const int lx1 = min(xhi, tile_clamp(floorf((mx + ex) / 16.0f) + 1.0f, cam.gx));
    const int ly0 = max(ylo, tile_clamp(floorf((my - ey) / 16.0f), cam.gy));
    const int ly1 = min(yhi, tile_clamp(floorf((my + ey) / 16.0f) + 1.0f, cam.gy));
    if (lx1 > lx0 && ly1 > ly0)
      out.listed = make_ushort4((unsigned short)lx0, (unsigned short)ly0, (unsigned short)lx1, (unsigned short)ly1);
  }
  return true;
}

__device__ __forceinline__ void store_record(const ViewJob& v, const SceneRec& g, const Projected& p) {
  ProjRec r = p.rec;
  r.b.w = log2f(g.mean_op.w);
  v.proj[__float_as_int(g.cov_b.w)] = r;
}

// Whether depth d lies in front of the cut of some block the rectangle meets
// (rectangles over more than kCutRect blocks are kept as they are).
constexpr int kCutRect = 64;
__device__ __forceinline__ bool in_front(const ushort4& r, uint32_t d, const uint32_t* __restrict__ zcut, int bw) {
  const int x0 = r.x >> 1, x1 = (r.z - 1) >> 1, y0 = r.y >> 1, y1 = (r.w - 1) >> 1;
  if ((x1 - x0 + 1) * (y1 - y0 + 1) > kCutRect) return true;
  for (int y = y0; y <= y1; ++y)
    for (int x = x0; x <= x1; ++x)
      if (d <= __ldg(zcut + y * bw + x)) return true;
  return false;
}

// Thread i projects Gaussian i of the spatially ordered copy; the record is
// stored at its original index (only if the Gaussian is kept), depth,
// rectangle and the kept bit in spatial order.
template <int N>
__global__ void __launch_bounds__(256) project_kernel(const __grid_constant__ ViewArgs<N> args) {
  const ViewJob& v = args.v[N == 1 ? 0 : blockIdx.y];
  const CamArgs& cam = v.cam;
  const int n = v.n;
  const bool cut = v.hist != nullptr;
  const int bw = cut_blocks(cam.gx);
  unsigned long long my_dups = 0, my_listed = 0;
  uint32_t my_vis = 0, my_dmin = 0xffffffffu, my_dmax = 0u;
  // whole warps take part in every round (the kept bits of 32 Gaussians are one word)
  for (int64_t i0 = blockIdx.x * 256 + (threadIdx.x & ~31); i0 < n; i0 += gridDim.x * 256) {
    const int64_t i = i0 + (threadIdx.x & 31);
    bool keep = false;
    if (i < n) {
      const SceneRec g = v.rec[i];
      Projected p;
      const bool vis = project_gaussian(g, cam, p);
      const uint32_t d = __float_as_uint(p.z);
      const bool listed = p.listed.z > p.listed.x;
      if (vis) {
        keep = listed && (!cut || in_front(p.listed, d, v.zcut, bw));
        my_vis += 1u;
        my_dups += (unsigned long long)p.area;
        if (listed) my_listed += (unsigned)((p.listed.z - p.listed.x) * (p.listed.w - p.listed.y));
        my_dmin = min(my_dmin, d);
        my_dmax = max(my_dmax, d);
        if (keep) store_record(v, g, p);
      }
      v.depth[i] = d;
      v.rect[i] = p.listed;
    }
    const unsigned word = __ballot_sync(0xffffffffu, keep);
    if ((threadIdx.x & 31) == 0) v.keep[i0 >> 5] = word;
  }
  // block reduction of the counters
  for (int off = 16; off > 0; off >>= 1) {
    my_dups += __shfl_down_sync(0xffffffffu, my_dups, off);
    my_listed += __shfl_down_sync(0xffffffffu, my_listed, off);
  }
  my_vis = __reduce_add_sync(0xffffffffu, my_vis);
  my_dmin = __reduce_min_sync(0xffffffffu, my_dmin);
  my_dmax = __reduce_max_sync(0xffffffffu, my_dmax);
  __shared__ unsigned long long s_dups[8], s_listed[8];
  __shared__ uint32_t s_vis[8], s_dmin[8], s_dmax[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    s_vis[warp] = my_vis; s_dups[warp] = my_dups; s_listed[warp] = my_listed;
    s_dmin[warp] = my_dmin; s_dmax[warp] = my_dmax;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long a = 0, b = 0, c = 0;
    uint32_t lo = 0xffffffffu, hi = 0u;
    for (int k = 0; k < 8; ++k) {
      a += s_vis[k]; b += s_dups[k]; c += s_listed[k]; lo = min(lo, s_dmin[k]); hi = max(hi, s_dmax[k]);
    }
    if (a) {
      atomicAdd(&v.hdr->visible, a);
      atomicAdd(&v.hdr->duplicates, b);
      atomicAdd(&v.hdr->listed, c);
      atomicMin(&v.hdr->drange[0], lo);
      atomicMax(&v.hdr->drange[1], hi);
    }
  }
}

// ---- depth cut ------------------------------------------------------------

// A pixel stops at optical depth 9.2; a block's pixels vary about its mean, and
// a tile with one open pixel costs a second pass, so the cut lies at a multiple
// of that.  1M blob Gaussians, 988x731 (4249 listed per tile without a cut):
// 739 listed per tile and 0.9% of the tiles open at 24, 826 and 0.1% at 28, 912
// and none at 32, 1066 at 40 (1920x1080: 3.5, 1.8, 0.8, 0.1% open).  With
// half the sample (1 << 17, of 1M) 5.3% were open at 24 and 1.4% at 32.  Few
// open tiles already cost a chunk its second pass (the 8 views of a chunk share
// it): 200 views 40.3 ms at 32, 39.0 at 42, 39.6 at 56.
constexpr int kCutSample = 1 << 18;      // Gaussians sampled per view, about
constexpr float kMassUnit = 4.0f;        // histogram units per pixel of optical depth 1
constexpr float kCutOptical = 42.0f;     // mean optical depth of a block at its cut
constexpr float kBlockPixels = 4.0f * kTilePixels;

template <int N>
__global__ void __launch_bounds__(256) cut_clear_kernel(const __grid_constant__ ViewArgs<N> args) {
  const ViewJob& v = args.v[N == 1 ? 0 : blockIdx.y];
  if (!v.hist) return;
  const int nq = cut_blocks(v.cam.gx) * cut_blocks(v.cam.gy) * (kCutBins / 4);
  for (int t = blockIdx.x * 256 + threadIdx.x; t < nq; t += gridDim.x * 256)
    reinterpret_cast<uint4*>(v.hist)[t] = make_uint4(0u, 0u, 0u, 0u);
}

// Sampled Gaussian -> its block's histogram at its depth.  Mass: the integral
// of -log(1 - alpha) over the image, 2 pi sigma^2 Li2(o) with Li2(o) about
// o + 0.645 o^3, for the footprint of a sphere of the Gaussian's mean
// projected area; at most what covers the block.
template <int N>
__global__ void __launch_bounds__(256) cut_mass_kernel(const __grid_constant__ ViewArgs<N> args) {
  const ViewJob& v = args.v[N == 1 ? 0 : blockIdx.y];
  if (!v.hist) return;
  const CamArgs& cam = v.cam;
  const int stride = max(1, v.n / kCutSample);
  const int bw = cut_blocks(cam.gx);
  const float* W = cam.vm;
  for (int64_t k = blockIdx.x * 256 + threadIdx.x; k * stride < v.n; k += gridDim.x * 256) {
    const int64_t i = k * stride;
    const float m0 = v.means[3 * i], m1 = v.means[3 * i + 1], m2 = v.means[3 * i + 2];
    const float s0 = v.scales[3 * i], s1 = v.scales[3 * i + 1], s2 = v.scales[3 * i + 2];
    const float o = fminf(v.opacity[i], 1.0f);
    const float z = W[8] * m0 + W[9] * m1 + W[10] * m2 + W[11];
    if (!(z > 0.2f) || !(o > 0.0f)) continue;
    const float inv = __fdividef(1.0f, z);
    const float px = (W[0] * m0 + W[1] * m1 + W[2] * m2 + W[3]) * inv * cam.fx + cam.cx;
    const float py = (W[4] * m0 + W[5] * m1 + W[6] * m2 + W[7]) * inv * cam.fy + cam.cy;
    if (!(px >= 0.0f && py >= 0.0f && px < (float)cam.width && py < (float)cam.height)) continue;
    const float s2m = (s0 * s1 + s1 * s2 + s0 * s2) * (1.0f / 3.0f);
    const float sig2 = cam.fx * cam.fy * inv * inv * s2m + 0.3f;
    const float mass = fminf(6.2831853f * sig2 * (o + 0.645f * o * o * o), 4.6f * kBlockPixels);
    const int block = ((int)py >> 5) * bw + ((int)px >> 5);
    const uint32_t bin = min((__float_as_uint(z) - kCutBase) >> kCutShift, (uint32_t)(kCutBins - 1));
    atomicAdd(&v.hist[(size_t)block * kCutBins + bin], (uint32_t)(mass * (kMassUnit * (float)stride) + 0.5f));
  }
}

// One warp per block: the upper end of the bin in which the mass in front
// reaches kCutOptical over the block.
template <int N>
__global__ void __launch_bounds__(256) cut_depth_kernel(const __grid_constant__ ViewArgs<N> args) {
  const ViewJob& v = args.v[N == 1 ? 0 : blockIdx.y];
  if (!v.hist) return;
  constexpr int kPer = kCutBins / 32;
  const int nb = cut_blocks(v.cam.gx) * cut_blocks(v.cam.gy), lane = threadIdx.x & 31;
  const unsigned long long need = (unsigned long long)(kCutOptical * kBlockPixels * kMassUnit);
  for (int b = blockIdx.x * 8 + (threadIdx.x >> 5); b < nb; b += gridDim.x * 8) {
    unsigned long long c[kPer], sum = 0;
#pragma unroll
    for (int q = 0; q < kPer / 4; ++q) {
      const uint4 x = reinterpret_cast<const uint4*>(v.hist + (size_t)b * kCutBins + lane * kPer)[q];
      c[4 * q] = x.x; c[4 * q + 1] = x.y; c[4 * q + 2] = x.z; c[4 * q + 3] = x.w;
      sum += c[4 * q] + c[4 * q + 1] + c[4 * q + 2] + c[4 * q + 3];
    }
    unsigned long long incl = sum;
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += y;
    }
    uint32_t cut = kNoCut;
    unsigned long long run = incl - sum;
    if (run < need && incl >= need) {
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        run += c[q];
        if (run >= need) {
          const uint32_t bin = (uint32_t)(lane * kPer + q);
          if (bin < (uint32_t)(kCutBins - 1)) cut = kCutBase + ((bin + 1u) << kCutShift) - 1u;
          break;
        }
      }
    }
    cut = __reduce_min_sync(0xffffffffu, cut);
    if (lane == 0) v.zcut[b] = cut;
  }
}

// Second pass: the kept bit of every Gaussian that reaches a block with a tile
// recorded as open, behind its cut, and its record, which the first pass stored
// only for the Gaussians it kept.  A CTA tests 1024
// Gaussians (four per thread, their loads in flight together), lists the few
// that pass and projects the list, so that the projection runs in full warps.
constexpr int kRecover = 1024;
template <int N>
__global__ void __launch_bounds__(256) recover_kernel(const __grid_constant__ ViewArgs<N> args) {
  const ViewJob& v = args.v[N == 1 ? 0 : blockIdx.y];
  if (v.hdr->open_tiles == 0u) return;
  const int bw = cut_blocks(v.cam.gx), ow = open_words(v.cam.gx);
  __shared__ int s_list[kRecover];
  __shared__ int s_cnt;
  const int lane = threadIdx.x & 31;
  for (int64_t base = (int64_t)blockIdx.x * kRecover; base < v.n; base += gridDim.x * kRecover) {
    if (threadIdx.x == 0) s_cnt = 0;
    ushort4 r[kRecover / 256];
    uint32_t d[kRecover / 256];
#pragma unroll
    for (int q = 0; q < kRecover / 256; ++q) {
      const int64_t i = base + q * 256 + threadIdx.x;
      r[q] = i < v.n ? v.rect[i] : make_ushort4(0, 0, 0, 0);
      d[q] = i < v.n ? v.depth[i] : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kRecover / 256; ++q) {
      const int64_t i = base + q * 256 + threadIdx.x;
      bool keep = false;
      if (r[q].z > r[q].x) {
        const int x0 = r[q].x >> 1, x1 = (r[q].z + 1) >> 1, y1 = (r[q].w + 1) >> 1;
        for (int by = r[q].y >> 1; by < y1 && !keep; ++by)
          for (int w = x0 >> 5; w <= (x1 - 1) >> 5 && !keep; ++w) {
            const int lo = max(x0 - 32 * w, 0), hi = min(x1 - 32 * w, 32);
            uint32_t m = __ldg(v.open_bits + by * ow + w) & (0xffffffffu << lo) & (0xffffffffu >> (32 - hi));
            for (; m != 0u && !keep; m &= m - 1u)
              keep = d[q] > __ldg(v.zcut + by * bw + 32 * w + __ffs(m) - 1);
          }
      }
      const unsigned word = __ballot_sync(0xffffffffu, keep);
      if (lane == 0 && i < v.n) v.keep[i >> 5] = word;
      int at = 0;
      if (lane == 0 && word) at = atomicAdd(&s_cnt, __popc(word));
      at = __shfl_sync(0xffffffffu, at, 0);
      if (keep) s_list[at + __popc(word & ((1u << lane) - 1u))] = (int)i;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < s_cnt; k += 256) {
      const int i = s_list[k];
      Projected p;
      const SceneRec g = v.rec[i];
      if (project_gaussian(g, v.cam, p)) store_record(v, g, p);
    }
    __syncthreads();
  }
}

// Calls f(std::integral_constant<N>) with the launch-parameter capacity for nv views.
template <typename F>
cudaError_t with_views(const ViewJob* v, int nv, F&& f) {
  if (nv <= 0) return cudaSuccess;
  if (nv > kMaxDrainJobs) return cudaErrorInvalidValue;
  if (nv == 1) return f(*reinterpret_cast<const ViewArgs<1>*>(v));
  if (nv <= 8) {
    ViewArgs<8> a;
    for (int k = 0; k < 8; ++k) a.v[k] = v[k < nv ? k : 0];
    return f(a);
  }
  ViewArgs<kMaxDrainJobs> a;
  for (int k = 0; k < kMaxDrainJobs; ++k) a.v[k] = v[k < nv ? k : 0];
  return f(a);
}

int largest_n(const ViewJob* v, int nv) {
  int n = 1;
  for (int k = 0; k < nv; ++k) n = v[k].n > n ? v[k].n : n;
  return n;
}

// CTAs per view: enough for the view's `items` CTAs' worth of work, at most
// per_sm CTAs per SM over all the views.
int view_grid(int items, int nv, int per_sm) {
  const int most = (num_sms() * per_sm + nv - 1) / nv;
  return items < 1 ? 1 : (items < most ? items : most);
}

}  // namespace

// Measured per view in chunks of 8 (1M Gaussians, 988x731): cut 5 us, count 3
// and fill 9 us, against 17 and 63 us for the whole tile lists, one view at a
// time; 200-view uplift 51.8 -> 42.0 ms.
cudaError_t launch_depth_cut(const ViewJob* v, int nv, cudaStream_t st) {
  int blocks = 0;
  for (int k = 0; k < nv; ++k)
    if (v[k].hist) {
      const int b = cut_blocks(v[k].cam.gx) * cut_blocks(v[k].cam.gy);
      blocks = b > blocks ? b : blocks;
    }
  if (blocks == 0) return cudaSuccess;
  return with_views(v, nv, [&](const auto& a) {
    constexpr int N = sizeof(a.v) / sizeof(a.v[0]);
    const int n = largest_n(v, nv), sample = n < 2 * kCutSample ? n : 2 * kCutSample;
    cut_clear_kernel<N><<<dim3(view_grid(blocks / 2 + 1, nv, 8), nv), 256, 0, st>>>(a);
    cut_mass_kernel<N><<<dim3(view_grid((sample + 255) / 256, nv, 8), nv), 256, 0, st>>>(a);
    cut_depth_kernel<N><<<dim3(view_grid((blocks + 7) / 8, nv, 8), nv), 256, 0, st>>>(a);
    g_launches += 3;
    return cudaGetLastError();
  });
}

cudaError_t launch_project(const ViewJob* v, int nv, cudaStream_t st) {
  return with_views(v, nv, [&](const auto& a) {
    constexpr int N = sizeof(a.v) / sizeof(a.v[0]);
    project_kernel<N><<<dim3(view_grid((largest_n(v, nv) + 255) / 256, nv, 8), nv), 256, 0, st>>>(a);
    g_launches += 1;
    return cudaGetLastError();
  });
}

cudaError_t launch_recover(const ViewJob* v, int nv, cudaStream_t st) {
  return with_views(v, nv, [&](const auto& a) {
    constexpr int N = sizeof(a.v) / sizeof(a.v[0]);
    const dim3 grid(view_grid((largest_n(v, nv) + kRecover - 1) / kRecover, nv, 8), nv);
    recover_kernel<N><<<grid, 256, 0, st>>>(a);
    g_launches += 1;
    return cudaGetLastError();
  });
}

}  // namespace scoup
