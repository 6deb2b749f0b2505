// loss.cu -- the L2 loss between decoded features and per-pixel region
// targets, and its gradient (the loss of the differentiable sparse render).
//
// The target of pixel p is the decoded code of its region,
// F*(p) = sum_j v_j C[j] over the s entries (j, v_j) of code_{r(p)} (the
// region codes of Eq. 5, decoded with the codebook C of Eq. 8).  The loss is
// L = sum_p |F(p) - F*(p)|^2 over labelled pixels, and dL/dF(p) = 2 (F - F*).
// A first kernel decodes every region's target once (R x D floats, resident
// in L2), a second one streams the pixels: lanes over the features of a pixel
// row (eight at a time where the alignment allows).
#include <cuda_bf16.h>

#include "scoup_internal.cuh"

namespace scoup {
namespace {

// F*_r[d] = sum_j v_j C[j][d] for every region r: a thread per feature, 256
// features to a CTA or, where D is smaller, as many regions as fit; the code's
// entries loaded once into shared memory and eight codebook loads in flight per
// thread (a warp per region with the entries re-read for every feature took 41
// us for 200 regions, 8 entries, D = 512, against 4.6; a CTA per region whatever
// D lost 10 us to it at 3000 regions, 70 entries, D = 16).
constexpr int kCodeChunk = 64;
__global__ void __launch_bounds__(256) region_target_kernel(const int32_t* __restrict__ ci,
                                                            const float* __restrict__ cv, int R, int s,
                                                            const float* __restrict__ codebook, int C, int D,
                                                            float* __restrict__ target, int* __restrict__ status) {
  __shared__ int s_j[8][kCodeChunk];
  __shared__ float s_v[8][kCodeChunk];
  const int per = D < 256 ? (D + 31) & ~31 : 256;  // threads of a region
  const int regions = 256 / per, q = threadIdx.x / per, t = threadIdx.x - q * per;
  const int d = blockIdx.x * 256 + t;
  for (int64_t r0 = (int64_t)blockIdx.y * regions; r0 < R; r0 += (int64_t)gridDim.y * regions) {
    const int64_t r = r0 + q;
    const bool live = q < regions && r < R;
    float acc = 0.0f;
    for (int e0 = 0; e0 < s; e0 += kCodeChunk) {
      const int m = min(kCodeChunk, s - e0);
      __syncthreads();
      if (live)
        for (int e = t; e < m; e += per) {
          const int j = ci[r * s + e0 + e];
          if (j >= C) atomicOr(status, kStatDeviceCheck);
          s_j[q][e] = j < C ? j : -1;
          s_v[q][e] = cv[r * s + e0 + e];
        }
      __syncthreads();
      if (live && d < D)
        for (int e = 0; e < m; e += 8) {
          float x[8];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            x[u] = e + u < m && s_j[q][e + u] >= 0 ? codebook[(int64_t)s_j[q][e + u] * D + d] : 0.0f;
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (e + u < m && s_j[q][e + u] >= 0) acc = fmaf(s_v[q][e + u], x[u], acc);
        }
    }
    if (live && d < D) target[r * D + d] = acc;
  }
}

// Eight consecutive features as one access.
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&x)[8]) {
  const uint4 w = *reinterpret_cast<const uint4*>(p);
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&w);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 f = __bfloat1622float2(h[k]);
    x[2 * k] = f.x;
    x[2 * k + 1] = f.y;
  }
}
__device__ __forceinline__ void load8(const float* p, float (&x)[8]) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
  x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float (&x)[8]) {
  uint4 w;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&w);
#pragma unroll
  for (int k = 0; k < 4; ++k) h[k] = __floats2bfloat162_rn(x[2 * k], x[2 * k + 1]);
  *reinterpret_cast<uint4*>(p) = w;
}
__device__ __forceinline__ void store8(float* p, const float (&x)[8]) {
  reinterpret_cast<float4*>(p)[0] = make_float4(x[0], x[1], x[2], x[3]);
  reinterpret_cast<float4*>(p)[1] = make_float4(x[4], x[5], x[6], x[7]);
}

// Rows of D features, D a multiple of 8, both matrices and the targets 16-byte
// aligned: 1 << lg lanes to a row (32, fewer for short rows), eight features per
// lane and step, so that a 512-feature bf16 row is two 16-byte loads and stores
// per lane.  Bound by HBM: read and write once (480k x 512 bf16, 983 MB: 200 us
// with a feature per lane and step, 174 now).  A whole warp to a row of 64 left
// 24 lanes idle (480k x 64 FP32: 120 us; 89 with a feature per lane; 56 so).
template <typename TIn, typename TOut>
__global__ void __launch_bounds__(256) l2_grad_vec_kernel(const TIn* __restrict__ F, int64_t P, int D, int lg,
                                                          const int32_t* __restrict__ rmap, int R,
                                                          const float* __restrict__ target, TOut* __restrict__ dF,
                                                          double* __restrict__ loss, int* __restrict__ status) {
  const int lane = threadIdx.x & 31, in_row = lane & ((1 << lg) - 1), rows = 32 >> lg;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  double part = 0.0;
  for (int64_t p = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * rows + (lane >> lg); p < P;
       p += warps * rows) {
    int r = rmap[p];
    if (r >= R) {
      if (in_row == 0) atomicOr(status, kStatDeviceCheck);
      r = -1;
    }
    float sq = 0.0f;
#pragma unroll 2
    for (int d = 8 * in_row; d < D; d += 8 << lg) {
      float f[8], t[8];
      load8(F + p * D + d, f);
      // unlabelled pixels (region -1) have no target: no loss, no gradient
      if (r >= 0) load8(target + (int64_t)r * D + d, t);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float diff = r >= 0 ? f[k] - t[k] : 0.0f;
        sq = fmaf(diff, diff, sq);
        f[k] = 2.0f * diff;
      }
      store8(dF + p * D + d, f);
    }
    part += (double)sq;
  }
  for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
  if (lane == 0 && loss && part != 0.0) atomicAdd(loss, part);
}

template <bool kInBF16, bool kOutBF16>
__global__ void __launch_bounds__(256) l2_grad_kernel(const void* __restrict__ F, int64_t P, int D,
                                                      const int32_t* __restrict__ rmap, int R,
                                                      const float* __restrict__ target, void* __restrict__ dF,
                                                      double* __restrict__ loss, int* __restrict__ status) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  double part = 0.0;
  for (int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); p < P; p += warps) {
    int r = rmap[p];
    if (r >= R) {
      if (lane == 0) atomicOr(status, kStatDeviceCheck);
      r = -1;
    }
    float sq = 0.0f;
    for (int d = lane; d < D; d += 32) {
      float f;
      if constexpr (kInBF16) f = __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(F)[p * D + d]);
      else f = reinterpret_cast<const float*>(F)[p * D + d];
      // unlabelled pixels (region -1) have no target: no loss, no gradient
      const float diff = r >= 0 ? f - target[(int64_t)r * D + d] : 0.0f;
      sq = fmaf(diff, diff, sq);
      if constexpr (kOutBF16) reinterpret_cast<__nv_bfloat16*>(dF)[p * D + d] = __float2bfloat16_rn(2.0f * diff);
      else reinterpret_cast<float*>(dF)[p * D + d] = 2.0f * diff;
    }
    part += (double)sq;
  }
  for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
  if (lane == 0 && loss && part != 0.0) atomicAdd(loss, part);
}

int blocks_for_warps(int64_t rows) {
  int64_t b = (rows + 7) / 8;
  if (b > num_sms() * 16) b = num_sms() * 16;
  return (int)(b > 0 ? b : 1);
}

}  // namespace

cudaError_t launch_region_targets(const int32_t* ci, const float* cv, int R, int s, const float* codebook, int C,
                                  int D, float* target, int* status, cudaStream_t st) {
  if (R <= 0) return cudaSuccess;
  const int regions = D < 256 ? 256 / ((D + 31) & ~31) : 1;  // of a CTA, as in the kernel
  const int blocks = (R - 1) / regions + 1;
  region_target_kernel<<<dim3((D + 255) / 256, blocks < 65535 ? blocks : 65535), 256, 0, st>>>(ci, cv, R, s, codebook,
                                                                                             C, D, target, status);
  g_launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_l2_grad(const void* F, int F_bf16, int64_t P, int D, const int32_t* rmap, int R,
                           const float* target, void* dF, int dF_bf16, double* loss, int* status, cudaStream_t st) {
  if (P <= 0) return cudaSuccess;
  const int b = blocks_for_warps(P);
  // The targets lie in the caller's workspace, which may start at any 4-byte
  // boundary.  FP32 rows whose few targets stay in L1 stream faster with a feature
  // per lane (480k rows of FP32 to FP32, us, 16-byte kernel / the other: 1 region
  // D = 136 134 / 101, 256 169 / 135, 512 318 / 258; 4 regions 134 / 112, 170 /
  // 152, 318 / 295; 200 regions 134 / 124, 171 / 171, 327 / 325, and to bf16
  // 250 / 264; D = 64 56 / 89 whatever the regions).
  const bool words = !F_bf16 && R <= 8 && D > 128;
  if (!words && D % 8 == 0 && (((uintptr_t)F | (uintptr_t)dF | (uintptr_t)target) & 15u) == 0) {
    int lg = 0;  // lanes of a row: a power of two, enough for the row or all
    while (lg < 5 && (8 << lg) < D) ++lg;
    const int vb = blocks_for_warps((P - 1) / (32 >> lg) + 1);
    auto run = [&](auto* f, auto* d) {
      l2_grad_vec_kernel<<<vb, 256, 0, st>>>(f, P, D, lg, rmap, R, target, d, loss, status);
    };
    const __nv_bfloat16* fb = (const __nv_bfloat16*)F;
    __nv_bfloat16* db = (__nv_bfloat16*)dF;
    if (F_bf16 && dF_bf16) run(fb, db);
    else if (F_bf16) run(fb, (float*)dF);
    else if (dF_bf16) run((const float*)F, db);
    else run((const float*)F, (float*)dF);
    g_launches += 1;
    return cudaGetLastError();
  }
  if (F_bf16 && dF_bf16) l2_grad_kernel<true, true><<<b, 256, 0, st>>>(F, P, D, rmap, R, target, dF, loss, status);
  else if (F_bf16) l2_grad_kernel<true, false><<<b, 256, 0, st>>>(F, P, D, rmap, R, target, dF, loss, status);
  else if (dF_bf16) l2_grad_kernel<false, true><<<b, 256, 0, st>>>(F, P, D, rmap, R, target, dF, loss, status);
  else l2_grad_kernel<false, false><<<b, 256, 0, st>>>(F, P, D, rmap, R, target, dF, loss, status);
  g_launches += 1;
  return cudaGetLastError();
}

}  // namespace scoup
