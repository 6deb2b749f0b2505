// topk.cu -- Top-K consensus filter + L1 normalisation (paper Eq. 6, Alg. 1)
// and the per-code Top-K of Algorithm 1 for codes with more than K entries.
//
// One warp per accumulator row.  Lane l holds entries l, l+32, l+64, ... in
// registers; the row is read once from HBM (coalesced).  The pass is bound by
// instruction issue, not by HBM (86% of the issue rate at 27% of the bandwidth
// before the 32-row spans).
//  - 3 <= K <= 16: the K-th largest of the 32 lane maxima
//    (K warp max-reductions of one word) is a lower bound of the row's K-th
//    entry, so only entries at or above it can be kept, about K + 2 of them;
//    they are compacted in atom order and each finds its place by counting the
//    candidates in front of it.  (K rounds of a full arg-max, each a scan of
//    the lane's entries and two reductions, took 740 us on a 30%-dense 1M x 256
//    accumulator with the entropy, K = 8; 390 us so.)
//  - K <= 2, K > 16 (topk_rounds_kernel), and a row with more than 32 candidates
//    (many equal entries): each of the K rounds picks the largest remaining
//    positive entry, ties to the lower atom index.  One or two rounds are less
//    work than the bound and the compaction (us, rounds / candidates: K = 1,
//    400k x 96 74 / 109, 400k x 256 103 / 122, 60k x 1024 57 / 66; K = 2, 400k x
//    96 83 / 99, 60k x 384 28 / 33).  Above 16 a warp per row keeps twice the
//    warps in flight that spans of rows do (60k x 256, K = 24: 128 / 151).
// With a compensation array (the compensated uplift) each entry is the FP32
// sum of the running sum and its compensation.  Optionally the same pass
// writes the entropy of the row's coefficient distribution,
// H = -sum p log p with p = w / sum w over the positive entries (0 for an
// empty row), computed as log S - (sum w log w) / S; the per-entry logarithms
// use the fast intrinsic (absolute error about 1e-6, so H is off by at most
// that much: far inside the FP32 tolerance of the entropy).
#include "scoup_internal.cuh"

namespace scoup {
namespace {

constexpr unsigned kFull = 0xffffffffu;

constexpr int kFastK = 16;  // largest K of the candidate form

// sum w and sum w log w over the positive entries of the row.
template <int VPL>
__device__ __forceinline__ void entropy_sums(const float (&v)[VPL], float& S, float& WL) {
  S = 0.0f;
  WL = 0.0f;
#pragma unroll
  for (int k = 0; k < VPL; ++k)
    if (v[k] > 0.0f) {
      S += v[k];
      WL = fmaf(v[k], __logf(v[k]), WL);
    }
  for (int off = 16; off > 0; off >>= 1) {
    S += __shfl_xor_sync(kFull, S, off);
    WL += __shfl_xor_sync(kFull, WL, off);
  }
}

// K rounds of arg-max over the row's entries v (in registers).
template <int VPL>
__device__ __forceinline__ int topk_rounds(const float (&v)[VPL], int K, int32_t* __restrict__ orow_i,
                                           float* __restrict__ orow_v, float& sum) {
  const int lane = threadIdx.x & 31;
  unsigned taken = 0u;
  int r = 0;
  for (; r < K; ++r) {
    float bv = 0.0f;
    int bj = 0x7fffffff;
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      if (!((taken >> k) & 1u) && v[k] > bv) { bv = v[k]; bj = lane + 32 * k; }
    }
    const unsigned mb = __reduce_max_sync(kFull, __float_as_uint(bv));
    if (mb == 0u) break;  // no positive entry left
    bj = __reduce_min_sync(kFull, __float_as_uint(bv) == mb ? bj : 0x7fffffff);
    bv = __uint_as_float(mb);
    if ((bj & 31) == lane) taken |= 1u << (bj >> 5);
    if (lane == 0) { orow_i[r] = bj; orow_v[r] = bv; }
    sum += bv;
  }
  return r;
}

// One warp per row, K rounds.
template <int VPL>
__global__ void __launch_bounds__(256) topk_rounds_kernel(const float* __restrict__ acc, const float* __restrict__ comp,
                                                          int64_t n, int C, int64_t ld, int K,
                                                          int32_t* __restrict__ idx, float* __restrict__ val,
                                                          float* __restrict__ entropy) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * 8;
  for (int64_t row = blockIdx.x * (int64_t)8 + (threadIdx.x >> 5); row < n; row += warps) {
    const float* a = acc + row * ld;
    float v[VPL];
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const int j = lane + 32 * k;
      v[k] = j < C ? (comp ? __fadd_rn(a[j], comp[row * ld + j]) : a[j]) : 0.0f;
    }
    if (entropy) {
      float S, WL;
      entropy_sums<VPL>(v, S, WL);
      if (lane == 0) entropy[row] = S > 0.0f ? fmaxf(0.0f, logf(S) - WL / S) : 0.0f;
    }
    int32_t* orow_i = idx + row * K;
    float* orow_v = val + row * K;
    float sum = 0.0f;
    const int r = topk_rounds<VPL>(v, K, orow_i, orow_v, sum);
    __syncwarp();
    for (int k = lane; k < K; k += 32) {
      if (k < r) {
        orow_v[k] = orow_v[k] / sum;
      } else {
        orow_i[k] = -1;
        orow_v[k] = 0.0f;
      }
    }
    __syncwarp();
  }
}

// A warp takes `span` (<= 32) consecutive rows at a time; the lane of a row in
// its span keeps the row's entropy sums, so that the logarithm and quotient
// that finish an entropy run once per span, in every lane, and not once per
// row in one.  KT: K when it is known at compile time (unrolled), else 0.
// kPlain: rows of exactly 32 VPL entries without compensation terms.
template <int VPL, bool kEntropy, int KT, bool kPlain>
__global__ void __launch_bounds__(256) topk_kernel(const float* __restrict__ acc, const float* __restrict__ comp,
                                                   int64_t n, int C, int64_t ld, int Kr, int span,
                                                   int32_t* __restrict__ idx, float* __restrict__ val,
                                                   float* __restrict__ entropy) {
  const int K = KT ? KT : Kr;
  constexpr int kCand = 32 * VPL;
  __shared__ alignas(16) float s_cv[8][kCand];  // per warp: candidates in atom order
  __shared__ uint16_t s_cj[8][kCand];
  __shared__ alignas(16) float s_top[8][kFastK];  // the kept values in order
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t step = (int64_t)gridDim.x * 8 * span;
  for (int64_t base = (blockIdx.x * (int64_t)8 + warp) * span; base < n; base += step) {
    float keep_s = 0.0f, keep_wl = 0.0f;
    const int rows = (int)min((int64_t)span, n - base);
    const float* a = acc + base * ld + lane;
    const float* ac = kPlain || !comp ? nullptr : comp + base * ld + lane;
    int32_t* orow_i = idx + base * K;
    float* orow_v = val + base * K;
    for (int it = 0; it < rows; ++it, a += ld, orow_i += K, orow_v += K) {
      float v[VPL];
#pragma unroll
      for (int k = 0; k < VPL; ++k) {
        if constexpr (kPlain) v[k] = a[32 * k];
        else v[k] = lane + 32 * k < C ? (ac ? __fadd_rn(a[32 * k], ac[it * ld + 32 * k]) : a[32 * k]) : 0.0f;
      }
      if constexpr (kEntropy) {
        float S, WL;
        entropy_sums<VPL>(v, S, WL);
        if (lane == it) { keep_s = S; keep_wl = WL; }
      }
      float sum = 0.0f;
      int r = 0;
      bool fast = false;
      {
        float m = 0.0f;
#pragma unroll
        for (int k = 0; k < VPL; ++k) m = fmaxf(m, v[k]);
        unsigned t = 0u;
#pragma unroll
        for (int q = 0; q < K; ++q) {
          t = __reduce_max_sync(kFull, __float_as_uint(m));  // 0 once fewer than K lanes hold a positive entry
          if (__float_as_uint(m) == t) m = 0.0f;
          if (!KT && t == 0u) break;
        }
        const float bound = t ? __uint_as_float(t) : 1e-45f;
        int cnt = 0;
#pragma unroll
        for (int k = 0; k < VPL; ++k) {
          const bool c = v[k] >= bound;
          const unsigned b = __ballot_sync(kFull, c);
          if (c) {
            const int at = cnt + __popc(b & ((1u << lane) - 1u));
            s_cv[warp][at] = v[k];
            s_cj[warp][at] = (uint16_t)(lane + 32 * k);
          }
          cnt += __popc(b);
        }
        if (cnt <= 32) {
          fast = true;
          r = min(cnt, K);
          if (lane < 4 && cnt + lane < kCand) s_cv[warp][cnt + lane] = 0.0f;  // read four at a time below
          __syncwarp();
          const float mine = lane < cnt ? s_cv[warp][lane] : 0.0f;
          int rank = 0;
          for (int q = 0; q < cnt; q += 4) {
            const float4 o = *reinterpret_cast<const float4*>(&s_cv[warp][q]);
            rank += (o.x > mine || (o.x == mine && q < lane)) ? 1 : 0;
            rank += (o.y > mine || (o.y == mine && q + 1 < lane)) ? 1 : 0;
            rank += (o.z > mine || (o.z == mine && q + 2 < lane)) ? 1 : 0;
            rank += (o.w > mine || (o.w == mine && q + 3 < lane)) ? 1 : 0;
          }
          if (lane < cnt && rank < K) {
            s_top[warp][rank] = mine;
            orow_i[rank] = s_cj[warp][lane];
          }
          __syncwarp();
          if (KT) {
            float top[KT ? KT : 1];
#pragma unroll
            for (int q = 0; q < KT; ++q) top[q] = s_top[warp][q];
#pragma unroll
            for (int q = 0; q < KT; ++q) sum += q < r ? top[q] : 0.0f;
          } else {
            for (int q = 0; q < r; ++q) sum += s_top[warp][q];
          }
          if (lane < r) orow_v[lane] = s_top[warp][lane] / sum;
        }
      }
      if (!fast) {
        r = topk_rounds<VPL>(v, K, orow_i, orow_v, sum);
        __syncwarp();
        for (int k = lane; k < r; k += 32) orow_v[k] = orow_v[k] / sum;
      }
      for (int k = r + lane; k < K; k += 32) {
        orow_i[k] = -1;
        orow_v[k] = 0.0f;
      }
      __syncwarp();
    }
    if (kEntropy && lane < rows)
      entropy[base + lane] = keep_s > 0.0f ? fmaxf(0.0f, logf(keep_s) - keep_wl / keep_s) : 0.0f;
  }
}

// Per code row: keep the K largest entries (ties to the lower atom id), pad -1.
__global__ void code_topk_kernel(const int32_t* __restrict__ ci, const float* __restrict__ cv,
                                 int64_t R, int s, int K, int32_t* __restrict__ co,
                                 float* __restrict__ cvo) {
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < R;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int32_t* a = ci + r * s;
    const float* b = cv + r * s;
    int w = 0;
    for (int p = 0; p < s; ++p) {
      if (a[p] < 0) continue;
      int better_cnt = 0;
      for (int q = 0; q < s; ++q) {
        if (q == p || a[q] < 0) continue;
        if (b[q] > b[p] || (b[q] == b[p] && a[q] < a[p])) ++better_cnt;
      }
      if (better_cnt < K) { co[r * K + w] = a[p]; cvo[r * K + w] = b[p]; ++w; }
    }
    for (; w < K; ++w) { co[r * K + w] = -1; cvo[r * K + w] = 0.0f; }
  }
}

template <int VPL, bool kEntropy>
cudaError_t launch_vpl(const float* acc, const float* comp, int64_t n, int C, int64_t ld, int K, int32_t* idx,
                       float* val, float* entropy, cudaStream_t st) {
  if (K <= 2 || K > kFastK) {
    const int64_t blocks = (n + 7) / 8 < num_sms() * 16 ? (n + 7) / 8 : num_sms() * 16;
    topk_rounds_kernel<VPL><<<(int)blocks, 256, 0, st>>>(acc, comp, n, C, ld, K, idx, val, entropy);
    g_launches += 1;
    return cudaGetLastError();
  }
  // 32-row spans once there are enough rows for 64 warps per SM (32 warps: 60k x
  // 16, K = 16, few positive entries 28 us against 25)
  int64_t span = n / (num_sms() * 64);
  span = span < 1 ? 1 : span > 32 ? 32 : span;
  int64_t blocks = (n + 8 * span - 1) / (8 * span);
  if (blocks > num_sms() * 16) blocks = num_sms() * 16;
  auto kern = topk_kernel<VPL, kEntropy, 0, false>;
  if (C == 32 * VPL && !comp)
    kern = K == 8   ? topk_kernel<VPL, kEntropy, 8, true>
           : K == 4 ? topk_kernel<VPL, kEntropy, 4, true>
                    : topk_kernel<VPL, kEntropy, 0, true>;
  kern<<<(int)blocks, 256, 0, st>>>(acc, comp, n, C, ld, K, (int)span, idx, val, entropy);
  g_launches += 1;
  return cudaGetLastError();
}

template <bool kEntropy>
cudaError_t launch_rows(const float* acc, const float* comp, int64_t n, int C, int64_t ld, int K, int32_t* idx,
                        float* val, float* entropy, cudaStream_t st) {
  if (C <= 32) return launch_vpl<1, kEntropy>(acc, comp, n, C, ld, K, idx, val, entropy, st);
  if (C <= 64) return launch_vpl<2, kEntropy>(acc, comp, n, C, ld, K, idx, val, entropy, st);
  if (C <= 128) return launch_vpl<4, kEntropy>(acc, comp, n, C, ld, K, idx, val, entropy, st);
  if (C <= 256) return launch_vpl<8, kEntropy>(acc, comp, n, C, ld, K, idx, val, entropy, st);
  if (C <= 512) return launch_vpl<16, kEntropy>(acc, comp, n, C, ld, K, idx, val, entropy, st);
  return launch_vpl<32, kEntropy>(acc, comp, n, C, ld, K, idx, val, entropy, st);
}

}  // namespace

cudaError_t launch_topk(const float* acc, const float* comp, int64_t n, int C, int K, int32_t* idx, float* val,
                        float* entropy, cudaStream_t st, int64_t ld) {
  if (n <= 0) return cudaSuccess;
  if (ld <= 0) ld = C;
  return entropy ? launch_rows<true>(acc, comp, n, C, ld, K, idx, val, entropy, st)
                 : launch_rows<false>(acc, comp, n, C, ld, K, idx, val, nullptr, st);
}

cudaError_t launch_code_topk(const int32_t* ci, const float* cv, int64_t R, int s, int K,
                             int32_t* ci_out, float* cv_out, cudaStream_t st) {
  if (R <= 0) return cudaSuccess;
  int64_t blocks = (R + 255) / 256;
  if (blocks > num_sms() * 8) blocks = num_sms() * 8;
  code_topk_kernel<<<(int)blocks, 256, 0, st>>>(ci, cv, R, s, K, ci_out, cv_out);
  g_launches += 1;
  return cudaGetLastError();
}

}  // namespace scoup
