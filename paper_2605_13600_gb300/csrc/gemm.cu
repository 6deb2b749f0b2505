// gemm.cu -- BF16 tensor-core GEMM on tcgen05 for the codebook decode
// (paper Sec. 4.3, Eq. 8: F = What C) and the text-query similarity.
//
//   out[M, N] = A[M, K] * Bt[N, K]^T      (A, Bt bf16, K-major; f32 accumulate)
//
// Persistent: one CTA per SM walks the output in units of BM x BN (BM = 128).
// Warp 0 streams 128-byte-swizzled K-major A and Bt tiles (BK = 64 bf16, one
// swizzle row) with TMA into a kStages ring guarded by mbarriers; warp 1
// allocates two BN-column TMEM accumulators and one thread issues
// tcgen05.mma (M=128, N=BN, K=16) into them alternately, so the epilogue of
// one unit overlaps the MMAs of the next; warps 2-5 and 6-9 are two epilogue
// groups whose warps each own a 32-lane TMEM quarter (32 output rows): a unit's
// row chunks of 128 bytes are split between the groups, read back with
// tcgen05.ld, taken through the epilogue, staged 128-byte-swizzled in shared
// memory and written with TMA tile stores (double-buffered per warp).  Two
// groups, because with one warp per scheduler every epilogue instruction waits
// for the one before; and the issuing warps run their loops together (uniform
// registers), because one diverged thread takes longer to build a stage's
// descriptors than the tensor core takes for its MMAs.  480000 bf16 rows to
// 512 features with their norms: K = 64 143 -> 100 us, K = 256 147 -> 145 us
// (768 features, K = 128: 203 -> 145 us).  Epilogues:
//   kOutBF16 : bf16 output, optional per-row sum of squares of the rounded values
//   kOutF32  : f32 output
//   kOutCos  : f32 output / (|row| |column|), 0 where |row| < 1e-12
// Every mbarrier wait is bounded; a wait that gives up records an error in
// *status, raises the CTA's abort flag, and every role leaves after draining
// its own copies in flight; TMEM is freed on every path.  No lane
// is left behind at a warp barrier that another one has skipped (wait_or_abort,
// issuer_wait).
#include <cuda.h>
#include <cuda_bf16.h>

#include "scoup_internal.cuh"
#include "sm100_ptx.cuh"

namespace scoup {
namespace {

constexpr int BM = 128, BK = 64;
constexpr int kEpiWarps = 8;  // two groups of four
constexpr int kGemmThreads = 64 + 32 * kEpiWarps;
constexpr uint32_t kWaitIters = 1u << 22;

template <int BN>
struct GemmCfg {
  static constexpr int kStages = BN >= 256 ? 3 : 4;
  static constexpr uint32_t kTmemCols = 2 * BN;  // two accumulators
};

template <int BN>
struct GemmSmem {
  alignas(1024) __nv_bfloat16 a[GemmCfg<BN>::kStages][BM * BK];
  alignas(1024) __nv_bfloat16 b[GemmCfg<BN>::kStages][BN * BK];
  alignas(1024) unsigned char out[kEpiWarps][2][32 * 128];  // per epilogue warp, two 32-row x 128-byte chunks
  uint64_t full[GemmCfg<BN>::kStages];
  uint64_t empty[GemmCfg<BN>::kStages];
  uint64_t acc_full[2];
  uint64_t acc_empty[2];
  uint64_t part_full[4][4];  // per slot and TMEM quarter: `part` is written
  float part[4][BM];         // half a unit's squared row norms, from one epilogue group to the other
  uint64_t drain;
  uint32_t tmem;
  volatile int abort;
  int ignored;  // what the MMA warp's lanes beside lane 0 report (issuer_wait)
};

// The lanes of a warp poll a barrier and read the flag on their own, and one of
// them may see what the next one has just missed.  A warp whose loop holds warp
// barriers or warp-wide instructions therefore votes, and all its lanes leave
// together (the vote also keeps an issuing warp converged: the producers' loops
// have no other warp barrier).
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, volatile int* abort, int* status) {
  if (__all_sync(0xffffffffu, ptx::mbar_wait_bounded(bar, parity, kWaitIters))) return true;
  atomicOr(status, kStatTimeout);
  *abort = 1;
  return false;
}

__device__ __forceinline__ bool gave_up(const volatile int* abort) { return __any_sync(0xffffffffu, *abort != 0); }

// The MMA issuer does not vote: in front of every stage's MMAs the vote costs 2 to
// 8 % (2073600 FP32 rows of 256 to 512 features 802 us, 741 so).  Its loop holds
// nothing warp-wide, so a lane may leave alone, and lane 0, which issues, alone
// decides: the other lanes report into words that nobody reads, and one that
// gives up only stops keeping lane 0 company.  (Words instead of a branch on the
// lane, which costs as much as the vote.)
__device__ __forceinline__ bool issuer_wait(uint64_t* bar, uint32_t parity, int* abort, int* status) {
  if (ptx::mbar_wait_bounded(bar, parity, kWaitIters)) return true;
  atomicOr(status, kStatTimeout);
  *(volatile int*)abort = 1;
  return false;
}

// acc += the squares of the two bf16 values of w (one packed FP32 FMA).
__device__ __forceinline__ void add_squares(uint32_t w, unsigned long long& acc) {
  asm("{\n\t.reg .b32 l, h;\n\t.reg .b64 v;\n\tshl.b32 l, %1, 16;\n\tand.b32 h, %1, 0xffff0000;\n\t"
      "mov.b64 v, {l, h};\n\tfma.rn.f32x2 %0, v, v, %0;\n\t}"
      : "+l"(acc)
      : "r"(w));
}

__device__ __forceinline__ uint32_t pack_bf16x2(float x, float y) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// Division by a column norm, from the norm and its reciprocal: the quotient
// q = x (1 / norm) is corrected by its exact residual, q + (x - q norm) (1 /
// norm) (Markstein 1990: correctly rounded from a correctly rounded
// reciprocal).  Norms outside 2^-100 .. 2^100 have the second value 0.
__device__ __forceinline__ float2 norm_entry(float n) {
  return make_float2(n, n >= 0x1p-100f && n <= 0x1p100f ? 1.0f / n : 0.0f);
}

__device__ __forceinline__ float div_by_norm(float x, float n, float inv) {
  const float q = x * inv;
  return fabsf(q) < INFINITY ? fmaf(fmaf(-q, n, x), inv, q) : q;  // an infinite x stays so
}

// 32 columns col0 .. of a thread's row in v through the epilogue `mode` into
// the row's 128 bytes of the staging buffer (16-byte pieces swizzled by lane;
// hh: which half of them, a bf16 output has 64 columns there); adds the
// rounded values' squares to ss2 where norms are wanted.
__device__ __forceinline__ void epi_cols(const GemmEpi& ep, int mode, bool norms, bool write, float (&v)[32], int col0,
                                         int hh, int nlim, float rinv, unsigned char* rowp, int lane,
                                         unsigned long long (&ss2)[2]) {
  if (mode == kOutBF16) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint4 w = make_uint4(pack_bf16x2(v[8 * j], v[8 * j + 1]), pack_bf16x2(v[8 * j + 2], v[8 * j + 3]),
                                 pack_bf16x2(v[8 * j + 4], v[8 * j + 5]), pack_bf16x2(v[8 * j + 6], v[8 * j + 7]));
      if (write) *reinterpret_cast<uint4*>(rowp + (((4 * hh + j) ^ (lane & 7)) << 4)) = w;
      if (norms) {
        add_squares(w.x, ss2[0]);
        add_squares(w.y, ss2[1]);
        add_squares(w.z, ss2[0]);
        add_squares(w.w, ss2[1]);
      }
    }
  } else {
    if (mode == kOutCos || mode == kOutRel) {
      // one norm load and one division per lane and chunk, passed around the
      // warp: a load and a branchy division per column are a serial chain of
      // several thousand cycles per row block
      const int col = col0 + lane;
      const float2 mine = norm_entry(col < nlim ? ep.colnorm[col] : 1.0f);
      if (__all_sync(0xffffffffu, mine.y != 0.0f)) {
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          const float n = __shfl_sync(0xffffffffu, mine.x, c), inv = __shfl_sync(0xffffffffu, mine.y, c);
          const float s = div_by_norm(v[c] * rinv, n, inv);
          v[c] = rinv == 0.0f ? 0.0f : s;
        }
      } else {  // a norm of 0 or at the ends of the range: a column without a norm gives 0
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          const float n = __shfl_sync(0xffffffffu, mine.x, c);
          v[c] = (rinv == 0.0f || n == 0.0f) ? 0.0f : v[c] * rinv / n;
        }
      }
    }
    if (mode == kOutRel) {
      // Eq. 9 on the thread's whole row of similarities (at most 32
      // columns, one column tile): R_q = min_k 1 / (1 + e^{a (s_k - s_q)})
      // is the term of the largest canonical similarity; query q is
      // column n_canon + q, staged at column q of the relevancy row
      float smax = -INFINITY;
#pragma unroll
      for (int c = 0; c < 32; ++c)
        if (c < ep.n_canon) smax = fmaxf(smax, v[c]);
      float* rowf = reinterpret_cast<float*>(rowp);
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        const int qq = c - ep.n_canon;
        if (qq >= 0 && c < nlim) {
          const float r = relevancy_term(ep.alpha, smax, v[c]);
          rowf[(((qq >> 2) ^ (lane & 7)) << 2) + (qq & 3)] = r;
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        *reinterpret_cast<float4*>(rowp + ((j ^ (lane & 7)) << 4)) =
            make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
    }
  }
}

// Position of a CTA's i-th unit.  Plain: units u = blockIdx.x + i gridDim.x
// in row-block-major order.  Fused query: the CTA's row blocks
// rb = blockIdx.x + j gridDim.x, each as its n_tiles column units followed by
// the query unit (so one epilogue thread sees every column of its row).
struct UnitPos {
  int m0, n0;
  bool query, valid;
};

template <int BN, bool kQuery>
__device__ __forceinline__ UnitPos unit_at(int i, int n_tiles, int m_blocks) {
  UnitPos p;
  if constexpr (!kQuery) {
    const int u = blockIdx.x + i * (int)gridDim.x;
    p.m0 = (u / n_tiles) * BM;
    p.n0 = (u % n_tiles) * BN;
    p.query = false;
    p.valid = u < m_blocks * n_tiles;
  } else {
    const int per = n_tiles + 1, rb = blockIdx.x + (i / per) * (int)gridDim.x, j = i % per;
    p.m0 = rb * BM;
    p.n0 = j * BN;
    p.query = j == n_tiles;
    p.valid = rb < m_blocks;
  }
  return p;
}

// kQuery: the fused query unit (compiled out of the plain launches).
template <int BN, bool kQuery>
__global__ void __launch_bounds__(kGemmThreads, 1) gemm_bf16_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                    const __grid_constant__ CUtensorMap tmB,
                                                                    const __grid_constant__ CUtensorMap tmO,
                                                                    const __grid_constant__ CUtensorMap tmG,
                                                                    const __grid_constant__ CUtensorMap tmS,
                                                                    GemmEpi ep) {
  using Cfg = GemmCfg<BN>;
  constexpr int kStages = Cfg::kStages;
  extern __shared__ __align__(1024) unsigned char gsm_raw[];
  unsigned char* base = gsm_raw + ((1024 - (ptx::smem_u32(gsm_raw) & 1023u)) & 1023u);
  GemmSmem<BN>& sm = *reinterpret_cast<GemmSmem<BN>*>(base);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kt = (ep.K + BK - 1) / BK;
  const int n_tiles = (ep.N + BN - 1) / BN;
  const int m_blocks = (ep.M + BM - 1) / BM;
  constexpr bool fused = kQuery;
  constexpr uint32_t kBytesA = BM * BK * 2, kBytesB = BN * BK * 2;
  const uint32_t kBytesG = (uint32_t)ep.sim_n * BK * 2;
  constexpr uint32_t idesc = ptx::idesc_bf16_f32(BM, BN);
  const uint32_t idesc_q = ep.sim_n == 16 ? ptx::idesc_bf16_f32(BM, 16) : ptx::idesc_bf16_f32(BM, 32);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(&sm.full[s], 1);
      ptx::mbar_init(&sm.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(&sm.acc_full[b], 1);
      ptx::mbar_init(&sm.acc_empty[b], kEpiWarps);
    }
    for (int i = 0; i < 16; ++i) ptx::mbar_init(&sm.part_full[i >> 2][i & 3], 1);
    ptx::mbar_init(&sm.drain, 1);
    sm.abort = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(&tmA);
    ptx::prefetch_tmap(&tmB);
    ptx::prefetch_tmap(&tmO);
    if (fused) {
      ptx::prefetch_tmap(&tmG);
      ptx::prefetch_tmap(&tmS);
    }
  }
  if (warp == 1) {
    ptx::tmem_alloc(&sm.tmem, Cfg::kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = sm.tmem;

  if (warp == 0) {
    // ---- TMA producer: the warp runs the loop together, so that addresses
    // and coordinates stay in uniform registers, and lane 0 issues ----
    int it = 0;
    for (int i = 0; !ep.stall_loads && !gave_up(&sm.abort); ++i) {
      const UnitPos t = unit_at<BN, kQuery>(i, n_tiles, m_blocks);
      if (!t.valid) break;
      const CUtensorMap* mb = t.query ? &tmG : &tmB;
      const int nb = t.query ? 0 : t.n0;
      for (int kb = 0; kb < kt; ++kb, ++it) {
        const int s = it % kStages;
        if (it >= kStages && !wait_or_abort(&sm.empty[s], ((it / kStages) - 1) & 1, &sm.abort, ep.status)) break;
        if (lane == 0) {
          ptx::mbar_arrive_expect_tx(&sm.full[s], kBytesA + (t.query ? kBytesG : kBytesB));
          ptx::tma_load_2d(sm.a[s], &tmA, &sm.full[s], kb * BK, t.m0);
          ptx::tma_load_2d(sm.b[s], mb, &sm.full[s], kb * BK, nb);
        }
      }
    }
    // wait (bounded) for the last copy issued into each stage before leaving
    for (int s = 0; s < kStages && s < it; ++s) {
      const int last = s + ((it - 1 - s) / kStages) * kStages;
      if (!ptx::mbar_wait_bounded(&sm.full[s], (last / kStages) & 1, kWaitIters)) atomicOr(ep.status, kStatTimeout);
    }
  } else if (warp == 1) {
    // ---- MMA issuer: the warp runs the loop together, so that descriptors
    // and addresses stay in uniform registers, and lane 0 issues ----
    const uint64_t da0 = ptx::smem_desc_k128(ptx::smem_u32(sm.a[0])), db0 = ptx::smem_desc_k128(ptx::smem_u32(sm.b[0]));
    int it = 0, local = 0;
    bool ok = true;
    int* const my_abort = lane == 0 ? const_cast<int*>(&sm.abort) : &sm.ignored;
    int* const my_status = lane == 0 ? ep.status : &sm.ignored;
    for (int i = 0; ok && !sm.abort; ++i, ++local) {
      const UnitPos t = unit_at<BN, kQuery>(i, n_tiles, m_blocks);
      if (!t.valid) break;
      const uint32_t id = t.query ? idesc_q : idesc;
      const int b = local & 1, use = local >> 1;
      if (local >= 2 && !issuer_wait(&sm.acc_empty[b], (use - 1) & 1, my_abort, my_status)) break;
      ptx::tc_fence_after();
      const uint32_t d = tmem + (uint32_t)(b * BN);
      for (int kb = 0; kb < kt; ++kb, ++it) {
        const int s = it % kStages;
        if (!issuer_wait(&sm.full[s], (it / kStages) & 1, my_abort, my_status)) {
          ok = false;
          break;
        }
        ptx::tc_fence_after();
        const uint64_t da = da0 + (uint64_t)(s * (int)(kBytesA >> 4)), db = db0 + (uint64_t)(s * (int)(kBytesB >> 4));
        if (lane == 0) {
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) ptx::mma_f16(d, da + 2 * k, db + 2 * k, id, (kb > 0 || k > 0) ? 1u : 0u);
          ptx::mma_commit(&sm.empty[s]);
        }
      }
      if (ok && lane == 0) ptx::mma_commit(&sm.acc_full[b]);
    }
    // every issued MMA has completed once `drain` flips
    if (lane == 0) {
      ptx::mma_commit(&sm.drain);
      if (!ptx::mbar_wait_bounded(&sm.drain, 0, kWaitIters)) atomicOr(ep.status, kStatTimeout);
    }
    __syncwarp();
  } else if (warp >= 2) {
    // ---- epilogue ----
    const int q = warp & 3;               // TMEM lane quarter this warp may access
    const int grp = (warp - 2) >> 2;      // epilogue group
    constexpr int kCW = 64;               // bf16 columns per 128-byte chunk (32 for f32 output)
    const int per = n_tiles + 1;          // fused query: units of a row block
    const bool norms = fused || ep.rownorm2;
    int local = 0, sbuf = 0, ex = 0;      // ex: units whose norms the groups have exchanged
    float ss_row = 0.0f;  // fused query: squared norm of the row's rounded outputs over its row block
    for (int i = 0; !gave_up(&sm.abort); ++i, ++local) {
      const UnitPos t = unit_at<BN, kQuery>(i, n_tiles, m_blocks);
      if (!t.valid) break;
      const int m0 = t.m0, n0 = t.query ? 0 : t.n0;
      const int mode = (kQuery && t.query) ? ep.sim_mode : ep.mode;
      const bool f32out = mode != kOutBF16;
      const int cw = f32out ? 32 : kCW;
      const int ncols = (kQuery && t.query) ? ep.sim_n : BN;  // accumulator columns of this unit (sim_n <= 32)
      const int nlim = t.query ? ep.sim_n : ep.N;
      const bool write = kQuery ? (t.query || ep.store) : true;
      const CUtensorMap* mo = t.query ? &tmS : &tmO;
      const int b = local & 1, use = local >> 1;
      // The lead group takes a unit of one chunk alone, or the first half of
      // the chunks; it gathers the row norms.  Units of a row block with a
      // query unit have one lead, and the groups lead by turns.
      const int lead = (kQuery ? i / per : local) & 1;
      const bool split = ncols > cw;
      const int half = split ? ((ncols / cw + 1) / 2) * cw : ncols;
      const int c_begin = grp == lead ? 0 : half, c_end = grp == lead ? half : ncols;
      if (!wait_or_abort(&sm.acc_full[b], use & 1, &sm.abort, ep.status)) break;
      ptx::tc_fence_after();
      const int row = m0 + q * 32 + lane;
      if (fused && !t.query && t.n0 == 0) ss_row = 0.0f;
      float rinv = 0.0f;
      if ((mode == kOutCos || mode == kOutRel) && c_begin < c_end && row < ep.M) {
        const float rn = sqrtf(t.query ? ss_row : ep.rownorm2[row]);
        rinv = rn < 1e-12f ? 0.0f : 1.0f / rn;
      }
      unsigned long long ss2[2] = {0ull, 0ull};
      const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * BN);
      if (c_begin >= c_end) {  // nothing to read in this unit
        if (lane == 0) ptx::mbar_arrive(&sm.acc_empty[b]);
      }
      for (int c0 = c_begin; c0 < c_end; c0 += cw) {
        unsigned char* buf = sm.out[warp - 2][sbuf];
        unsigned char* rowp = buf + lane * 128;
        // a box that starts past the last row or column stores nothing
        const bool dead = n0 + c0 >= nlim || m0 + q * 32 >= ep.M;
        if (write && !dead) {
          if (lane == 0) ptx::bulk_wait_read<1>();  // this buffer's previous store has read it
          __syncwarp();
        }
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          if (hh * 32 >= cw) break;
          float v[32];
          ptx::tmem_ld32(tbase + (uint32_t)(c0 + 32 * hh), v);
          if (c0 + 32 * (hh + 1) >= c_end) {
            // the group's part is drained: the MMA warp may reuse the accumulator
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&sm.acc_empty[b]);
          }
          if (!dead) epi_cols(ep, mode, norms, write, v, n0 + c0 + 32 * hh, hh, nlim, rinv, rowp, lane, ss2);
        }
        if (dead) continue;
        if (!write) continue;
        ptx::fence_async_shared();
        __syncwarp();
        if (lane == 0) {
          ptx::tma_store_2d(mo, buf, n0 + c0, m0 + q * 32);
          ptx::bulk_commit();
        }
        sbuf ^= 1;
      }
      if (norms && !f32out) {
        const float2 s0 = *reinterpret_cast<const float2*>(&ss2[0]), s1 = *reinterpret_cast<const float2*>(&ss2[1]);
        float ss = (s0.x + s1.x) + (s0.y + s1.y);
        if (split) {
          // four slots: a slot is written again four units on, and that unit's
          // MMAs wait for both groups to have left the unit before last
          uint64_t* const bar = &sm.part_full[ex & 3][q];
          float* const part = &sm.part[ex & 3][q * 32 + lane];
          if (grp != lead) {
            *part = ss;
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar);
          } else {
            if (!wait_or_abort(bar, (ex >> 2) & 1, &sm.abort, ep.status)) break;
            ss += *part;
          }
          ++ex;
        }
        if (fused)
          ss_row += ss;
        else if (row < ep.M && grp == lead)
          atomicAdd(&ep.rownorm2[row], ss);
      }
      if (fused && t.query && grp == lead && ep.rownorm2 && row < ep.M) ep.rownorm2[row] = ss_row;
    }
    if (lane == 0) ptx::bulk_wait<0>();  // stores complete before the CTA leaves
    __syncwarp();
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, Cfg::kTmemCols);
  }
}

// ---- rows kept in shared memory (K <= 256) ----
//
// out = A Bt^T as above for the decode's shapes: many rows, K <= 256.  A CTA
// takes a block of rows at a time: its A (up to 4 slabs of 64 columns) stays
// in shared memory while the column tiles of 128 stream past it, where the
// kernel above loads A again for every column unit.  What bounds both is the
// ring of loads in front of the MMAs: a stage comes back about 1.8 us after
// it was freed, so the bytes per row block over the bytes in flight count.
//   bf16 A: 256 rows to a block (every Bt tile serves two MMAs), epilogue
//     group g owns row half g over all columns.  All 128 KB of A are in use,
//     so a slab is refilled as soon as the block's last unit has read it; the
//     next block is fetched into L2 ahead.  The query unit goes first and
//     waits as 32 registers per row, so that its MMAs do not stand between
//     the last column tile and the refill.
//   FP32 A: six more warps round the values to bf16 on the way in, in place of
//     a conversion pass over memory.  128 rows to a block and 6 slots, so that
//     the next block is converted under this one's MMAs; the epilogue groups
//     split the columns and pass the row norms on in shared memory.
// 2073600 x 256 -> 512 and 32 phrases: bf16 880 -> 643 us, FP32 1514 -> 998
// us; FP32 without the phrases 1127 -> 741 us, of which 625 are the bytes.
constexpr int RN = 128;
constexpr int kMaxSlabs = 4;
constexpr int kCvtWarps = 6;  // two teams that take the slabs by turns

template <bool kF32A>
struct RowsCfg {
  static constexpr int kHalves = kF32A ? 1 : 2;         // 128-row halves of a block
  static constexpr int kRows = kHalves * BM;
  static constexpr int kASlots = kF32A ? 6 : kMaxSlabs;
  static constexpr int kBStages = kF32A ? 6 : 4;
  static constexpr int kAcc = 4 / kHalves;              // accumulators of kHalves x RN TMEM columns
  static constexpr int kThreads = 64 + 32 * kEpiWarps + (kF32A ? 32 * kCvtWarps : 0);
};
constexpr int kParts = 3;

template <bool kF32A>
struct RowsSmem {
  using Cfg = RowsCfg<kF32A>;
  alignas(1024) __nv_bfloat16 a[Cfg::kASlots][Cfg::kHalves][BM * BK];
  alignas(1024) __nv_bfloat16 b[Cfg::kBStages][RN * BK];
  alignas(1024) unsigned char out[kEpiWarps][32 * 128];
  float part[kF32A ? kParts : 1][BM];  // squared row norms over the other group's columns, for the lead group
  uint64_t part_full[kParts][4];       // per slot and TMEM quarter: `part` is written
  uint64_t a_full[Cfg::kASlots];
  uint64_t a_empty[Cfg::kASlots];
  uint64_t b_full[Cfg::kBStages];
  uint64_t b_empty[Cfg::kBStages];
  uint64_t acc_full[Cfg::kAcc];
  uint64_t acc_empty[Cfg::kAcc];
  uint64_t drain;
  uint32_t tmem;
  volatile int abort;
  int ignored;  // what the MMA warp's lanes beside lane 0 report (issuer_wait)
};
static_assert(sizeof(RowsSmem<false>) + 1024 <= 227 * 1024, "shared memory of one CTA");
static_assert(sizeof(RowsSmem<true>) + 1024 <= 227 * 1024, "shared memory of one CTA");

template <bool kQuery, bool kF32A>
__global__ void __launch_bounds__(RowsCfg<kF32A>::kThreads, 1)
    gemm_rows_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmG,
                     const __grid_constant__ CUtensorMap tmS, const float* __restrict__ a32, GemmEpi ep) {
  using Cfg = RowsCfg<kF32A>;
  constexpr int kH = Cfg::kHalves, kRows = Cfg::kRows, kASlots = Cfg::kASlots, kBStages = Cfg::kBStages;
  constexpr int kAcc = Cfg::kAcc;
  extern __shared__ __align__(1024) unsigned char gsm_raw[];
  unsigned char* base = gsm_raw + ((1024 - (ptx::smem_u32(gsm_raw) & 1023u)) & 1023u);
  RowsSmem<kF32A>& sm = *reinterpret_cast<RowsSmem<kF32A>*>(base);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kt = (ep.K + BK - 1) / BK;  // slabs, at most kMaxSlabs
  const int n_tiles = (ep.N + RN - 1) / RN, per = n_tiles + (kQuery ? 1 : 0);
  constexpr int kU0 = kQuery ? 1 : 0;   // unit of column tile 0: the query unit is unit 0
  const int blocks = (ep.M - 1) / kRows + 1;
  constexpr uint32_t kBytesA = kRows * BK * 2, kBytesB = RN * BK * 2;
  const uint32_t kBytesG = (uint32_t)ep.sim_n * BK * 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kASlots; ++s) {
      ptx::mbar_init(&sm.a_full[s], kF32A ? 32 * kCvtWarps / 2 : 1);
      ptx::mbar_init(&sm.a_empty[s], 1);
    }
    for (int s = 0; s < kBStages; ++s) {
      ptx::mbar_init(&sm.b_full[s], 1);
      ptx::mbar_init(&sm.b_empty[s], 1);
    }
    for (int b = 0; b < kAcc; ++b) {
      ptx::mbar_init(&sm.acc_full[b], 1);
      ptx::mbar_init(&sm.acc_empty[b], kEpiWarps);
    }
    for (int i = 0; i < 4 * kParts; ++i) ptx::mbar_init(&sm.part_full[i >> 2][i & 3], 1);
    ptx::mbar_init(&sm.drain, 1);
    sm.abort = 0;
    ptx::fence_mbar_init();
    if (!kF32A) ptx::prefetch_tmap(&tmA);
    ptx::prefetch_tmap(&tmB);
    ptx::prefetch_tmap(&tmO);
    if (kQuery) {
      ptx::prefetch_tmap(&tmG);
      ptx::prefetch_tmap(&tmS);
    }
  }
  if (warp == 1) {
    ptx::tmem_alloc(&sm.tmem, kAcc * kH * RN);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = sm.tmem;

  if (warp == 0) {
    // ---- TMA producer (see above): the units of every row block, a slab of A
    // ahead of the first unit that needs it ----
    int ia = 0, it = 0;
    bool ok = !ep.stall_loads;
    for (int rb = blockIdx.x; ok && rb < blocks && !gave_up(&sm.abort); rb += (int)gridDim.x) {
      const int m0 = rb * kRows, next = rb + (int)gridDim.x;
      for (int u = 0; ok && u < per; ++u) {
        const bool query = kQuery && u == 0;
        for (int kb = 0; kb < kt; ++kb, ++it) {
          if (!kF32A && u == 0) {
            const int s = ia % kASlots;
            if (ia >= kASlots && !wait_or_abort(&sm.a_empty[s], ((ia / kASlots) - 1) & 1, &sm.abort, ep.status)) {
              ok = false;
              break;
            }
            if (lane == 0) {
              ptx::mbar_arrive_expect_tx(&sm.a_full[s], kBytesA);
              for (int h = 0; h < kH; ++h) ptx::tma_load_2d(sm.a[s][h], &tmA, &sm.a_full[s], kb * BK, m0 + h * BM);
            }
            ++ia;
          }
          const int s = it % kBStages;
          if (it >= kBStages && !wait_or_abort(&sm.b_empty[s], ((it / kBStages) - 1) & 1, &sm.abort, ep.status)) {
            ok = false;
            break;
          }
          if (lane == 0) {
            ptx::mbar_arrive_expect_tx(&sm.b_full[s], query ? kBytesG : kBytesB);
            ptx::tma_load_2d(sm.b[s], query ? &tmG : &tmB, &sm.b_full[s], kb * BK, query ? 0 : (u - kU0) * RN);
          }
        }
        if (!kF32A && lane == 0 && u == 0 && next < blocks)
          for (int kb = 0; kb < kt; ++kb)
            for (int h = 0; h < kH; ++h)
              if (next * kRows + h * BM < ep.M) ptx::tma_prefetch_2d(&tmA, kb * BK, next * kRows + h * BM);
      }
    }
    // wait (bounded) for the last copy issued into each slot before leaving
    for (int s = 0; s < kBStages && s < it; ++s) {
      const int last = s + ((it - 1 - s) / kBStages) * kBStages;
      if (!ptx::mbar_wait_bounded(&sm.b_full[s], (last / kBStages) & 1, kWaitIters)) atomicOr(ep.status, kStatTimeout);
    }
    for (int s = 0; s < kASlots && s < ia; ++s) {
      const int last = s + ((ia - 1 - s) / kASlots) * kASlots;
      if (!ptx::mbar_wait_bounded(&sm.a_full[s], (last / kASlots) & 1, kWaitIters)) atomicOr(ep.status, kStatTimeout);
    }
  } else if (warp == 1) {
    // ---- MMA issuer (see above) ----
    constexpr uint32_t idesc = ptx::idesc_bf16_f32(BM, RN);
    const uint32_t idesc_q = ep.sim_n == 16 ? ptx::idesc_bf16_f32(BM, 16) : ptx::idesc_bf16_f32(BM, 32);
    const uint64_t da0 = ptx::smem_desc_k128(ptx::smem_u32(sm.a[0][0])), db0 = ptx::smem_desc_k128(ptx::smem_u32(sm.b[0]));
    int ia = 0, it = 0, local = 0;
    bool ok = true;
    int* const my_abort = lane == 0 ? const_cast<int*>(&sm.abort) : &sm.ignored;
    int* const my_status = lane == 0 ? ep.status : &sm.ignored;
    for (int rb = blockIdx.x; ok && rb < blocks && !sm.abort; rb += (int)gridDim.x, ia += kt) {
      for (int u = 0; ok && u < per; ++u, ++local) {
        const uint32_t id = kQuery && u == 0 ? idesc_q : idesc;
        const int b = local % kAcc, use = local / kAcc;
        if (local >= kAcc && !issuer_wait(&sm.acc_empty[b], (use - 1) & 1, my_abort, my_status)) {
          ok = false;
          break;
        }
        ptx::tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(b * kH * RN);
        for (int kb = 0; kb < kt; ++kb, ++it) {
          const int sa = (ia + kb) % kASlots, s = it % kBStages;
          if ((u == 0 && !issuer_wait(&sm.a_full[sa], ((ia + kb) / kASlots) & 1, my_abort, my_status)) ||
              !issuer_wait(&sm.b_full[s], (it / kBStages) & 1, my_abort, my_status)) {
            ok = false;
            break;
          }
          ptx::tc_fence_after();
          const uint64_t da = da0 + (uint64_t)(sa * (int)(kBytesA >> 4)), db = db0 + (uint64_t)(s * (int)(kBytesB >> 4));
          if (lane == 0) {
#pragma unroll
            for (int h = 0; h < kH; ++h)
#pragma unroll
              for (int k = 0; k < BK / 16; ++k)
                ptx::mma_f16(d + (uint32_t)(h * RN), da + h * (BM * BK * 2 >> 4) + 2 * k, db + 2 * k, id,
                             (kb > 0 || k > 0) ? 1u : 0u);
            ptx::mma_commit(&sm.b_empty[s]);
            if (u == per - 1) ptx::mma_commit(&sm.a_empty[sa]);
          }
        }
        if (ok && lane == 0) ptx::mma_commit(&sm.acc_full[b]);
      }
    }
    // every issued MMA has completed once `drain` flips
    if (lane == 0) {
      ptx::mma_commit(&sm.drain);
      if (!ptx::mbar_wait_bounded(&sm.drain, 0, kWaitIters)) atomicOr(ep.status, kStatTimeout);
    }
    __syncwarp();
  } else if (warp >= 2 && warp < 2 + kEpiWarps) {
    // ---- epilogue ----
    const int q = warp & 3, grp = (warp - 2) >> 2;  // TMEM lane quarter; epilogue group
    const bool norms = kQuery || ep.rownorm2;
    unsigned char* const buf = sm.out[warp - 2];
    unsigned char* const rowp = buf + lane * 128;
    int local = 0;
    bool ok = true;
    for (int rb = blockIdx.x, j = 0; ok && rb < blocks && !gave_up(&sm.abort); rb += (int)gridDim.x, ++j) {
      // one half to a block: the lead group takes the first half of each
      // column tile, gathers the row norms and does the query unit; the groups
      // lead by turns.  Two halves: each group leads its own rows.
      const bool lead = kH == 2 || grp == (j & 1);
      const int r0 = rb * kRows + (kH == 2 ? grp * BM : 0) + q * 32, row = r0 + lane;
      const bool live = r0 < ep.M;
      const int c_begin = lead ? 0 : RN / 2, c_end = kH == 2 || !lead ? RN : RN / 2;
      unsigned long long ss2[2] = {0ull, 0ull};  // squared norm of the thread's rounded outputs
      float dots[32];                            // the query unit's sums
      for (int u = 0; u < per; ++u, ++local) {
        const int b = local % kAcc, use = local / kAcc;
        if (!wait_or_abort(&sm.acc_full[b], use & 1, &sm.abort, ep.status)) {
          ok = false;
          break;
        }
        ptx::tc_fence_after();
        const uint32_t taddr =
            tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * kH * RN + (kH == 2 ? grp * RN : 0));
        if (kQuery && u == 0) {
          if (lead) ptx::tmem_ld32(taddr, dots);
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&sm.acc_empty[b]);
          continue;
        }
        const int n0 = (u - kU0) * RN;
        const bool bf16 = ep.mode == kOutBF16, write = !kQuery || ep.store;
        const int cw = bf16 ? 64 : 32;  // columns of a 128-byte chunk
        for (int c0 = c_begin; c0 < c_end; c0 += cw) {
          const bool dead = n0 + c0 >= ep.N || !live;  // a box that starts past the last row or column
          if (write && !dead) {
            if (lane == 0) ptx::bulk_wait_read<0>();  // the previous store has read the buffer
            __syncwarp();
          }
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            if (hh * 32 >= cw) break;
            float v[32];
            ptx::tmem_ld32(taddr + (uint32_t)(c0 + 32 * hh), v);
            if (c0 + 32 * (hh + 1) >= c_end) {
              // this warp's part is drained: the MMA warp may reuse the accumulator
              ptx::tc_fence_before();
              __syncwarp();
              if (lane == 0) ptx::mbar_arrive(&sm.acc_empty[b]);
            }
            if (!dead) epi_cols(ep, ep.mode, norms, write, v, n0 + c0 + 32 * hh, hh, ep.N, 0.0f, rowp, lane, ss2);
          }
          if (dead || !write) continue;
          ptx::fence_async_shared();
          __syncwarp();
          if (lane == 0) {
            ptx::tma_store_2d(&tmO, buf, n0 + c0, r0);
            ptx::bulk_commit();
          }
        }
      }
      if (!ok || !norms) continue;
      const float2 s0 = *reinterpret_cast<const float2*>(&ss2[0]), s1 = *reinterpret_cast<const float2*>(&ss2[1]);
      float ss = (s0.x + s1.x) + (s0.y + s1.y);
      if constexpr (kH == 1) {
        // a unit's MMAs wait until both groups have left the unit before the
        // one kAcc back; with at least two units to a block (N > 128) that is
        // past the block kParts back, whose slot is written again here
        uint64_t* const bar = &sm.part_full[j % kParts][q];
        float* const part = &sm.part[j % kParts][q * 32 + lane];
        if (!lead) {
          *part = ss;
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(bar);
          continue;
        }
        if (!wait_or_abort(bar, (j / kParts) & 1, &sm.abort, ep.status)) {
          ok = false;
          continue;
        }
        ss += *part;
      }
      if (ep.rownorm2 && row < ep.M) ep.rownorm2[row] = ss;
      if (kQuery && live) {
        const float rn = sqrtf(ss);
        if (lane == 0) ptx::bulk_wait_read<0>();
        __syncwarp();
        epi_cols(ep, ep.sim_mode, false, true, dots, 0, 0, ep.sim_n, rn < 1e-12f ? 0.0f : 1.0f / rn, rowp, lane, ss2);
        ptx::fence_async_shared();
        __syncwarp();
        if (lane == 0) {
          ptx::tma_store_2d(&tmS, buf, 0, r0);
          ptx::bulk_commit();
        }
      }
    }
    if (lane == 0) ptx::bulk_wait<0>();  // stores complete before the CTA leaves
    __syncwarp();
  } else if (kF32A && warp >= 2 + kEpiWarps) {
    // ---- converters: FP32 rows to swizzled bf16 slabs ----
    // Two teams of three warps take the slabs by turns.  16 threads read 64
    // columns of a row (256 bytes), a thread's rows of the slab all in flight;
    // every thread writes 8 bytes of a row's 128-byte swizzle line.
    constexpr int kTeam = 32 * kCvtWarps / 2, kRowsPer = kTeam / 16, kBatch = (BM + kRowsPer - 1) / kRowsPer;
    const int t = threadIdx.x - 32 * (2 + kEpiWarps), team = t / kTeam, rt = (t % kTeam) >> 4, ct = (t & 15) * 4;
    int ia = 0;
    bool ok = true;
    for (int rb = blockIdx.x; ok && rb < blocks && !gave_up(&sm.abort); rb += (int)gridDim.x) {
      const int m0 = rb * kRows, next = rb + (int)gridDim.x;
      if (t == 0 && next < blocks) {
        const int rows = min(kRows, ep.M - next * kRows);
        ptx::bulk_prefetch_l2(a32 + (int64_t)next * kRows * ep.K, (uint32_t)rows * (uint32_t)ep.K * 4u);
      }
      for (int kb = 0; kb < kt; ++kb, ++ia) {
        if ((ia & 1) != team) continue;
        const int s = ia % kASlots, col = kb * BK + ct;
        float4 x[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
          const int r = i * kRowsPer + rt;
          x[i] = r < BM && m0 + r < ep.M && col < ep.K
                     ? __ldcs(reinterpret_cast<const float4*>(a32 + (int64_t)(m0 + r) * ep.K + col))
                     : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        if (ia >= kASlots && !wait_or_abort(&sm.a_empty[s], ((ia / kASlots) - 1) & 1, &sm.abort, ep.status)) {
          ok = false;
          break;
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
          const int r = i * kRowsPer + rt;
          unsigned char* line = reinterpret_cast<unsigned char*>(sm.a[s][0]) + r * 128;
          if (r < BM)
            *reinterpret_cast<uint2*>(line + ((((ct >> 3) ^ (r & 7)) << 4) | ((ct & 4) << 1))) =
                make_uint2(pack_bf16x2(x[i].x, x[i].y), pack_bf16x2(x[i].z, x[i].w));
        }
        ptx::fence_async_shared();  // the slab is read by the tensor core (async proxy)
        ptx::mbar_arrive(&sm.a_full[s]);
      }
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, kAcc * kH * RN);
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

// Row-major 2-D matrix [rows, cols] (row stride cols elements), box
// [box_rows, box_cols], 128-byte swizzle (box_cols x element size = 128 bytes).
bool make_tmap(CUtensorMap* m, const void* ptr, CUtensorMapDataType dt, int esize, int64_t rows, int64_t cols,
               int box_cols, int box_rows) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * (cuuint64_t)esize};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1u, 1u};
  return enc(m, dt, 2, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Gt (bf16 [sim_n, K]) is the fused query's operand; null without one.
template <int BN>
cudaError_t launch_bn(const void* A, const void* Bt, const void* Gt, const GemmEpi& ep, cudaStream_t st) {
  CUtensorMap ta, tb, to, tg, ts;
  const bool f32out = ep.mode != kOutBF16;
  const bool fused = ep.sim_n > 0;
  if (!make_tmap(&ta, A, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ep.M, ep.K, BK, BM) ||
      !make_tmap(&tb, Bt, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ep.N, ep.K, BK, BN))
    return cudaErrorInvalidValue;
  // without stored rows (fused query, store = 0) the output map is never used:
  // it is encoded on the operand Bt so that it is valid
  if (!ep.store) to = tb;
  else if (!(f32out ? make_tmap(&to, ep.out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, ep.M, ep.ldo, 32, 32)
                    : make_tmap(&to, ep.out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ep.M, ep.ldo, 64, 32)))
    return cudaErrorInvalidValue;
  if (fused) {
    if (!make_tmap(&tg, Gt, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ep.sim_n, ep.K, BK, ep.sim_n) ||
        !make_tmap(&ts, ep.sim_out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, ep.M, ep.sim_ldo, 32, 32))
      return cudaErrorInvalidValue;
  } else {
    tg = tb;  // unused
    ts = to;
  }
  const size_t smem = sizeof(GemmSmem<BN>) + 1024;
  auto kern = fused ? gemm_bf16_kernel<BN, true> : gemm_bf16_kernel<BN, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t m_blocks = (ep.M + BM - 1) / BM;
  const int64_t units = fused ? m_blocks : m_blocks * ((ep.N + BN - 1) / BN);
  const int grid = (int)(units < num_sms() ? units : num_sms());
  kern<<<grid, kGemmThreads, smem, st>>>(ta, tb, to, tg, ts, ep);
  g_launches += 1;
  return cudaGetLastError();
}

template <bool kQuery, bool kF32A>
cudaError_t launch_rows(const void* A, const void* Bt, const void* Gt, const GemmEpi& ep, cudaStream_t st) {
  CUtensorMap ta, tb, to, tg, ts;
  if (!make_tmap(&tb, Bt, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ep.N, ep.K, BK, RN)) return cudaErrorInvalidValue;
  ta = to = tg = ts = tb;  // a map that is never used is still valid
  if (!kF32A && !make_tmap(&ta, A, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ep.M, ep.K, BK, BM)) return cudaErrorInvalidValue;
  if (ep.store &&
      !(ep.mode == kOutF32 ? make_tmap(&to, ep.out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, ep.M, ep.ldo, 32, 32)
                           : make_tmap(&to, ep.out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ep.M, ep.ldo, 64, 32)))
    return cudaErrorInvalidValue;
  if (kQuery && (!make_tmap(&tg, Gt, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ep.sim_n, ep.K, BK, ep.sim_n) ||
                 !make_tmap(&ts, ep.sim_out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, ep.M, ep.sim_ldo, 32, 32)))
    return cudaErrorInvalidValue;
  const size_t smem = sizeof(RowsSmem<kF32A>) + 1024;
  auto kern = gemm_rows_kernel<kQuery, kF32A>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int blocks = (ep.M - 1) / RowsCfg<kF32A>::kRows + 1, grid = blocks < num_sms() ? blocks : num_sms();
  kern<<<grid, RowsCfg<kF32A>::kThreads, smem, st>>>(ta, tb, to, tg, ts, (const float*)A, ep);
  g_launches += 1;
  return cudaGetLastError();
}

// ---- small conversion kernels ----
__global__ void f32_to_bf16_kernel(const float* __restrict__ x, __nv_bfloat16* __restrict__ y, int64_t n, WsHeader* hdr) {
  if (hdr && blockIdx.x == 0)  // a call's first launch clears its header
    for (int i = threadIdx.x; i < (int)(sizeof(WsHeader) / 4); i += blockDim.x) ((uint32_t*)hdr)[i] = 0u;
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * 4; i < n; i += (int64_t)gridDim.x * blockDim.x * 4) {
    if (i + 3 < n) {
      const float4 v = *reinterpret_cast<const float4*>(x + i);
      *reinterpret_cast<__nv_bfloat162*>(y + i) = __floats2bfloat162_rn(v.x, v.y);
      *reinterpret_cast<__nv_bfloat162*>(y + i + 2) = __floats2bfloat162_rn(v.z, v.w);
    } else {
      for (int64_t j = i; j < n; ++j) y[j] = __float2bfloat16_rn(x[j]);
    }
  }
}

// The work in front of a GEMM call in one launch (a memset or a small kernel
// of its own is about 2 us of a call of 30): the call's header cleared, and
// part by part of the grid what the operands want.
constexpr int kPrepThreads = 256;

__device__ __forceinline__ void clear_words(uint32_t* p, int64_t n, int block, int blocks) {
  for (int64_t i = (int64_t)block * kPrepThreads + threadIdx.x; i < n; i += (int64_t)blocks * kPrepThreads) p[i] = 0u;
}

// Bt[d][c] = bf16(B[c][d]) (B is [C, D] row-major), 32 x 32 at a time through
// shared memory so that both sides are coalesced
__device__ void transpose_tiles(const float* __restrict__ B, __nv_bfloat16* __restrict__ Bt, int C, int D, int block,
                                int blocks) {
  __shared__ float t[32][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int ct = (C + 31) / 32;
  const int64_t tiles = (int64_t)ct * ((D + 31) / 32);
  for (int64_t k = block; k < tiles; k += blocks) {
    const int c0 = (int)(k % ct) * 32, d0 = (int)(k / ct) * 32;
    __syncthreads();
    for (int r = w; r < 32; r += kPrepThreads / 32)
      if (c0 + r < C && d0 + lane < D) t[r][lane] = B[(int64_t)(c0 + r) * D + d0 + lane];
    __syncthreads();
    for (int r = w; r < 32; r += kPrepThreads / 32)
      if (d0 + r < D && c0 + lane < C) Bt[(int64_t)(d0 + r) * C + c0 + lane] = __float2bfloat16_rn(t[lane][r]);
  }
}

// One warp per (q, c): Gt[q][c] = bf16(sum_d text[q][d] codebook[c][d]) with
// FP32 sums; the warps of c = 0 also write |text_q|.
__device__ void text_codebook(const float* __restrict__ text, const float* __restrict__ codebook, int Q, int C, int D,
                              __nv_bfloat16* __restrict__ Gt, float* __restrict__ tnorm, int block, int blocks) {
  const int lane = threadIdx.x & 31;
  for (int64_t w = ((int64_t)block * kPrepThreads + threadIdx.x) / 32; w < (int64_t)Q * C;
       w += (int64_t)blocks * kPrepThreads / 32) {
    const int qi = (int)(w / C), c = (int)(w - (int64_t)qi * C);
    float dot = 0.0f, sq = 0.0f;
    for (int d = lane; d < D; d += 32) {
      const float t = text[(int64_t)qi * D + d];
      dot = fmaf(t, codebook[(int64_t)c * D + d], dot);
      sq = fmaf(t, t, sq);
    }
    for (int off = 16; off > 0; off >>= 1) {
      dot += __shfl_xor_sync(0xffffffffu, dot, off);
      sq += __shfl_xor_sync(0xffffffffu, sq, off);
    }
    if (lane == 0) {
      Gt[w] = __float2bfloat16_rn(dot);
      if (c == 0) tnorm[qi] = sqrtf(sq);
    }
  }
}

// Blocks 0 .. tblocks - 1: the header and the transpose; the rest: the text
// product (Q > 0) or the cleared row norms.
__global__ void __launch_bounds__(kPrepThreads) decode_prep_kernel(GemmPrep p, int tblocks) {
  const int b = blockIdx.x;
  if (b < tblocks) {
    if (b == 0) clear_words((uint32_t*)p.hdr, sizeof(WsHeader) / 4, 0, 1);
    transpose_tiles(p.codebook, (__nv_bfloat16*)p.Bt, p.C, p.D, b, tblocks);
  } else if (p.Q > 0) {
    text_codebook(p.text, p.codebook, p.Q, p.C, p.D, (__nv_bfloat16*)p.Gt, p.tnorm, b - tblocks, gridDim.x - tblocks);
  } else {
    clear_words((uint32_t*)p.rownorm2, p.rows, b - tblocks, gridDim.x - tblocks);
  }
}

// One warp per text vector: its bf16 row and the row's norm; block 0 clears the header.
__global__ void __launch_bounds__(kPrepThreads) text_prep_kernel(WsHeader* hdr, const float* __restrict__ text, int Q,
                                                                 int D, __nv_bfloat16* __restrict__ tb,
                                                                 float* __restrict__ tnorm) {
  if (blockIdx.x == 0) clear_words((uint32_t*)hdr, sizeof(WsHeader) / 4, 0, 1);
  const int lane = threadIdx.x & 31;
  for (int64_t r = (blockIdx.x * (int64_t)kPrepThreads + threadIdx.x) / 32; r < Q; r += (int64_t)gridDim.x * kPrepThreads / 32) {
    float s = 0.0f;
    for (int d = lane; d < D; d += 32) {
      const __nv_bfloat16 h = __float2bfloat16_rn(text[r * D + d]);
      const float v = __bfloat162float(h);
      tb[r * D + d] = h;
      s += v * v;
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) tnorm[r] = sqrtf(s);
  }
}

// norms (or squared norms) of the rows of a bf16 [R, D] matrix
__global__ void row_norm_bf16_kernel(const __nv_bfloat16* __restrict__ X, int64_t R, int D, float* __restrict__ out,
                                     int squared) {
  const int lane = threadIdx.x & 31;
  for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32; r < R;
       r += (int64_t)gridDim.x * blockDim.x / 32) {
    float s = 0.0f;
    for (int d = lane; d < D; d += 32) {
      const float v = __bfloat162float(X[r * D + d]);
      s += v * v;
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) out[r] = squared ? s : sqrtf(s);
  }
}

int blocks_for(int64_t n, int per) {
  int64_t b = (n + per - 1) / per;
  if (b > num_sms() * 16) b = num_sms() * 16;
  return (int)(b > 0 ? b : 1);
}

}  // namespace

// FP32 rows.  Up to K = 128 the rows kernel is the faster one from the smallest
// call on (us, against conversion and GEMM: 100 x 64 -> 512 16 / 18, 20000 x
// 128 -> 256 20 / 22, 480000 x 128 -> 768 174 / 219).  Above that a call of a
// few waves spreads better over the other kernel's units (40000 x 256 -> 768
// 49 / 43, 78000 x 256 -> 512 53 / 59, 480000 x 256 -> 512 194 / 274).
bool gemm_takes_f32(int64_t M, int N, int K) {
  return N > RN && (K <= 2 * BK || (K <= kMaxSlabs * BK && M >= (int64_t)4 * BM * num_sms()));
}

// bf16 rows with the query unit: from four waves of 256 rows on (K = 256, N =
// 512, us: 78000 rows 59 / 57, 150000 75 / 80, 480000 178 / 198, 2073600 645 /
// 770; K = 64, 480000 rows 124 / 137).  Without it the column units of the
// other kernel are as fast (480000 rows 143 / 141) and need no whole blocks.
static bool query_takes_rows(int64_t M, int N, int K) {
  return N > RN && K <= kMaxSlabs * BK && M >= (int64_t)4 * 2 * BM * num_sms();
}

cudaError_t launch_gemm_bf16(const void* A, const void* Bt, const GemmEpi& ep, cudaStream_t st) {
  if (ep.M <= 0 || ep.N <= 0) return cudaSuccess;
  if (ep.a_f32)
    return !ep.sim_n && (ep.mode == kOutBF16 || ep.mode == kOutF32) && gemm_takes_f32(ep.M, ep.N, ep.K)
               ? launch_rows<false, true>(A, Bt, nullptr, ep, st)
               : cudaErrorInvalidValue;
  // bf16 output is read back from TMEM 64 columns at a time: BN >= 64 (the
  // columns past N are the zero fill of the Bt tile)
  if (ep.sim_n) return cudaErrorInvalidValue;  // launch_gemm_bf16_query
  if (ep.N <= 32 && ep.mode != kOutBF16) return launch_bn<32>(A, Bt, nullptr, ep, st);
  if (ep.N <= 64) return launch_bn<64>(A, Bt, nullptr, ep, st);
  if (ep.N <= 128) return launch_bn<128>(A, Bt, nullptr, ep, st);
  return launch_bn<256>(A, Bt, nullptr, ep, st);
}

cudaError_t launch_gemm_bf16_query(const void* A, const void* Bt, const void* Gt, const GemmEpi& ep,
                                   cudaStream_t st) {
  if (ep.M <= 0 || ep.N <= 0) return cudaSuccess;
  if (ep.mode != kOutBF16 || (ep.sim_n != 16 && ep.sim_n != 32) || !Gt || !ep.sim_out ||
      (ep.sim_mode != kOutCos && ep.sim_mode != kOutRel) || (ep.store && !ep.out))
    return cudaErrorInvalidValue;
  if (ep.a_f32)
    return gemm_takes_f32(ep.M, ep.N, ep.K) ? launch_rows<true, true>(A, Bt, Gt, ep, st) : cudaErrorInvalidValue;
  if (query_takes_rows(ep.M, ep.N, ep.K)) return launch_rows<true, false>(A, Bt, Gt, ep, st);
  if (ep.N <= 64) return launch_bn<64>(A, Bt, Gt, ep, st);
  if (ep.N <= 128) return launch_bn<128>(A, Bt, Gt, ep, st);
  return launch_bn<256>(A, Bt, Gt, ep, st);
}

cudaError_t launch_f32_to_bf16(const float* x, void* y, int64_t n, cudaStream_t st, WsHeader* hdr) {
  if (n <= 0) return cudaSuccess;
  f32_to_bf16_kernel<<<blocks_for(n / 4 + 1, 256), 256, 0, st>>>(x, (__nv_bfloat16*)y, n, hdr);
  g_launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_decode_prep(const GemmPrep& p, cudaStream_t st) {
  const int64_t tiles = (int64_t)((p.C + 31) / 32) * ((p.D + 31) / 32);
  const int tblocks = blocks_for(tiles, 1);
  const int more = p.Q > 0 ? blocks_for((int64_t)p.Q * p.C, kPrepThreads / 32)
                           : p.rownorm2 ? blocks_for(p.rows, 4 * kPrepThreads) : 0;
  decode_prep_kernel<<<tblocks + more, kPrepThreads, 0, st>>>(p, tblocks);
  g_launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_text_prep(WsHeader* hdr, const float* text, int Q, int D, void* tb, float* tnorm, cudaStream_t st) {
  text_prep_kernel<<<blocks_for(Q, kPrepThreads / 32), kPrepThreads, 0, st>>>(hdr, text, Q, D, (__nv_bfloat16*)tb, tnorm);
  g_launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_row_norm_bf16(const void* X, int64_t R, int D, float* out, int squared, cudaStream_t st) {
  if (R <= 0) return cudaSuccess;
  row_norm_bf16_kernel<<<blocks_for(R * 32, 256), 256, 0, st>>>((const __nv_bfloat16*)X, R, D, out, squared);
  g_launches += 1;
  return cudaGetLastError();
}

bool gemm_tma_available() { return encode_fn() != nullptr; }

// Runs small GEMMs whose producer issues no loads, one in each form of the two
// kernels (plain and with the query unit, bf16 and FP32 rows): the MMA and
// epilogue warps' bounded waits run out, the kernel records kStatTimeout and
// frees its TMEM, and the context stays usable.
int gemm_timeout_selftest(void* workspace, size_t ws_bytes, cudaStream_t st) {
  constexpr int M = 16, N = 144, K = 64, Q = 16;
  constexpr size_t kA = 256, kB = kA + (size_t)M * K * 4, kG = kB + (size_t)N * K * 2, kNorm = kG + (size_t)Q * K * 2,
                   kSim = kNorm + 256, kOut = kSim + (size_t)M * Q * 4, need = kOut + (size_t)M * N * 2;
  static_assert(need <= 49408, "the documented workspace");
  if (!workspace || ws_bytes < 49408 || ((uintptr_t)workspace & 255u)) return SCOUP_ERR_INVALID_ARG;
  char* w = (char*)workspace;
  GemmEpi ep;
  ep.M = M;
  ep.N = N;
  ep.K = K;
  ep.mode = kOutBF16;
  ep.out = w + kOut;
  ep.ldo = N;
  ep.rownorm2 = nullptr;
  ep.colnorm = (const float*)(w + kNorm);
  ep.status = (int*)w;
  ep.stall_loads = 1;
  GemmEpi eq = ep;
  eq.sim_n = Q;
  eq.sim_mode = kOutCos;
  eq.sim_out = w + kSim;
  eq.sim_ldo = Q;
  const void *A = w + kA, *B = w + kB, *G = w + kG;
  for (int form = 0; form < 5; ++form) {
    if (cudaMemsetAsync(w, 0, need, st) != cudaSuccess) return SCOUP_ERR_CUDA;
    const cudaError_t e = form == 0   ? launch_bn<256>(A, B, nullptr, ep, st)
                          : form == 1 ? launch_bn<256>(A, B, G, eq, st)
                          : form == 2 ? launch_rows<true, false>(A, B, G, eq, st)
                          : form == 3 ? launch_rows<false, true>(A, B, nullptr, ep, st)
                                      : launch_rows<true, true>(A, B, G, eq, st);
    int h = 0;
    if (e != cudaSuccess || cudaMemcpyAsync(&h, w, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return SCOUP_ERR_CUDA;
    if (!(h & kStatTimeout)) return SCOUP_OK;
  }
  return SCOUP_ERR_TIMEOUT;
}

}  // namespace scoup
