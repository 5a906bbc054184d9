// Gate/up projection of calls with many tokens on CTA pairs (bf16 contexts of wide models whose weights stay in L2): proj_tc.cu's unsplit
// operation, the same sums and order, bit for bit.
//
// What bounds it there is the fill of shared memory from L2 (55 bytes a clock and SM): a CTA stages 128 rows of both matrices and all tokens of
// its pass.  A pair (tcgen05.mma.cta_group::2, M = 256) stages half of the tokens per CTA, and gate and up lie in one tile, row by row in
// turns, 64 outputs a CTA.  XL shape, 216 tokens: 440 KB a CTA in the place of 760.
// A stage is two k-blocks where five such stages fit (passes of up to 96 tokens), else one: four stages of two are too coarse for the way from
// a stage's last MMA to the loads that fill it again (18 layers of the XL shape, two / one: 108 tokens 585.8 / 595.4 us, 144 623.0 / 626.2, 180 660.1 /
// 662.4; 198 711.4 / 705.5, 252 835.8 / 830.9, 288 880.8 / 879.6).
// 18 layers of the XL shape, proj_tc.cu / this kernel (us): 108 tokens 604.0 / 587.3, 126 616.6 / 598.4, 144 640.2 / 624.3, 180 670.9 / 659.8, 216 802.6
// / 789.3, 252 856.6 / 831.5, 288 896.3 / 879.8.  Passes of more than 160 tokens lose in the epilogue what they gain in the fill (of 192: 360 tokens
// 957.8 / 949.5, 378 961.6 / 966.3, 14 sequences of 27 rows 876.7 / 887.3; of 224: 396 tokens 974.4 / 991.5), and QKV on pairs gains nothing (144 tokens
// 637.8 / 636.9, 288 896 / 912): those stay in proj_tc.cu.  Other widths, and up to how many tokens a pass each may have: plan_gateup_pair.
#include "tc_common.cuh"
#include "vvs_internal.cuh"

namespace vvs {

using namespace tc;
using namespace proj;

namespace {

constexpr int kThreads = 512;

struct Params {
  int m, nt, kb_total, stages, up_first;                          // nt: tokens of a pass; kb_total: stages' worth of k-blocks (SUB each)
  uint32_t tmem_cols;
  int32_t* status;
  const float* ss_in; int ss_parts; float inv_d, eps;
  __nv_bfloat16* act; int ff;
  const uint8_t* ahead[2]; uint32_t ahead_bytes; AheadShare share;
};

template <int SUB>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
gateup_pair_kernel(const __grid_constant__ Params p, const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], acc_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;
  __shared__ float s_rs[kPairTok];

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int rank = (int)(blockIdx.x & 1), tile = (int)blockIdx.x, pass = (int)blockIdx.y;          // tile: of this CTA's rows
  const int tok0 = pass * p.nt, ntok = min(p.nt, p.m - tok0);
  const uint32_t b_bytes = (uint32_t)p.nt * kBlockK, stage_bytes = SUB * (kATileBytes + b_bytes);  // (half of the tokens)

  if (tid == 0) {
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(&full_bar[i], 1);
      mbar_init(&empty_bar[i], 1);
    }
    mbar_init(&acc_bar, 1);
    s_abort = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tm_a);
    tma_prefetch_desc(&tm_b);
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(p.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_sync();                             // both CTAs' barriers are ready
  const uint32_t tmem = tmem_slot;
  pdl_launch_dependents();

  if (warp == kThreads / 32 - 1 && p.ahead_bytes > 0) {
    // This CTA's share of a later projection's weights, HBM -> L2 (proj_tc.cu has the measurements)
    const uint32_t begin = (blockIdx.y * gridDim.x + blockIdx.x) * p.share.every, end = min(begin + p.share.bytes, p.ahead_bytes);
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (p.ahead[i])
        for (uint32_t at = begin + lane * 4096u; at < end; at += 32 * 4096u) prefetch_l2(p.ahead[i] + at, min(4096u, end - at));
  }
  if (warp == 0) {
    // ---- TMA producer: weights of the first stages before the wait ---------------------------------------------------
    auto load_w = [&](uint32_t stage, int kb) {
      if (elect_one()) {
        const uint32_t bar0 = mapa(smem_u32(&full_bar[stage]), 0);
        uint8_t* st = smem + (size_t)stage * stage_bytes;
        if (rank == 0) mbar_expect_tx(&full_bar[stage], 2 * stage_bytes);
#pragma unroll
        for (int h = 0; h < SUB; ++h) tma_load_pair_4d(st + h * kATileBytes, &tm_a, bar0, 0, 0, tile * 64, kb * SUB + h);
      }
    };
    auto load_act = [&](uint32_t stage, int kb) {
      if (elect_one()) {
        const uint32_t bar0 = mapa(smem_u32(&full_bar[stage]), 0);
        uint8_t* st = smem + (size_t)stage * stage_bytes + SUB * kATileBytes;
#pragma unroll
        for (int h = 0; h < SUB; ++h)
          tma_load_pair_2d(st + h * b_bytes, &tm_b, bar0, (kb * SUB + h) * (int)kBlockK, tok0 + rank * (p.nt >> 1));
      }
    };
    const int n_pre = min(p.kb_total, p.stages);
    for (int i = 0; i < n_pre; ++i) load_w(i, i);
    pdl_wait();
    for (int i = 0; i < n_pre; ++i) load_act(i, i);
    uint32_t stage = 0, par = 0;                  // stage of block i, parity of its previous release
    int issued = n_pre;
    bool ok = true;
    for (int i = n_pre; i < p.kb_total; ++i, ++issued) {
      if (!(ok = __all_sync(0xffffffffu, wait_or_abort(&empty_bar[stage], par, &s_abort)))) break;
      load_w(stage, i);
      load_act(stage, i);
      if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1; }
    }
    if (!ok) {
      if (lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
      s_abort = 1;
      if (rank == 0)                              // nothing may be in flight when the pair leaves (bounded)
        for (int i = issued > p.stages ? issued - p.stages : 0; i < issued; ++i)
          for (uint32_t k = 0; k < kSpinLimit && !mbar_try_wait_cluster(&full_bar[i % p.stages], (i / p.stages) & 1); ++k) {}
    }
  } else if (warp == 1 && rank == 0) {
    // ---- MMA issuer of the pair (a wait that ran out is reported and the loop goes on over what is there) -------------------
    const uint32_t idesc = idesc_bf16_f32(256, (uint32_t)p.nt), lo0 = desc_lo_sw128(smem_u32(smem)), stage_lo = stage_bytes >> 4;
    uint32_t stage = 0, par = 0;
    for (int i = 0; i < p.kb_total; ++i) {
      bool got = false;
      for (uint32_t k = 0; k < kSpinLimit && !got; ++k) got = mbar_try_wait_cluster(&full_bar[stage], par) || ((k & 1023u) == 1023u && s_abort);
      if (!got) {
        atomicOr(p.status, VVS_DEV_TIMEOUT);
        s_abort = 1;
      }
      __syncwarp();
      tc_fence_after();
      const uint32_t a_lo = lo0 + stage * stage_lo;
#pragma unroll
      for (int h = 0; h < SUB; ++h)
        mma_pair_k64(tmem, a_lo + h * (kATileBytes >> 4), a_lo + ((SUB * kATileBytes + h * b_bytes) >> 4), idesc, (uint32_t)(i | h));
      commit_pair(&empty_bar[stage]);
      if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1; }
    }
    commit_pair(&acc_bar);
  }
  __syncwarp();
  pdl_wait();

  // ---- 1/rms of the pass's tokens, while the MMAs run: eight tokens' loads in flight per warp ---------------------------
  if (warp >= 3) {
    const int n4 = p.ss_parts >> 2;
    for (int t0 = (warp - 3) * 8; t0 < ntok; t0 += 8 * (kThreads / 32 - 3)) {
      float ss[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      for (int i = lane; i < n4; i += 32) {
        float4 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
          v[j] = __ldcg(reinterpret_cast<const float4*>(p.ss_in + (size_t)(tok0 + min(t0 + j, ntok - 1)) * p.ss_parts) + i);
#pragma unroll
        for (int j = 0; j < 8; ++j) ss[j] += (v[j].x + v[j].y) + (v[j].z + v[j].w);
      }
      warp_sums(ss, lane);
      const int j = warp_sums_index<8>(lane);
      if ((lane & 3) == 0 && t0 + j < kPairTok) s_rs[t0 + j] = rsqrtf(ss[0] * p.inv_d + p.eps);
    }
  }
  const int row_t = (warp & 3) * 32 + lane;   // weight row of this thread in TMEM
  const bool odd = lane & 1, second = lane & 2;
  {
    bool got = false;
    for (uint32_t k = 0; k < kSpinLimit && !got; ++k) got = mbar_try_wait_cluster(&acc_bar, 0) || ((k & 1023u) == 1023u && s_abort);
    if (!got) {
      if (lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
      s_abort = 1;
    }
  }
  tc_fence_after();
  __syncthreads();                            // s_rs
  // ---- epilogue from TMEM, sixteen tokens at a time, to a token-major tile over the stages, which have drained ------------------
  const uint32_t t_row = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  constexpr int kOutLd = 144;                 // bytes per token: 64 outputs and a pad
#pragma unroll 1
  for (int c0 = (warp >> 2) * 16; c0 < ntok; c0 += kThreads / 8) {
    float y[16];
    tmem_ld16(t_row + (uint32_t)c0, y);
#pragma unroll
    for (int j = 0; j < 16; ++j) y[j] *= s_rs[c0 + j];
    // lane pairs: the even lane goes on with tokens 0-7, the odd one with tokens 8-15; lo and hi are their even and odd row
    float lo[8], hi[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float got = __shfl_xor_sync(0xffffffffu, odd ? y[j] : y[8 + j], 1);
      lo[j] = odd ? got : y[j];
      hi[j] = odd ? y[8 + j] : got;
    }
    float a[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float gate = p.up_first ? hi[j] : lo[j], up = p.up_first ? lo[j] : hi[j];
      a[j] = __fdividef(gate, 1.f + expf(-gate)) * up;
    }
    // neighbouring outputs are two lanes apart: four of the eight tokens each
    uint8_t* out = smem + (size_t)(c0 + (odd ? 8 : 0) + (second ? 4 : 0)) * kOutLd + (row_t >> 2) * 4;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float got = __shfl_xor_sync(0xffffffffu, second ? a[j] : a[4 + j], 2);
      *reinterpret_cast<uint32_t*>(out + j * kOutLd) = second ? pack_bf16(got, a[4 + j]) : pack_bf16(a[j], got);
    }
  }
  tc_fence_before();
  __syncthreads();
  // ---- 16-byte pieces: eight outputs of a token -----------------------------------------------------------------------------
  const int n8 = tile * 64 + (tid & 7) * 8;
  if (n8 < p.ff) {
#pragma unroll 4
    for (int t = tid >> 3; t < ntok; t += kThreads / 8)
      *reinterpret_cast<uint4*>(p.act + (size_t)(tok0 + t) * p.ff + n8) = *reinterpret_cast<const uint4*>(smem + (size_t)t * kOutLd + (tid & 7) * 16);
  }
  __syncwarp();
  cluster_sync();                             // no CTA leaves while the pair's MMAs or signals may still reach it
  tc_fence_after();
  if (warp == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
}

}  // namespace

int launch_gateup_pair(const GateupPairPlan& pl, const ProjArgs& g, cudaStream_t s) {
  Params kp{};
  kp.m = g.m; kp.nt = pl.nt; kp.kb_total = pl.kb_total; kp.stages = pl.stages; kp.up_first = g.up_first ? 1 : 0;
  kp.tmem_cols = (uint32_t)pl.tmem_cols; kp.status = g.status;
  kp.ss_in = g.ss_in; kp.ss_parts = g.ss_parts; kp.inv_d = 1.f / (float)g.d; kp.eps = g.eps; kp.act = g.act; kp.ff = g.ff;
  kp.ahead[0] = static_cast<const uint8_t*>(g.ahead[0]); kp.ahead[1] = static_cast<const uint8_t*>(g.ahead[1]);
  kp.ahead_bytes = g.ahead[0] ? g.ahead_bytes : 0;
  kp.share = ahead_share(kp.ahead_bytes, (uint32_t)(2 * pl.pairs * pl.passes));
  auto* fn = pl.sub == 2 ? gateup_pair_kernel<2> : gateup_pair_kernel<1>;
  if (ensure_dynamic_smem(reinterpret_cast<const void*>(fn), 222 * 1024) != cudaSuccess) return VVS_ERR_CUDA;
  return launch_kernel(fn, dim3(2 * pl.pairs, pl.passes), dim3(kThreads), (size_t)pl.smem_bytes, g.pdl, s, kp, *g.tm_a, *g.tm_b) == cudaSuccess
                 ? VVS_OK : VVS_ERR_CUDA;
}

}  // namespace vvs
