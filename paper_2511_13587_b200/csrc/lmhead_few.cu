// LM head of a call with few feature rows (at most kMaxCols, decision rows x guidance halves): one CTA per 128 codebook
// rows, every feature row on the MMA's N side, guided logits written out and the tile's softmax partial (max, sum exp) of
// every decision row taken from registers.
//
// What bounds it: the stream of codebook rows, if nothing else gets in its way.  Two warps issue, every other k-block each with
// an accumulator of its own (one issuing lane in a branch of its own reached a k-block every ~600 cycles, which is slower than
// the stream fills a stage; issuing by converged warps moved a call of one image and 16384 codes no further than its runs
// differ); nor is the loading lane alone: with its ring's 600 cycles a k-block d 4096, 4096 or 8192 codes took 27 to 28 us a call of one image, decision included, 20 as a converged warp
// (d 2048, 9472 codes 19.9 -> 17.8; d 1280, 8192 codes 16.1 -> 14.8); the pipeline is as deep as shared memory allows and its weights are
// requested before griddepcontrol.wait.  Up to one tile per SM a CTA takes the whole SM's shared memory; with more, two
// CTAs share an SM so that one's epilogue runs under the other's stream.  With one issuer and a thread per decision row
// summing 128 values from shared memory (2.1 us) a call of one image and 16384 codes took 21.8 us, decision included; 15.3
// with this kernel.
#include <math_constants.h>

#include "tc_common.cuh"
#include "vvs_internal.cuh"

namespace vvs {

using namespace tc;

namespace {

constexpr int kMaxCols = 96;           // feature rows
constexpr int kMaxStages = 12;
constexpr int kThreads = 256;
constexpr uint32_t kTileRows = 128;
constexpr uint32_t kBlockK = 64;
constexpr uint32_t kATileBytes = kTileRows * kBlockK * 2;

struct Params {
  int v, bt, n_cfg, nd_pad, kb_total, stages, n_tiles;
  uint32_t tmem_cols;
  float cfg_scale, inv_temp;
  float* part_m; float* part_s;         // [bt][n_tiles]
  float* logits;                        // [bt][v]
  int32_t* status;
};


__global__ void __launch_bounds__(kThreads, 2)
lmhead_few_kernel(const Params p, const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages];
  __shared__ __align__(8) uint64_t empty_bar[kMaxStages];
  __shared__ __align__(8) uint64_t acc_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;
  __shared__ float s_m[4][kMaxCols], s_s[4][kMaxCols];    // partials of the tile's four groups of 32 codes

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int tile = blockIdx.x, C = p.n_cfg, nt = p.nd_pad * C;
  const uint32_t half_bytes = (uint32_t)p.nd_pad * kBlockK * 2u, stage_bytes = kATileBytes + half_bytes * (uint32_t)C;

  if (tid == 0) {
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(&full_bar[i], 1);
      mbar_init(&empty_bar[i], 1);
    }
    mbar_init(&acc_bar, 2);               // two issuing threads
    s_abort = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tm_a);
    tma_prefetch_desc(&tm_b);
  }
  if (warp == 1) {
    tmem_alloc(&tmem_slot, p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  pdl_launch_dependents();

  const int n_pre = p.kb_total < p.stages ? p.kb_total : p.stages;
  // loads by one lane of a converged warp (mma_bf16_k64)
  auto load_a = [&](int i, uint32_t stage) {
    if (elect_one()) {
      mbar_expect_tx(&full_bar[stage], stage_bytes);
      tma_load_2d(smem + (size_t)stage * stage_bytes, &tm_a, &full_bar[stage], i * (int)kBlockK, tile * (int)kTileRows);
    }
  };
  auto load_b = [&](int i, uint32_t stage, int half) {
    if (elect_one())
      tma_load_2d(smem + (size_t)stage * stage_bytes + kATileBytes + (half ? half_bytes : 0u), &tm_b, &full_bar[stage], i * (int)kBlockK,
                  half ? p.bt : 0);
  };
  if (warp == 0) {
    // ---- TMA producer: the weights of the free stages go out before the wait ------------------------------
    for (int i = 0; i < n_pre; ++i) load_a(i, i);
    pdl_wait();
    for (int i = 0; i < n_pre; ++i) load_b(i, i, 0);
    uint32_t stage = 0, par = 0;
    for (int i = n_pre; i < p.kb_total; ++i) {
      if (!__all_sync(0xffffffffu, wait_or_abort(&empty_bar[stage], par, &s_abort))) {
        if (lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
        s_abort = 1;
        break;
      }
      load_a(i, stage);
      load_b(i, stage, 0);
      if (C == 2) load_b(i, stage, 1);
      if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1; }
    }
  } else if (warp == 3) {
    // the unconditional feature rows of the first stages, beside the producer's conditional ones
    if (C == 2) {
      pdl_wait();
      for (int i = 0; i < n_pre; ++i) load_b(i, i, 1);
    }
  } else if (warp == 1 || warp == 2) {
    // ---- MMA issuers: every other k-block each; the number of stages is even, or they are all used once, so that a
    // stage always belongs to the same one ---------------------------------------------------------------------
    const int me = __shfl_sync(0xffffffffu, warp, 0) - 1;
    const uint32_t idesc = idesc_bf16_f32(kTileRows, (uint32_t)nt), d = tmem + (uint32_t)(me * nt);
    const uint32_t lo0 = desc_lo_sw128(smem_u32(smem)), stage_lo = stage_bytes >> 4;
    uint32_t stage = (uint32_t)me, par = 0, add = 0;
    for (int i = me; i < p.kb_total; i += 2) {
      if (!__all_sync(0xffffffffu, wait_or_abort(&full_bar[stage], par, &s_abort))) {
        if (lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
        s_abort = 1;
        break;
      }
      tc_fence_after();
      const uint32_t a_lo = lo0 + stage * stage_lo;
      mma_bf16_k64(d, a_lo, a_lo + (kATileBytes >> 4), idesc, add);
      add = 1;
      if (i + p.stages < p.kb_total) mma_commit_elect(&empty_bar[stage]);
      stage += 2;
      if (stage >= (uint32_t)p.stages) { stage -= p.stages; par ^= 1; }
    }
    mma_commit_elect(&acc_bar);
  }
  __syncwarp();
  pdl_wait();
  const bool got = wait_or_abort(&acc_bar, 0, &s_abort);
  if (!got) s_abort = 1;
  if (__syncthreads_or(got ? 0 : 1)) {
    if (tid == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
  } else {
    tc_fence_after();
    // ---- epilogue: thread = code, sixteen decision rows at a time --------------------------------------------------
    const int group = warp & 3, n = tile * (int)kTileRows + group * 32 + lane;
    const bool n_ok = n < p.v, two = p.kb_total > 1;
    const uint32_t t_row = tmem + ((uint32_t)(group * 32) << 16);
    for (int c0 = (warp >> 2) * 16; c0 < p.bt; c0 += 32) {
      float l[16], t[16];
      tmem_ld16(t_row + (uint32_t)c0, l);
      if (two) {
        tmem_ld16(t_row + (uint32_t)(nt + c0), t);
#pragma unroll
        for (int j = 0; j < 16; ++j) l[j] += t[j];
      }
      if (C == 2) {
        float u[16];
        tmem_ld16(t_row + (uint32_t)(p.nd_pad + c0), u);
        if (two) {
          tmem_ld16(t_row + (uint32_t)(nt + p.nd_pad + c0), t);
#pragma unroll
          for (int j = 0; j < 16; ++j) u[j] += t[j];
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) l[j] = u[j] + p.cfg_scale * (l[j] - u[j]);
      }
      float mx[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        l[j] *= p.inv_temp;
        if (n_ok && c0 + j < p.bt) p.logits[(size_t)(c0 + j) * p.v + n] = l[j];
        if (!n_ok) l[j] = -CUDART_INF_F;
        asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(mx[j]) : "f"(l[j]));
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) l[j] = mx[j] > -CUDART_INF_F ? expf(l[j] - mx[j]) : 0.f;
      warp_sums(l, lane);
      const int j0 = warp_sums_index<16>(lane);
      float m0 = mx[0];
#pragma unroll
      for (int j = 1; j < 16; ++j) m0 = j == j0 ? mx[j] : m0;
      if (!(lane & 1) && c0 + j0 < p.bt) {
        s_m[group][c0 + j0] = m0;
        s_s[group][c0 + j0] = l[0];
      }
    }
    __syncthreads();
    if (tid < p.bt) {
      const float a = s_m[0][tid], b = s_m[1][tid], c = s_m[2][tid], e = s_m[3][tid];
      const float m = fmaxf(fmaxf(a, b), fmaxf(c, e));
      float s = 0.f;
      if (m > -CUDART_INF_F)
        s = s_s[0][tid] * expf(a - m) + s_s[1][tid] * expf(b - m) + s_s[2][tid] * expf(c - m) + s_s[3][tid] * expf(e - m);
      p.part_m[(size_t)tid * p.n_tiles + tile] = m;
      p.part_s[(size_t)tid * p.n_tiles + tile] = s;
    }
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, p.tmem_cols);
}

}  // namespace

// (96: above it the pair kernel, which reads a feature tile once for 256 codes, is the faster one)
bool lmhead_few_applicable(const LmHeadArgs& a) {
  return !a.row_mode && a.n_draft_max == 0 && a.logits_out && (a.bt + 15) / 16 * 16 * a.n_cfg <= kMaxCols;
}

int launch_lmhead_few(const LmHeadArgs& a, cudaStream_t s) {
  Params p{};
  p.v = a.v; p.bt = a.bt; p.n_cfg = a.n_cfg; p.nd_pad = lmhead_box_rows(a.bt); p.n_tiles = (a.v + 127) / 128;
  p.kb_total = (a.k + (int)kBlockK - 1) / (int)kBlockK;
  p.cfg_scale = a.cfg_scale; p.inv_temp = a.inv_temp; p.part_m = a.part_m; p.part_s = a.part_s; p.logits = a.logits_out;
  p.status = a.status;
  const int nt = p.nd_pad * a.n_cfg, stage_bytes = (int)kATileBytes + nt * (int)kBlockK * 2;
  const int n_sms = a.n_sms > 0 ? a.n_sms : 148, budget = (p.n_tiles <= n_sms ? 220 : 106) * 1024;
  p.stages = budget / stage_bytes;
  if (p.stages > kMaxStages) p.stages = kMaxStages;
  if (p.stages >= p.kb_total) p.stages = p.kb_total;
  else p.stages &= ~1;                    // a stage that is used again always belongs to the same issuer
  uint32_t cols = 32;
  while (cols < 2u * (uint32_t)nt) cols <<= 1;
  p.tmem_cols = cols;
  if (ensure_dynamic_smem(reinterpret_cast<const void*>(lmhead_few_kernel), 221 * 1024) != cudaSuccess) return VVS_ERR_CUDA;
  return launch_kernel(lmhead_few_kernel, dim3(p.n_tiles), dim3(kThreads), (size_t)p.stages * stage_bytes + 1024, a.pdl, s, p, *a.tm_a,
                       *a.tm_b) == cudaSuccess ? VVS_OK : VVS_ERR_CUDA;
}

}  // namespace vvs
