// LM head of larger calls on CTA pairs (bf16): guided logits written out, softmax partials per 128 codes.
//
// A pair of SMs works on one 256-code x 256-column tile (tcgen05.mma.cta_group::2, M = 256): each CTA stages its own 128
// codebook rows and HALF of the feature columns, and keeps the accumulators of its 128 codes.  With guidance the
// columns are up to 128 decision rows, conditional (staged by rank 0) then unconditional (rank 1); without, up to 256
// decision rows.  What bounds a one-CTA tile of this shape is the fill of shared memory from L2 (48 KB per k-block
// for 128 codes, against ~60 B per clock and SM); the pair needs 32 KB, 64 B per clock at the full tensor rate.  The
// accumulators are double-buffered (2 x 256 TMEM columns), so the epilogue of a tile runs under the next tile's MMAs.
// Pairs stay resident and walk (tile, pass) units, passes first: the pairs that share codebook rows read them at
// the same time and all but one find them in L2.
// Roles: warp 0 loads (both CTAs; bytes are counted on rank 0's barriers), warp 1 of rank 0 issues the MMAs, warps 4-19
// turn their 32 lanes' accumulators into logits and partials.  Four epilogue warps, one per scheduler, took 7 to 11 us a unit, more than
// the MMAs of a unit of d = 1280 and all of it in the open behind the last one.  Sixteen, and loads and MMAs issued by converged
// warps (a lone lane: 3 to 4 % more everywhere), epilogue and decisions, us: d 1280, 16384 codes, 16 images of 9 rows 35.1 -> 24.5; 20000
// codes, 40 images of 6 rows without guidance 67.9 -> 41.1; 4096 codes, 64 images 42.5 -> 29.5; d 2048, 8192 codes, 20 images of 11 rows
// 32.2 -> 26; 30000 codes, 12 images of 13 rows without guidance 58.3 -> 44; d 4096, 16384 codes, 32 images, 64 neighbours 87.6 -> 80.2; 65536
// codes, 64 images of 17 rows 921 -> 833 (the groups' tiles leave room for a third stage of 256 columns).
#include <math_constants.h>

#include "tc_common.cuh"
#include "vvs_internal.cuh"

namespace vvs {

using namespace tc;

namespace {

constexpr int kMaxStages = 6;
constexpr int kGroups = 4;            // of four epilogue warps, one per lane quarter of the tensor memory
constexpr int kThreads = 128 + kGroups * 128;
constexpr int kChunk = 16;            // decision rows per epilogue step of a group
constexpr int kTileBytes = kGroups * kChunk * 128 * 4;     // the groups' logit tiles
constexpr uint32_t kBlockK = 64;
constexpr uint32_t kABytes = 128 * kBlockK * 2;
// k-blocks per pipeline stage: a wait and a commit of the issuing warp per stage, and a k-block's four MMAs run 512 cycles at
// full width (chosen when a lone lane issued, which paid some 270 cycles for the two; one k-block a stage was not measured since)
constexpr uint32_t kSub = 2;

struct Params {
  int v, bt, n_cfg, nd, passes, units, kb_total, stages /* of kSub k-blocks */, n_tiles;    // nd: decision rows per pass (padded)
  uint32_t b_rows;                    // feature rows staged by a CTA
  float cfg_scale, inv_temp;
  float* part_m; float* part_s;       // [bt][n_tiles], tiles of 128 codes
  float* logits;                      // [bt][v]
  int32_t* status;
};

__device__ __forceinline__ void arrive_remote(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// bounded wait; gives up when another role of the CTA already did
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int32_t* status) {
  for (uint32_t i = 0; i < kSpinLimit; ++i) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((i & 1023u) == 1023u && *abort_flag) return false;
  }
  *abort_flag = 1;
  atomicOr(status, VVS_DEV_TIMEOUT);
  return false;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
lmhead_pair_kernel(const Params p, const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int rank = (int)(blockIdx.x & 1), pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
  const uint32_t b_bytes = p.b_rows * kBlockK * 2u, stage_bytes = kSub * (kABytes + b_bytes);
  float* sL = reinterpret_cast<float*>(smem + (size_t)p.stages * stage_bytes);      // [kGroups][kChunk][128]

  if (tid == 0) {
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(&full_bar[i], 1);
      mbar_init(&empty_bar[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], 8 * kGroups);      // the epilogue warps of both CTAs
    }
    s_abort = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tm_a);
    tma_prefetch_desc(&tm_b);
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_sync();                             // both CTAs' barriers are ready
  const uint32_t tmem = tmem_slot;
  pdl_launch_dependents();

  if (warp == 0) {
    // ---- TMA producer, a converged warp of which one lane issues (codebook rows of the first stages may be requested before the
    // features exist) ---------------------------------------------------------------------------------------------------
    uint32_t stage = 0, par = 1;
    int issued = 0;
    bool ok = true;
    auto load_a = [&](uint32_t i, int kb, int y) {
      if (elect_one()) {
        const uint32_t bar0 = mapa(smem_u32(&full_bar[i]), 0);
        uint8_t* st = smem + (size_t)i * stage_bytes;
        if (rank == 0) mbar_expect_tx(&full_bar[i], 2 * stage_bytes);
#pragma unroll
        for (uint32_t h = 0; h < kSub; ++h) tma_load_pair_2d(st + h * kABytes, &tm_a, bar0, (kb * (int)kSub + (int)h) * (int)kBlockK, y);
      }
    };
    auto load_b = [&](uint32_t i, int kb, int y) {
      if (elect_one()) {
        const uint32_t bar0 = mapa(smem_u32(&full_bar[i]), 0);
        uint8_t* st = smem + (size_t)i * stage_bytes + kSub * kABytes;
#pragma unroll
        for (uint32_t h = 0; h < kSub; ++h) tma_load_pair_2d(st + h * b_bytes, &tm_b, bar0, (kb * (int)kSub + (int)h) * (int)kBlockK, y);
      }
    };
    const int n_pre = p.kb_total < p.stages ? p.kb_total : p.stages;
    for (int u = pair; u < p.units && ok; u += n_pairs) {
      const int tile = u / p.passes, row0 = (u - tile * p.passes) * p.nd;
      const int ya = tile * 256 + rank * 128;
      const int yb = p.n_cfg == 2 ? rank * p.bt + row0 : row0 + rank * (int)p.b_rows;
      const int done = u == pair ? n_pre : 0;       // codebook blocks requested already
      if (done) {
        for (int i = 0; i < n_pre; ++i) load_a(i, i, ya);
        pdl_wait();
      }
      for (int kb = 0; kb < p.kb_total; ++kb) {
        if (kb >= done) {
          if (!(ok = __all_sync(0xffffffffu, wait_or_abort(&empty_bar[stage], par, &s_abort, p.status)))) break;
          load_a(stage, kb, ya);
        }
        load_b(stage, kb, yb);
        ++issued;
        if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1u; }
      }
    }
    if (!ok && rank == 0) {                       // gave up: nothing may be in flight when the pair leaves (bounded)
      for (int i = issued > p.stages ? issued - p.stages : 0; i < issued; ++i)
        for (uint32_t k = 0; k < kSpinLimit && !mbar_try_wait_cluster(&full_bar[i % p.stages], (i / p.stages) & 1); ++k) {}
    }
  } else if (warp == 1 && rank == 0) {
    // ---- MMA issuer --------------------------------------------------------------------------------------------------
    const uint32_t n_cols = p.n_cfg == 2 ? 2u * (uint32_t)p.nd : (uint32_t)p.nd;
    const uint32_t idesc = idesc_bf16_f32(256, n_cols);
    const uint32_t lo0 = desc_lo_sw128(smem_u32(smem)), stage_lo = stage_bytes >> 4;
    uint32_t stage = 0, par = 0;
    int it = 0, issued = 0;
    bool ok = true;
    for (int u = pair; u < p.units && ok; u += n_pairs, ++it) {
      const uint32_t buf = it & 1, d = tmem + buf * 256u;
      if (!(ok = __all_sync(0xffffffffu, wait_or_abort(&acc_empty[buf], ((it >> 1) & 1) ^ 1, &s_abort, p.status)))) break;
      tc_fence_after();
      for (int kb = 0; kb < p.kb_total; ++kb) {
        if (!(ok = __all_sync(0xffffffffu, wait_or_abort(&full_bar[stage], par, &s_abort, p.status)))) break;
        tc_fence_after();
        const uint32_t a_lo = lo0 + stage * stage_lo;
#pragma unroll
        for (uint32_t h = 0; h < kSub; ++h)
          mma_pair_k64(d, a_lo + h * (kABytes >> 4), a_lo + ((kSub * kABytes + h * b_bytes) >> 4), idesc, kb > 0 || h > 0);
        commit_pair(&empty_bar[stage]);
        ++issued;
        if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1u; }
      }
      if (ok) commit_pair(&acc_full[buf]);        // (half an accumulator is nobody's)
    }
    if (!ok && issued > 0) {                      // gave up: the MMAs issued so far end before the pair leaves (bounded)
      const int i = issued - 1;
      for (uint32_t k = 0; k < kSpinLimit && !mbar_try_wait_cluster(&empty_bar[i % p.stages], (i / p.stages) & 1); ++k) {}
    }
  } else if (warp >= 4) {
    // ---- epilogue: a group takes every fourth chunk of 16 decision rows; thread = one code, logits out and to the group's tile
    // (codes of row r at code ^ 8 (r & 3): no two threads on a bank in either direction), then eight threads per row for the partials
    const int grp = (warp - 4) >> 2, q = warp & 3, e = q * 32 + lane;
    const uint32_t t_lane = (uint32_t)(q * 32) << 16;
    const uint32_t empty0 = mapa(smem_u32(&acc_empty[0]), 0), empty1 = mapa(smem_u32(&acc_empty[1]), 0);
    float* tile_s = sL + grp * (kChunk * 128);
    const int prow = e >> 3, part = e & 7;
    const unsigned mates = 0xffu << (lane & 24);
    int it = 0;
    pdl_wait();
    for (int u = pair; u < p.units; u += n_pairs, ++it) {
      const int tile = u / p.passes, row0 = (u - tile * p.passes) * p.nd, buf = it & 1;
      const int nd = min(p.nd, p.bt - row0);
      const int n = tile * 256 + rank * 128 + e, t128 = tile * 2 + rank;
      const bool n_ok = n < p.v;
      // (a thread that saw another role's abort in time may be beside one that saw the accumulator: the group leaves or stays as one,
      // since it meets at barriers below)
      if (!named_bar_all(1 + grp, 128, wait_or_abort(&acc_full[buf], (it >> 1) & 1, &s_abort, p.status))) break;
      tc_fence_after();
      const uint32_t t_row = tmem + (uint32_t)buf * 256u + t_lane;
      auto release = [&]() {                      // the accumulator has been read: the next unit but one may have it
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_remote(buf ? empty1 : empty0);
      };
      if (grp * kChunk >= nd) release();
      for (int c0 = grp * kChunk; c0 < nd; c0 += kGroups * kChunk) {
        const int rows = min(kChunk, nd - c0);
        float l[16];
        tmem_ld16(t_row + c0, l);
        if (p.n_cfg == 2) {
          float lu[16];
          tmem_ld16(t_row + (uint32_t)p.nd + c0, lu);
#pragma unroll
          for (int j = 0; j < 16; ++j) l[j] = lu[j] + p.cfg_scale * (l[j] - lu[j]);
        }
        if (c0 + kGroups * kChunk >= nd) release();
        float* dst = p.logits + (size_t)(row0 + c0) * p.v + n;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          l[j] *= p.inv_temp;
          tile_s[j * 128 + (e ^ (8 * (j & 3)))] = n_ok ? l[j] : -CUDART_INF_F;
          if (n_ok && j < rows) *dst = l[j];
          dst += p.v;
        }
        named_bar_sync(1 + grp, 128);
        if (t128 < p.n_tiles && prow < rows) {
          const float* row = tile_s + prow * 128;
          float x[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) x[i] = row[(part + 8 * i) ^ (8 * (prow & 3))];
          float mx = x[0];
#pragma unroll
          for (int i = 1; i < 16; ++i) mx = fmaxf(mx, x[i]);
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(mates, mx, o));
          float sum = 0.f;
          if (mx > -CUDART_INF_F) {
#pragma unroll
            for (int i = 0; i < 16; ++i) sum += expf(x[i] - mx);
          }
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) sum += __shfl_xor_sync(mates, sum, o);
          if (part == 0) {
            const size_t at = (size_t)(row0 + c0 + prow) * p.n_tiles + t128;
            p.part_m[at] = mx;
            p.part_s[at] = sum;
          }
        }
        named_bar_sync(1 + grp, 128);             // the tile is written again
      }
    }
  }
  __syncwarp();
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  cluster_sync();                             // no CTA leaves while the pair's MMAs or signals may still reach it
  tc_fence_after();
  if (warp == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

int pass_rows(int bt, int n_cfg, int* passes) {
  const int most = n_cfg == 2 ? 128 : 256, step = n_cfg == 2 ? 16 : 32;
  const int n = (bt + most - 1) / most, per = (bt + n - 1) / n;
  const int nd = (per + step - 1) / step * step;
  *passes = (bt + nd - 1) / nd;
  return nd;
}

}  // namespace

bool lmhead_pair_applicable(const LmHeadArgs& a) {
  return !a.row_mode && a.n_draft_max == 0 && a.logits_out && a.bt * a.n_cfg > 96;
}

int lmhead_pair_box_rows(int bt, int n_cfg) {
  int passes;
  const int nd = pass_rows(bt, n_cfg, &passes);
  return n_cfg == 2 ? nd : nd / 2;
}

int launch_lmhead_pair(const LmHeadArgs& a, cudaStream_t s) {
  Params p{};
  p.v = a.v; p.bt = a.bt; p.n_cfg = a.n_cfg; p.nd = pass_rows(a.bt, a.n_cfg, &p.passes);
  p.n_tiles = (a.v + 127) / 128;
  p.units = (a.v + 255) / 256 * p.passes;
  p.kb_total = (a.k + (int)(kSub * kBlockK) - 1) / (int)(kSub * kBlockK);
  p.b_rows = (uint32_t)lmhead_pair_box_rows(a.bt, a.n_cfg);
  p.cfg_scale = a.cfg_scale; p.inv_temp = a.inv_temp; p.part_m = a.part_m; p.part_s = a.part_s; p.logits = a.logits_out;
  p.status = a.status;
  const int stage_bytes = (int)(kSub * (kABytes + p.b_rows * kBlockK * 2));
  p.stages = (224 * 1024 - kTileBytes) / stage_bytes;
  if (p.stages > kMaxStages) p.stages = kMaxStages;
  if (ensure_dynamic_smem(reinterpret_cast<const void*>(lmhead_pair_kernel), 225 * 1024) != cudaSuccess) return VVS_ERR_CUDA;
  // (all of the SM's shared memory: the two CTAs of a pair wait for each other, so neither may find its tensor memory
  // held by a CTA of another stream's kernel that waits in the same way)
  int pairs = a.n_sms / 2;
  if (pairs > p.units) pairs = p.units;
  return launch_kernel(lmhead_pair_kernel, dim3(2 * pairs), dim3(kThreads), (size_t)225 * 1024, a.pdl,
                       s, p, *a.tm_a, *a.tm_b) == cudaSuccess ? VVS_OK : VVS_ERR_CUDA;
}

}  // namespace vvs
