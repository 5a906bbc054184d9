// Weight-streaming projections of calls with few tokens (bf16 contexts of wide models): the same operations as proj_tc.cu on
// tiles of 64 weight rows.  Of models whose weights do not stay in L2 it gives the same bits too (APART below; which projections
// these are and what it gives: plan_proj_few, launch_plans.h).
//
// What bounds such a projection is the chain of one CTA: wait for the kernel before, activations from L2, MMAs, exchange, epilogue.
// - An MMA of 64 rows reads half the shared memory of one of 128 and takes 24 cycles in the place of 40 (N = 24 or 32), so a CTA
//   can hold more of the K range: gate/up all of it, QKV half, output and down projection a quarter (a cluster of S CTAs then
//   exchanges partial sums, each pushing 64 rows in the place of 128: a CTA pushes some 32 bytes a cycle into its cluster).
// - A stage is several k-blocks, loaded by one request and waited for once.  Gate and up are one tensor of two matrices at the distance of
//   their addresses: as two requests per k-block they took a late CTA 1 us (18 tokens 704 -> 697 us, a tree of 54 868 -> 862).
// - All stages' weights are requested before tensor memory and the CTA's barrier, the activations as soon as the kernel before has ended, by
//   a warp that waits for neither, then whatever the epilogue needs besides
//   the sums (rows, places in the cache, rotation) is found, all before griddepcontrol.wait.
//   QKV, ADD  64 rows of one matrix;  GATEUP  32 rows of gate, then the same 32 of up, in the order of their addresses
// (All figures here: the XL shape and models like it, whose weights stay in L2.)
// An accumulator of M = 64 lies in lanes 0-15 of the four lane quarters; its rows go to shared memory as [token quad][rank][row]
// float4 (split: with st.async to the rank that owns the row, counted on its mbarrier), and the epilogue takes a pair of rows and
// two tokens per thread (four where 64 rows are finished at once, one of an output or down projection of up to 32), partial sums in rank order.
// (18 layers, 8, 18 and 28 tokens: activations requested by a warp that waits for nothing else 340.4 -> 338.8, 359.1 -> 357.1, 381.7 -> 380.0 us.
// One token a thread up to 32 tokens, 146 calls of 1 to 32 tokens at five widths: -0.4 % on average, -2.5 to +0.75 %; two tokens / one: XL shape,
// 12 tokens 323.1 / 321.1, 18 333.9 / 333.2, 28 349.0 / 346.6, 32 354.8 / 353.6; d_model 1024, 4 tokens 285.4 / 282.2, 32 323.5 / 324.3; 1536, d_ff
// 3008, 8 tokens 412.3 / 415.0, 18 442.3 / 437.5, 24 layers of 2048, 18 tokens 869.4 / 865.7.)
//
// Step of the XL shape against 128-row tiles: 18 tokens 876 -> 709 us, 28 tokens 920 -> 766, 54 tokens (a tree) 1061 -> 881; 18
// layers of it, 72 tokens 615 -> 538, 90 tokens 657 -> 585, 108 tokens 635 -> 641; of d_model 1024, 72 tokens 515 -> 473, 90
// tokens 540 -> 544, 108 tokens 556 -> 569: calls of up to 96 tokens come here.  K slices at 18 tokens: QKV 1 736 us, 2 709, 4 722;
// output projection 1 794, 2 733, 4 725; down projection 2 788, 4 733.
#include "tc_common.cuh"
#include "vvs_internal.cuh"

namespace vvs {

using namespace tc;
using namespace proj;

namespace {

constexpr int kThreads = 256;
constexpr uint32_t kRows = 64;
constexpr uint32_t kABytes = kRows * kBlockK * 2;

struct Params {
  int m, n, nt, kb_total, stages, group, parts, log_slices;      // parts: slices of proj_tc.cu's plan per CTA, log2 of all of them, columns
  int acc_ld;                                          // from one accumulator to the next (APART)
  uint32_t tmem_cols, recv_off;
  int32_t* status;
  const float* ss_in; int ss_parts; float inv_d, eps;                  // QKV, GATEUP: [token][ss_parts], a multiple of 4
  float* x; __nv_bfloat16* xg; const __nv_bfloat16* scale; float* ss_out; int ss_out_parts; int d;   // ADD
  __nv_bfloat16* q; __nv_bfloat16* kv_k; __nv_bfloat16* kv_v; const int32_t* slot_pos;               // QKV
  const float* rope_cos; const float* rope_sin; int n_heads, hd, s_max, layer, kv_rows, t_len;
  __nv_bfloat16* act; int ff, up_first;                                                            // GATEUP
  const uint8_t* ahead[2]; uint32_t ahead_bytes; AheadShare share;      // weights of the projection after next, to be brought into L2
};

// LOG_S: log2 of the slices of K; GROUP: k-blocks per stage (0: the plan's); RING: stages are filled again; TPI: tokens per item of the
// epilogue.  APART: every partial sum that proj_tc.cu's plan
// would take has an accumulator of its own (each of its slices; of a single matrix every other k-block), they are added in that
// kernel's order, and an ADD's sums of squares cover its rows in its order: the same bits, whichever of the two kernels runs.
// The issuing warp is alone in its loop, where every wait, vote and branch shows: 80 MMAs of 64 x 24 x 16 take 27.8 cycles each with
// ten k-blocks per wait, 31 with four, 47 with one, and 41 with four where a ring's bookkeeping is in the loop.  The loop over a stage's
// k-blocks is rolled all the same where all stages are there at once: a layer executes its code once, every line of which has to be
// fetched, and so the output and the down projection are the same code whatever their stages (18 layers of the XL shape 349.1 -> 341.3
// us, with the loop of qkv_attention_few.cu; only the down projection's stages as long as the output projection's: 343.3).
template <int EPI, int LOG_S, int GROUP, bool RING, bool APART, int TPI>
__global__ void __launch_bounds__(kThreads)
proj_few_kernel(const Params p, const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b) {
  constexpr bool DUAL = EPI == PROJ_GATEUP;
  constexpr int NACC = DUAL ? 2 : 1;
  constexpr bool SPLIT = LOG_S > 0;
  constexpr int S = 1 << LOG_S;
  const int parts = APART ? p.parts : 1;
  const uint32_t acc_ld = (uint32_t)p.acc_ld;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kFewStages];
  __shared__ __align__(8) uint64_t empty_bar[kFewStages];
  __shared__ __align__(8) uint64_t acc_bar;
  __shared__ __align__(8) uint64_t recv_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;
  __shared__ float s_rs[EPI == PROJ_ADD ? 1 : kFewTok];            // 1/rms of the tokens

  const int G = GROUP > 0 ? GROUP : p.group;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int tile = (int)blockIdx.x, rank = SPLIT ? (int)blockIdx.y : 0;
  const int nq = (p.m + 3) >> 2;
  const int kb0 = (rank * p.kb_total) >> LOG_S, nkb = (((rank + 1) * p.kb_total) >> LOG_S) - kb0, ng = (nkb + G - 1) / G;
  const uint32_t b_bytes = (uint32_t)p.nt * kBlockK * 2u, stage_bytes = G * (kABytes + b_bytes);   // weights, then activations
  uint8_t* recv = smem + p.recv_off;                               // [quad][source rank][row] float4

  auto load_w = [&](int i, uint32_t stage) {         // k-blocks i * G ..; by a converged warp
    uint8_t* st = smem + (size_t)stage * stage_bytes;
    if (elect_one()) {
      mbar_expect_tx(&full_bar[stage], stage_bytes);
      if (DUAL) {
        tma_load_4d(st, &tm_a, &full_bar[stage], 0, tile * (int)(kRows / 2), 0, kb0 + i * G);
      } else {
        tma_load_3d(st, &tm_a, &full_bar[stage], 0, tile * (int)kRows, kb0 + i * G);
      }
    }
  };
  const int n_pre = min(ng, p.stages);
  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&tm_b);
      for (int i = 0; i < p.stages; ++i) {
        mbar_init(&full_bar[i], 1);
        if (RING) mbar_init(&empty_bar[i], 1);
      }
      mbar_init(&acc_bar, 1);
      mbar_init(&recv_bar, 1);
      s_abort = 0;
      fence_barrier_init();
      fence_proxy_async();
      if (SPLIT) mbar_expect_tx(&recv_bar, (uint32_t)(nq * parts) * kRows * 16u);
    }
    __syncwarp();
    // All stages are free, so the weights go out first of all: a CTA that could only start when the kernel before it drained has
    // them sooner by what tensor memory and the barrier below take.
    for (int i = 0; i < n_pre; ++i) load_w(i, i);
  }
  if (warp == 2) {
    tmem_alloc(&tmem_slot, p.tmem_cols);
    tmem_relinquish();
  }
  auto load_act = [&](int i, uint32_t stage) {
    if (elect_one()) tma_load_3d(smem + (size_t)stage * stage_bytes + G * kABytes, &tm_b, &full_bar[stage], 0, 0, kb0 + i * G);
  };
  // The warp that requests does not wait for tensor memory: in a CTA that could only start when the kernel before it had ended, the
  // activations are requested 0.4 us sooner.
  if (warp == 0) {
    named_bar_arrive(1, kThreads);
    pdl_wait();
    for (int i = 0; i < n_pre; ++i) load_act(i, i);
    named_bar_sync(2, kThreads);
  } else {
    tc_fence_before();
    named_bar_sync(1, kThreads);
    pdl_launch_dependents();  // after this CTA holds its TMEM: a dependent grid cannot take it first
    named_bar_arrive(2, kThreads);
  }
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  if (SPLIT) cluster_arrive_relaxed();      // this rank's barrier is ready for its peers' pushes (fence_barrier_init above)

  // ---- this thread's first item of the epilogue: a pair of rows and TPI tokens, the last warps first (the first ones have other
  // work).  What does not depend on the kernel before is found here, under its tail; nothing waits for a load here.
  constexpr int rpr = (int)kRows >> LOG_S, log_np = (DUAL ? 4 : 5) - LOG_S;     // rows of a rank, log2 of the pairs it finishes
  const int eid = (kThreads / 32 - 1 - warp) * 32 + lane;
  constexpr int log_sub = TPI == 1 ? 2 : TPI == 2 ? 1 : 0;
  const int pair = (eid >> log_sub) & ((1 << log_np) - 1), sub = (eid & ((1 << log_sub) - 1)) * TPI;
  const int items = nq << (log_np + log_sub);
  const int row0 = DUAL ? tile * 32 : tile * (int)kRows + rank * rpr;       // first output row of this rank
  const int n = row0 + 2 * pair;
  const bool n_ok = n < p.n;
  const int sec = EPI == PROJ_QKV ? (tile * (int)kRows) / p.d : 0;          // (a tile lies in one head: 64 divides both)
  const int e = n - sec * p.d, h = EPI == PROJ_QKV ? e / p.hd : 0, i2 = e - h * p.hd;
  const float inv_t = EPI == PROJ_QKV ? 1.f / (float)p.t_len : 0.f;
  uint32_t scale2 = 0;                      // (converted where it is used: a conversion here would wait for it)
  if (EPI == PROJ_ADD && n_ok) scale2 = __ldg(reinterpret_cast<const uint32_t*>(p.scale + n));
  float cs[TPI], sn[TPI];
  __nv_bfloat16* dst[TPI];                  // null: not to be stored
  auto prepare = [&](int idx) {
    const int t0 = (idx >> (log_np + log_sub)) * 4 + sub;
#pragma unroll
    for (int j = 0; j < TPI; ++j) {
      const int tok = min(t0 + j, p.m - 1);
      cs[j] = 1.f;
      sn[j] = 0.f;
      if (EPI == PROJ_GATEUP) dst[j] = p.act + (size_t)tok * p.ff + n;
      if (EPI == PROJ_ADD) dst[j] = p.xg + (size_t)tok * p.d + n;
      if (EPI == PROJ_QKV) {
        if (sec < 2) {
          cs[j] = __ldg(p.rope_cos + (size_t)tok * (p.hd / 2) + (i2 >> 1));
          sn[j] = __ldg(p.rope_sin + (size_t)tok * (p.hd / 2) + (i2 >> 1));
        }
        if (sec == 0) {
          dst[j] = p.q + (size_t)tok * p.d + e;
        } else {
          const int slot = __ldg(p.slot_pos + tok), r = (int)(((float)tok + 0.5f) * inv_t);   // tok / t_len (exact below 2^21)
          const size_t row = (((size_t)p.layer * p.kv_rows + r) * p.n_heads + h) * p.s_max + slot;
          dst[j] = slot < 0 ? nullptr : (sec == 1 ? p.kv_k : p.kv_v) + row * p.hd + i2;
        }
      }
      if (idx >= items || !n_ok || t0 + j >= p.m) dst[j] = nullptr;
    }
  };
  if (warp >= 2) prepare(eid);
  if (warp == 2 && p.ahead_bytes > 0) {
    // This CTA's share of a later projection's weights, HBM -> L2 (proj_tc.cu has the measurements)
    const uint32_t begin = (blockIdx.y * gridDim.x + blockIdx.x) * p.share.every, end = min(begin + p.share.bytes, p.ahead_bytes);
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (p.ahead[i])
        for (uint32_t at = begin + lane * 4096u; at < end; at += 32 * 4096u) prefetch_l2(p.ahead[i] + at, min(4096u, end - at));
  }
  if (warp == 0) {
    if constexpr (RING) {
      uint32_t stage = 0, par = 0;                  // stage of group i, parity of its previous release
      for (int i = n_pre; i < ng; ++i) {
        if (!__all_sync(0xffffffffu, wait_or_abort(&empty_bar[stage], par, &s_abort))) {
          if (lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
          s_abort = 1;
          break;
        }
        load_w(i, stage);
        load_act(i, stage);
        if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1; }
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer -------------------------------------------------------------------------------
    const uint32_t idesc = idesc_bf16_f32(kRows, (uint32_t)p.nt), lo0 = desc_lo_sw128(smem_u32(smem)), stage_lo = stage_bytes >> 4;
    const uint32_t b_lo = b_bytes >> 4;
    // (a wait that ran out is reported and the loop goes on over what is there: no lane leaves the warp)
    auto wait_full = [&](uint32_t stage, uint32_t par) {
      if (!wait_or_abort(&full_bar[stage], par, &s_abort)) {
        atomicOr(p.status, VVS_DEV_TIMEOUT);
        s_abort = 1;
      }
      tc_fence_after();
    };
    auto block = [&](uint32_t a_lo, int j, uint32_t add) {
      mma_bf16_k64(tmem_base, a_lo + j * (kABytes >> 4), a_lo + G * (kABytes >> 4) + j * b_lo, idesc, add);
    };
    pdl_wait();
    if constexpr (APART) {
      // k-block at of slice q, which begins at k-block (rank * parts + q) * kb_total / slices: the boundaries of this CTA's range lie on them
      uint32_t stage = 0, par = 0, d = tmem_base;
      int at = 0, q = rank * parts, len = (((q + 1) * p.kb_total) >> p.log_slices) - kb0;
      for (int i = 0; i < ng; ++i) {
        wait_full(stage, par);
        const uint32_t a_lo = lo0 + stage * stage_lo;
#pragma unroll
        for (int j = 0; j < G; ++j) {
          if (i * G + j < nkb) {
            mma_bf16_k64(d + (DUAL || !(at & 1) ? 0u : acc_ld), a_lo + j * (kABytes >> 4), a_lo + G * (kABytes >> 4) + j * b_lo, idesc,
                         (uint32_t)(DUAL ? at : at >> 1));
            if (++at == len) {
              const int begin = (++q * p.kb_total) >> p.log_slices;
              len = (((q + 1) * p.kb_total) >> p.log_slices) - begin;
              at = 0;
              d += (DUAL ? 1u : 2u) * acc_ld;
            }
          }
        }
        if (i + p.stages < ng) mma_commit_elect(&empty_bar[stage]);  // a group is still to come into this stage
        if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1; }
      }
    } else if constexpr (RING) {
      uint32_t stage = 0, par = 0;
      for (int i = 0; i < ng; ++i) {
        wait_full(stage, par);
        const uint32_t a_lo = lo0 + stage * stage_lo;
        if (nkb - i * G >= G) {
#pragma unroll
          for (int j = 0; j < G; ++j) block(a_lo, j, j > 0 ? 1u : (uint32_t)i);
        } else {
#pragma unroll 1
          for (int j = 0; j < nkb - i * G; ++j) block(a_lo, j, (uint32_t)(i + j));
        }
        if (i + p.stages < ng) mma_commit_elect(&empty_bar[stage]);  // a group is still to come into this stage
        if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1; }
      }
    } else {
      for (int i = 0; i < ng; ++i) {
        wait_full(i, 0);
        const uint32_t a_lo = lo0 + i * stage_lo;
        const int n = min(G, nkb - i * G);
#pragma unroll 1
        for (int j = 0; j < n; ++j) block(a_lo, j, (uint32_t)(i + j));
      }
    }
    mma_commit_elect(&acc_bar);
  }
  __syncwarp();
  if (warp >= 2) pdl_wait();
  else prepare(eid);                        // (lanes past the last item too: the epilogue goes by whole warps and asks for their `dst`)
  float2 xo[TPI];
  auto load_x = [&](int idx) {
    const int t0 = (idx >> (log_np + log_sub)) * 4 + sub;
#pragma unroll
    for (int j = 0; j < TPI; ++j)
      xo[j] = *reinterpret_cast<const float2*>(p.x + (size_t)min(t0 + j, p.m - 1) * p.d + (n_ok ? n : 0));
  };
  if (EPI == PROJ_ADD && eid < items) load_x(eid);
  // ---- 1/rms of the tokens, while the MMAs run: eight tokens' loads in flight per warp ------------------------------
  if (EPI != PROJ_ADD && warp >= 3) {
    const int n4 = p.ss_parts >> 2;
    for (int t0 = (warp - 3) * 8; t0 < p.m; t0 += 8 * (kThreads / 32 - 3)) {
      float ss[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      for (int i = lane; i < n4; i += 32) {
        float4 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
          v[j] = __ldcg(reinterpret_cast<const float4*>(p.ss_in + (size_t)min(t0 + j, p.m - 1) * p.ss_parts) + i);
#pragma unroll
        for (int j = 0; j < 8; ++j) ss[j] += (v[j].x + v[j].y) + (v[j].z + v[j].w);
      }
      warp_sums(ss, lane);
      const int j = warp_sums_index<8>(lane);
      if ((lane & 3) == 0 && t0 + j < kFewTok) s_rs[t0 + j] = rsqrtf(ss[0] * p.inv_d + p.eps);
    }
  }
  if (SPLIT && EPI != PROJ_ADD) __syncthreads();    // s_rs
  // A CTA that gave up pushes whatever its accumulator holds: its peers' waits must still end.
  if (!wait_or_abort(&acc_bar, 0, &s_abort)) {
    if (lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
    s_abort = 1;
  }
  __syncwarp();       // each lane left the wait by itself, what follows is for a whole warp at once (.aligned)
  tc_fence_after();
  if (SPLIT) cluster_wait();
  // ---- rows to where the epilogue reads them ---------------------------------------------------------------------------
  {
    const int row_t = (warp & 3) * 16 + (lane & 15), owner = row_t >> (6 - LOG_S);
    const uint32_t at = smem_u32(recv) + (uint32_t)(SPLIT ? rank * parts * rpr + (row_t & (rpr - 1)) : row_t) * 16u;
    const uint32_t recv_dst = SPLIT ? mapa(at, (uint32_t)owner) : at, bar_dst = SPLIT ? mapa(smem_u32(&recv_bar), (uint32_t)owner) : 0u;
    const uint32_t t_row = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    for (int c0 = (warp >> 2) * 2; c0 < nq; c0 += 4) {
      float v[8];
      auto put = [&](uint32_t part) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (lane < 16 && c0 + j < nq) {
            const uint32_t dst = recv_dst + (uint32_t)((c0 + j) * (SPLIT ? parts : 1)) * (kRows * 16u) + part * (uint32_t)(rpr * 16);
            if (SPLIT) st_async4(dst, bar_dst, &v[4 * j]);
            else st_shared4(dst, &v[4 * j]);
          }
        }
      };
      if constexpr (APART) {
#pragma unroll 1
        for (int a = 0; a < parts; ++a) {
          const uint32_t t_acc = t_row + (uint32_t)(DUAL ? a : 2 * a) * acc_ld + (uint32_t)(c0 * 4);
          const int q = rank * parts + a;
          float w[8];
          tmem_ld8(t_acc, w);
          if (!DUAL && (((q + 1) * p.kb_total) >> p.log_slices) - ((q * p.kb_total) >> p.log_slices) > 1) {     // every other k-block
            float z[8];
            tmem_ld8(t_acc + acc_ld, z);
#pragma unroll
            for (int j = 0; j < 8; ++j) w[j] += z[j];
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = SPLIT || a == 0 ? w[j] : v[j] + w[j];
          if (SPLIT) put((uint32_t)a);
        }
        if (!SPLIT) put(0u);
      } else {
        tmem_ld8(t_row + (uint32_t)(c0 * 4), v);
        put(0u);
      }
    }
  }
  if (SPLIT) {
    // peers push after waits of at most kSpinLimit polls each, so this longer wait ends after their pushes
    bool got = false;
    for (uint32_t i = 0; i < 16u * kSpinLimit && !got; ++i) got = mbar_try_wait_cluster(&recv_bar, 0);
    if (!got && lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
  } else {
    tc_fence_before();
    __syncthreads();                          // the tile, s_rs
    if (warp == 2) tmem_dealloc(tmem_base, p.tmem_cols);
  }

  // ---- epilogue on finished sums ---------------------------------------------------------------------------------------
  const uint32_t src_row = (uint32_t)(2 * pair) * 16u + (uint32_t)sub * 4u;
  const int items_up = (items + 31) & ~31;                         // whole warps: the shuffles below need their lanes
  for (int idx = eid; idx < items_up; idx += kThreads) {
    const int quad = idx >> (log_np + log_sub), t0 = quad * 4 + sub;
    float acc[NACC][2][TPI];                                       // [row][token]
    const uint8_t* src = recv + (size_t)((idx < items ? quad : 0) * (SPLIT ? parts : 1)) * (kRows * 16u) + src_row;
#pragma unroll
    for (int a = 0; a < NACC; ++a)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint8_t* at = src + (DUAL ? a ^ p.up_first : 0) * (kRows / 2 * 16u) + i * 16;
        ld_shared_vec(at, acc[a][i]);
#pragma unroll
        for (int r = 1; r < (APART && SPLIT ? S * parts : S); ++r) {         // rank order
          float v[TPI];
          ld_shared_vec(at + r * rpr * 16, v);
#pragma unroll
          for (int j = 0; j < TPI; ++j) acc[a][i][j] += v[j];
        }
      }
    if constexpr (EPI == PROJ_ADD) {
      float sq[TPI], sq1[TPI];                 // APART: of the two rows, added last
      const float2 gsc = make_float2(__uint_as_float(scale2 << 16), __uint_as_float(scale2 & 0xffff0000u));
#pragma unroll
      for (int j = 0; j < TPI; ++j) {
        const float x0 = xo[j].x + acc[0][0][j], x1 = xo[j].y + acc[0][1][j];
        sq[j] = !dst[j] ? 0.f : APART ? __fmul_rn(x0, x0) : x0 * x0 + x1 * x1;
        sq1[j] = APART && dst[j] ? __fmul_rn(x1, x1) : 0.f;
        if (dst[j]) {
          *reinterpret_cast<float2*>(p.x + (size_t)(t0 + j) * p.d + n) = make_float2(x0, x1);
          *reinterpret_cast<uint32_t*>(dst[j]) = pack_bf16(x0 * gsc.x, x1 * gsc.y);
        }
      }
      // sums of squares over the rank's rows; the row of parts is a multiple of four long, the last CTA fills it up
      const int part = tile * S + rank, pad = p.ss_out_parts - (int)gridDim.x * S;
      float* ss = p.ss_out + part;
      if constexpr (TPI == 4) {
        warp_sums(sq, lane);
        const int j = warp_sums_index<4>(lane);
        if ((lane & 7) == 0 && t0 + j < p.m) ss[(size_t)(t0 + j) * p.ss_out_parts] = sq[0];
      } else {
        for (int o = 1 << (log_np + log_sub - 1); o >= 1 << log_sub; o >>= 1)
#pragma unroll
          for (int j = 0; j < TPI; ++j) {
            sq[j] += __shfl_xor_sync(0xffffffffu, sq[j], o);
            if (APART) sq1[j] += __shfl_xor_sync(0xffffffffu, sq1[j], o);
          }
        if (APART)
#pragma unroll
          for (int j = 0; j < TPI; ++j) sq[j] += sq1[j];
        if (idx < items && pair == 0)
#pragma unroll
          for (int j = 0; j < TPI; ++j)
            if (t0 + j < p.m) ss[(size_t)(t0 + j) * p.ss_out_parts] = sq[j];
      }
      if (part + 1 == (int)gridDim.x * S && pad > 0 && pair == 0 && idx < items)
        for (int j = 0; j < TPI; ++j)
          for (int i = 1; i <= pad; ++i)
            if (t0 + j < p.m) ss[(size_t)(t0 + j) * p.ss_out_parts + i] = 0.f;
    } else {
#pragma unroll
      for (int j = 0; j < TPI; ++j) {
        const float rs = s_rs[min(t0 + j, kFewTok - 1)];
        float a = acc[0][0][j] * rs, b = acc[0][1][j] * rs;
        if constexpr (DUAL) {
          a = __fdividef(a, 1.f + expf(-a)) * (acc[1][0][j] * rs);
          b = __fdividef(b, 1.f + expf(-b)) * (acc[1][1][j] * rs);
        } else {
          const float a0 = a;
          a = a0 * cs[j] - b * sn[j];         // (1, 0 for values)
          b = a0 * sn[j] + b * cs[j];
        }
        if (dst[j]) *reinterpret_cast<uint32_t*>(dst[j]) = pack_bf16(a, b);
      }
    }
    if (idx + kThreads < items_up) {
      prepare(idx + kThreads);
      if (EPI == PROJ_ADD) load_x(idx + kThreads);
    }
  }
  if (SPLIT) {
    tc_fence_before();
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem_base, p.tmem_cols);
  }
}

template <int EPI, int LOG_S, int GROUP, bool RING, bool APART = false>
cudaError_t launch_one(const ProjFewPlan& pl, const Params& kp, const ProjArgs& g, cudaStream_t s) {
  constexpr int kTpi = EPI == PROJ_GATEUP || LOG_S > 0 ? 2 : 4;
  auto* fn = proj_few_kernel<EPI, LOG_S, GROUP, RING, APART, kTpi>;
  if constexpr (EPI == PROJ_ADD && LOG_S > 0)          // up to 32 tokens every thread has one token's item at most
    if (kp.m <= 32) fn = proj_few_kernel<EPI, LOG_S, GROUP, RING, APART, 1>;

  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(fn), kFewSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(pl.tiles, pl.splits, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = pl.smem_bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (g.pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (LOG_S > 0) {                           // the K slices of a tile: one cluster along grid y
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = 1;
    attr[na].val.clusterDim.y = (unsigned)pl.splits;
    attr[na++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, fn, kp, *g.tm_a, *g.tm_b);
}

// (what plan_proj_few has no use for is not compiled: QKV has eight k-blocks or more and is split unless its sums are kept apart, an
// unsplit ADD has fewer than eight and needs no ring)
template <int EPI, int LOG_S>
cudaError_t launch_epi(const ProjFewPlan& pl, const Params& kp, const ProjArgs& g, cudaStream_t s) {
  if (pl.splits != 1 << LOG_S) return cudaErrorInvalidValue;
  if constexpr (EPI != PROJ_ADD || LOG_S > 0) {
    if (pl.parts > 0) return pl.group == 2 && pl.ring ? launch_one<EPI, LOG_S, 2, true, true>(pl, kp, g, s) : cudaErrorInvalidValue;
    if constexpr (EPI != PROJ_QKV || LOG_S > 0)
      if (pl.ring) return pl.group == 4 ? launch_one<EPI, LOG_S, 4, true>(pl, kp, g, s) : cudaErrorInvalidValue;
  }
  if (pl.parts > 0 || pl.ring) return cudaErrorInvalidValue;
  if constexpr (EPI != PROJ_QKV || LOG_S > 0) return launch_one<EPI, LOG_S, 0, false>(pl, kp, g, s);
  return cudaErrorInvalidValue;
}

}  // namespace

int launch_proj_few(int epi, const ProjFewPlan& pl, const ProjArgs& g, cudaStream_t s) {
  Params kp{};
  kp.m = g.m; kp.n = g.n; kp.nt = pl.nt; kp.kb_total = pl.kb_total; kp.stages = pl.stages; kp.group = pl.group; kp.parts = pl.parts; kp.acc_ld = pl.acc_ld;
  while ((1 << kp.log_slices) < pl.parts * pl.splits) ++kp.log_slices;
  kp.tmem_cols = (uint32_t)pl.tmem_cols; kp.recv_off = (uint32_t)pl.recv_off; kp.status = g.status;
  kp.ss_in = g.ss_in; kp.ss_parts = g.ss_parts; kp.inv_d = 1.f / (float)g.d; kp.eps = g.eps;
  kp.x = g.x; kp.xg = g.xg; kp.scale = g.scale; kp.ss_out = g.ss_out; kp.ss_out_parts = proj_ss_parts(pl); kp.d = g.d;
  kp.q = g.q; kp.kv_k = g.kv_k; kp.kv_v = g.kv_v; kp.slot_pos = g.slot_pos; kp.rope_cos = g.rope_cos;
  kp.rope_sin = g.rope_sin; kp.n_heads = g.n_heads; kp.hd = g.hd; kp.s_max = g.s_max; kp.layer = g.layer;
  kp.kv_rows = g.kv_rows; kp.t_len = g.t_len; kp.act = g.act; kp.ff = g.ff; kp.up_first = g.up_first ? 1 : 0;
  kp.ahead[0] = static_cast<const uint8_t*>(g.ahead[0]); kp.ahead[1] = static_cast<const uint8_t*>(g.ahead[1]);
  kp.ahead_bytes = g.ahead[0] ? g.ahead_bytes : 0;
  kp.share = ahead_share(kp.ahead_bytes, (uint32_t)(pl.tiles * pl.splits));
  cudaError_t e;
  switch (epi) {
    case PROJ_QKV: e = pl.splits == 2 ? launch_epi<PROJ_QKV, 1>(pl, kp, g, s) : launch_epi<PROJ_QKV, 0>(pl, kp, g, s); break;
    case PROJ_ADD: e = pl.splits == 4 ? launch_epi<PROJ_ADD, 2>(pl, kp, g, s) : launch_epi<PROJ_ADD, 0>(pl, kp, g, s); break;
    case PROJ_GATEUP: e = launch_epi<PROJ_GATEUP, 0>(pl, kp, g, s); break;
    default: return VVS_ERR_INVALID_ARG;
  }
  return e == cudaSuccess ? VVS_OK : VVS_ERR_CUDA;
}

}  // namespace vvs
