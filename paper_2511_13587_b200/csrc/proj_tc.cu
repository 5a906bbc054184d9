// Weight-streaming projections of the decoder with their epilogues folded in (bf16 contexts of wide models).
//
//   acc[n, tok] = sum_k w[n, k] * act[tok, k]          (w is [out_features, in_features])
//
// The 128 weight rows of a tile sit on the MMA's M side, the tokens on its N side (a batch-1 step has 18 tokens: no
// weight bandwidth is wasted on padding).  The K range of a tile is dealt to the S = 1, 2, 4 or 8 CTAs of a
// thread-block cluster.  Each accumulates its slice in TMEM and PUSHES the partial sums with st.async (registers -> the
// owner's shared memory, counted on the owner's mbarrier); rank r owns the r-th part of the tile's rows, adds the S
// partials in rank order -- no atomics, the same bits every call -- and applies the epilogue to finished sums:
//   QKV     1/rms, rotation of q and k, q to its buffer, k and v straight into the cache
//   GATEUP  1/rms, silu(gate) * up (two weight tiles on one activation tile, two accumulators)
//   ADD     residual x += acc, next norm's operand bf16(x * scale), partial sums of squares of x
// RMSNorm needs no kernel of its own: norm(x) W = rs * ((x * scale) W), so the ADD epilogue writes x * scale rounded
// once and the sums of squares per (token, row part), and the consumer multiplies its fp32 sums by rs.
//
// What bounds it: at 18 tokens the dependency chain (wait for the kernel before, activation tile from L2, a few MMAs,
// exchange, epilogue), not the weight stream, which is requested before griddepcontrol.wait while the previous
// kernels still run (programmatic dependent launch) -- as long as there is room for this kernel's CTAs beside
// theirs, which is why a CTA stays small; at some hundred tokens the fill of shared memory from L2.
// Step of the XL shape (36 layers, five kernels each, against ten with separate norm, rotation, cache append, gate and
// residual): 18 tokens 1012 -> 921 us (1535 in fixed-order contexts), 28 tokens 1720 -> 970, 288 tokens 2600 -> 1930;
// 7B shape, 18 tokens: 3410 -> 3025 us (4.9 TB/s over the whole step).  MMAs and loads issued by a converged warp in the place of a
// lone lane: 876, 920, 1821 and 2967 us (54 tokens, a tree: 1107 -> 1061).
#include "tc_common.cuh"
#include "vvs_internal.cuh"

namespace vvs {

using namespace tc;
using namespace proj;

namespace {

struct Params {
  int m, n, nt, kb_total, splits, log_s, stages, alias;
  uint32_t tmem_cols, recv_off;
  int32_t* status;
  const float* ss_in; int ss_parts; float inv_d, eps;                  // QKV, GATEUP: [token][ss_parts], a multiple of 4
  float* x; __nv_bfloat16* xg; const __nv_bfloat16* scale; float* ss_out; int ss_out_parts; int d;   // ADD
  __nv_bfloat16* q; __nv_bfloat16* kv_k; __nv_bfloat16* kv_v; const int32_t* slot_pos;               // QKV
  const float* rope_cos; const float* rope_sin; int n_heads, hd, s_max, layer, kv_rows, t_len;
  __nv_bfloat16* act; int ff;                                                                      // GATEUP
  const uint8_t* ahead[2]; uint32_t ahead_bytes;      // weights of the projection after next, to be brought into L2
};

// SIDE: grid (passes, slices, tiles), the passes of a tile side by side, in the place of (tiles, slices, passes)
template <int EPI, bool SPLIT, bool SIDE>
__global__ void __launch_bounds__(kMaxThreads)
proj_tc_kernel(const Params p, const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_a2,
               const __grid_constant__ CUtensorMap tm_b) {
  constexpr bool DUAL = EPI == PROJ_GATEUP;
  constexpr int NACC = DUAL ? 2 : 1;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages];
  __shared__ __align__(8) uint64_t empty_bar[kMaxStages];
  __shared__ __align__(8) uint64_t acc_bar;
  __shared__ __align__(8) uint64_t recv_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;
  __shared__ float s_rs[EPI == PROJ_ADD ? 1 : kMaxTok];            // 1/rms of the pass's tokens

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n_threads = (int)blockDim.x;
  const int tile = (int)(SIDE ? blockIdx.z : blockIdx.x), pass = (int)(SIDE ? blockIdx.x : blockIdx.z);
  const int rank = SPLIT ? (int)blockIdx.y : 0, S = SPLIT ? p.splits : 1;
  const int tok0 = pass * p.nt, ntok = min(p.nt, p.m - tok0), nq = (ntok + 3) >> 2;
  const int kb0 = (int)(((long long)rank * p.kb_total) / S);
  const int nkb = (int)(((long long)(rank + 1) * p.kb_total) / S) - kb0;
  constexpr uint32_t a_bytes = kATileBytes * NACC;
  const uint32_t stage_bytes = a_bytes + (uint32_t)p.nt * kBlockK * 2u;
  const int log_r = 7 - p.log_s, rpr = 1 << log_r;                 // rows per rank
  uint8_t* recv = smem + p.recv_off;                               // [accumulator][quad][source rank][row] float4

  if (tid == 0) {
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(&full_bar[i], 1);
      mbar_init(&empty_bar[i], DUAL ? 2 : 1);
    }
    mbar_init(&acc_bar, 2);                 // two issuing threads
    mbar_init(&recv_bar, 1);
    s_abort = 0;
    fence_barrier_init();
    mbar_expect_tx(&recv_bar, (uint32_t)((S - 1) * nq * rpr * 16 * NACC));
    tma_prefetch_desc(&tm_a);
    if (DUAL) tma_prefetch_desc(&tm_a2);
    tma_prefetch_desc(&tm_b);
  }
  if (warp == 1) {
    tmem_alloc(&tmem_slot, p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  pdl_launch_dependents();  // after this CTA holds its TMEM: a dependent grid cannot take it first
  if (SPLIT) cluster_arrive();              // this rank's barrier is ready for its peers' pushes

  if (warp == n_threads / 32 - 1 && p.ahead_bytes > 0) {
    // This CTA's share of a later projection's weights, HBM -> L2: a ring a few stages deep covers the latency of L2, not
    // that of HBM, and with some hundred tokens a tile's weights are read by several CTAs at once.  4 KB per request: the
    // unit that moves them takes ~50 cycles for each (1 KB pieces: 961 -> 1055 us per step of the XL shape, 16 KB: 972); by
    // the last warp, which has no token's 1/rms to find at up to 32 tokens (by the first of those that have: 967).
    const uint32_t n_cta = gridDim.x * gridDim.y * gridDim.z, cta = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    const uint32_t share = ((p.ahead_bytes + n_cta - 1) / n_cta + 4095u) & ~4095u, end = min((cta + 1) * share, p.ahead_bytes);
#pragma unroll
    for (int m = 0; m < 2; ++m)
      if (p.ahead[m])
        for (uint32_t at = cta * share + lane * 4096u; at < end; at += 32 * 4096u) prefetch_l2(p.ahead[m] + at, min(4096u, end - at));
  }
  if (warp == 0) {
    // ---- TMA producer: all stages are free, so the weights go out before the wait -----------------
    auto load_w = [&](int i, uint32_t stage) {
      if (elect_one()) {
        uint8_t* st = smem + (size_t)stage * stage_bytes;
        mbar_expect_tx(&full_bar[stage], stage_bytes);
        tma_load_2d(st, &tm_a, &full_bar[stage], (kb0 + i) * (int)kBlockK, tile * (int)kTileRows);
        if (DUAL) tma_load_2d(st + kATileBytes, &tm_a2, &full_bar[stage], (kb0 + i) * (int)kBlockK, tile * (int)kTileRows);
      }
    };
    const int n_pre = nkb < p.stages ? nkb : p.stages;
    for (int i = 0; i < n_pre; ++i) load_w(i, i);
    auto load_act = [&](int i, uint32_t stage) {
      if (elect_one()) tma_load_2d(smem + (size_t)stage * stage_bytes + a_bytes, &tm_b, &full_bar[stage], (kb0 + i) * (int)kBlockK, tok0);
    };
    pdl_wait();  // activations come from the previous kernel
    for (int i = 0; i < n_pre; ++i) load_act(i, i);
    uint32_t stage = 0, par = 0;                  // stage of block i, parity of its previous release
    for (int i = n_pre; i < nkb; ++i) {
      if (!__all_sync(0xffffffffu, wait_or_abort(&empty_bar[stage], par, &s_abort))) {
        if (lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
        s_abort = 1;
        break;
      }
      load_w(i, stage);
      load_act(i, stage);
      if (++stage == (uint32_t)p.stages) { stage = 0; par ^= 1; }
    }
  } else if (warp == 1 || warp == 2) {
    // ---- MMA issuers: one lane of the warp issues, all of it runs the loop (mma_bf16_k64).  Two warps share the work, each with
    // accumulators of its own: gate and up, or every other k-block of a single matrix (added below)
    const int me = __shfl_sync(0xffffffffu, warp, 0) - 1;
    const uint32_t idesc = idesc_bf16_f32(kTileRows, (uint32_t)p.nt), d = tmem_base + (uint32_t)(me * p.nt);
    const uint32_t lo0 = desc_lo_sw128(smem_u32(smem)), stage_lo = stage_bytes >> 4;
    uint32_t stage = DUAL ? 0 : me, par = 0, add = 0;
    if (stage >= (uint32_t)p.stages) { stage -= p.stages; par = 1; }
    for (int i = DUAL ? 0 : me; i < nkb; i += DUAL ? 1 : 2) {
      if (!__all_sync(0xffffffffu, wait_or_abort(&full_bar[stage], par, &s_abort))) {
        if (lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
        s_abort = 1;
        break;
      }
      tc_fence_after();
      const uint32_t a_lo = lo0 + stage * stage_lo;
      mma_bf16_k64(d, a_lo + (DUAL ? me * (kATileBytes >> 4) : 0u), a_lo + (a_bytes >> 4), idesc, add);
      add = 1;
      if (i + p.stages < nkb) mma_commit_elect(&empty_bar[stage]);  // a block is still to come into this stage
      stage += DUAL ? 1 : 2;
      while (stage >= (uint32_t)p.stages) { stage -= p.stages; par ^= 1; }
    }
    mma_commit_elect(&acc_bar);
  }
  __syncwarp();
  pdl_wait();

  // ---- 1/rms of the pass's tokens, while the MMAs run: a warp per token, eight tokens' loads in flight ---------------
  if (EPI != PROJ_ADD && warp >= 3) {
    const int n4 = p.ss_parts >> 2;
    for (int t0 = (warp - 3) * 8; t0 < ntok; t0 += 8 * (n_threads / 32 - 3)) {
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
      if ((lane & 3) == 0 && t0 + j < kMaxTok) s_rs[t0 + j] = rsqrtf(ss[0] * p.inv_d + p.eps);
    }
  }
  // this thread's first item of the epilogue: rows of rank `rank`, four tokens
  const int n0 = tile * (int)kTileRows + (rank << log_r);
  const int items = nq << log_r;
  float xo[4] = {0.f, 0.f, 0.f, 0.f}, gsc = 0.f;
  auto load_x = [&](int idx) {
    const int n = n0 + (idx & (rpr - 1)), t = tok0 + (idx >> log_r) * 4;
#pragma unroll
    for (int j = 0; j < 4; ++j) xo[j] = n < p.n && t + j < p.m ? p.x[(size_t)(t + j) * p.d + n] : 0.f;
  };
  if (SPLIT && EPI == PROJ_ADD && tid < items) {
    load_x(tid);                                                   // (n_threads is a multiple of rpr: the row stays)
    const int n = n0 + (tid & (rpr - 1));
    if (n < p.n) gsc = __bfloat162float(p.scale[n]);
  }

  // ---- unsplit: row of this thread, and what its first sixteen tokens' epilogue needs besides the sums -------------------
  const int row_t = (warp & 3) * 32 + lane;   // weight row of this thread in TMEM
  const int nu = tile * (int)kTileRows + row_t;
  const bool nu_ok = nu < p.n;
  int sec = 0, e = 0, h = 0, i2 = 0;
  if (!SPLIT && EPI == PROJ_QKV) {
    sec = nu / p.d;
    e = nu - sec * p.d;
    h = e / p.hd;
    i2 = e - h * p.hd;
  }
  const float gsc1 = !SPLIT && EPI == PROJ_ADD && nu_ok ? __bfloat162float(p.scale[nu]) : 0.f;
  float f0[16], f1[8];
  auto operands = [&](int c0) {
    if (EPI == PROJ_ADD) {
#pragma unroll
      for (int j = 0; j < 16; ++j) f0[j] = nu_ok && c0 + j < ntok ? p.x[(size_t)(tok0 + c0 + j) * p.d + nu] : 0.f;
    } else if (EPI == PROJ_QKV) {             // rotation of the eight tokens this lane finishes
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int tok = tok0 + min(c0 + j + ((lane & 1) ? 8 : 0), ntok - 1);
        f0[j] = sec < 2 ? __ldg(p.rope_cos + (size_t)tok * (p.hd / 2) + (i2 >> 1)) : 1.f;
        f1[j] = sec < 2 ? __ldg(p.rope_sin + (size_t)tok * (p.hd / 2) + (i2 >> 1)) : 0.f;
      }
    }
  };
  if (!SPLIT && (warp >> 2) * 16 < ntok) operands((warp >> 2) * 16);

  // A CTA that gave up pushes whatever its accumulator holds: its peers' waits must still end.
  if (!warp_wait_or_abort(&acc_bar, 0, &s_abort)) {
    if (lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
    s_abort = 1;
  }
  tc_fence_after();
  const bool two = !DUAL && nkb > 1;          // a second accumulator holds every other k-block
  if (SPLIT) {
    cluster_wait();
    if (p.alias) {                            // the exchange lies over the stages: every rank is done with them
      cluster_arrive();
      cluster_wait();
    }
  }
  const uint32_t t_row = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
  if constexpr (!SPLIT) {
    // ---- the sums are complete: epilogue straight from TMEM, sixteen tokens at a time.  The two rows of a lane pair trade
    // half their tokens, so that every lane finishes whole bf16 pairs; these go to shared memory (token-major, over the
    // stages, which have drained) and leave as 16-byte pieces.  Stores of 4 bytes by every other lane, with the addresses
    // of each, took 3 us per sixteen tokens.
    constexpr int kOutLd = 272;               // bytes per token: 128 rows and a pad
    __syncthreads();                          // s_rs; every warp has passed the accumulator's barrier
    const bool odd = lane & 1;
#pragma unroll 1
    for (int c0 = (warp >> 2) * 16; c0 < ntok; c0 += n_threads / 8) {
      float y[16], z[16];
      tmem_ld16(t_row + (uint32_t)c0, y);
      if (DUAL || two) tmem_ld16(t_row + (uint32_t)(p.nt + c0), z);
      if (two) {
#pragma unroll
        for (int j = 0; j < 16; ++j) y[j] += z[j];
      }
      if constexpr (EPI == PROJ_ADD) {
        float sq[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const bool ok = nu_ok && c0 + j < ntok;
          const float xn = f0[j] + y[j];
          if (ok) p.x[(size_t)(tok0 + c0 + j) * p.d + nu] = xn;
          y[j] = xn * gsc1;
          sq[j] = ok ? xn * xn : 0.f;
        }
        warp_sums(sq, lane);
        const int j = warp_sums_index<16>(lane);
        if (!odd && c0 + j < ntok) p.ss_out[(size_t)(tok0 + c0 + j) * p.ss_out_parts + tile * 4 + (warp & 3)] = sq[0];
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float rs = s_rs[c0 + j];
          y[j] *= rs;
          if (DUAL) y[j] = __fdividef(y[j], 1.f + expf(-y[j])) * (z[j] * rs);
        }
      }
      const int t8 = odd ? 8 : 0;             // this lane's eight tokens: rows (even, odd) of the pair
      uint8_t* out = smem + (size_t)(c0 + t8) * kOutLd + (row_t & ~1) * 2;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float keep = odd ? y[8 + j] : y[j], got = __shfl_xor_sync(0xffffffffu, odd ? y[j] : y[8 + j], 1);
        float a = odd ? got : keep, b = odd ? keep : got;
        if (EPI == PROJ_QKV) {                // (f0, f1: this lane's eight tokens; 1, 0 for values)
          const float a0 = a;
          a = a0 * f0[j] - b * f1[j];
          b = a0 * f1[j] + b * f0[j];
        }
        *reinterpret_cast<uint32_t*>(out + j * kOutLd) = pack_bf16(a, b);
      }
      if (c0 + n_threads / 8 < ntok) operands(c0 + n_threads / 8);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, p.tmem_cols);
    // ---- 16-byte pieces: eight rows of a token; a thread's rows are the same for all its tokens -------------------------
    const int c8 = tid & 15, n8 = tile * (int)kTileRows + c8 * 8;
    if (n8 >= p.n) return;
    __nv_bfloat16* dst0;
    size_t dst_ld = 0;
    int s8 = 0;
    if (EPI == PROJ_ADD) {
      dst0 = p.xg + n8;
      dst_ld = p.d;
    } else if (EPI == PROJ_GATEUP) {
      dst0 = p.act + n8;
      dst_ld = p.ff;
    } else {
      s8 = n8 / p.d;
      const int e8 = n8 - s8 * p.d, h8 = e8 / p.hd;
      dst0 = s8 == 0 ? p.q + e8
                     : (s8 == 1 ? p.kv_k : p.kv_v) + (((size_t)p.layer * p.kv_rows * p.n_heads + h8) * p.s_max) * p.hd + (e8 - h8 * p.hd);
      dst_ld = p.d;
    }
    const float inv_tl = EPI == PROJ_QKV ? 1.f / (float)p.t_len : 0.f;
#pragma unroll 4
    for (int t = tid >> 4; t < ntok; t += n_threads / 16) {
      const uint4 v = *reinterpret_cast<const uint4*>(smem + (size_t)t * kOutLd + c8 * 16);
      const int tok = tok0 + t;
      if (EPI == PROJ_QKV && s8 > 0) {
        const int slot = __ldg(p.slot_pos + tok), r = (int)(((float)tok + 0.5f) * inv_tl);   // tok / t_len (exact below 2^21)
        if (slot >= 0) *reinterpret_cast<uint4*>(dst0 + ((size_t)r * p.n_heads * p.s_max + slot) * p.hd) = v;
      } else {
        *reinterpret_cast<uint4*>(dst0 + (size_t)tok * dst_ld) = v;
      }
    }
    return;
  }
  // ---- exchange: every row's partial sums to the row's owner ---------------------------------------------------------
  {
    const int owner = row_t >> log_r;
    const uint32_t at = (uint32_t)((rank << log_r) + (row_t & (rpr - 1))) * 16u;        // inside a quad's [S][rpr]
    const bool self = owner == rank;
    const uint32_t recv_dst = mapa(smem_u32(recv) + at, (uint32_t)owner), bar_dst = mapa(smem_u32(&recv_bar), (uint32_t)owner);
    for (int c0 = (warp >> 2) * 4; c0 < nq; c0 += n_threads / 32) {
#pragma unroll
      for (int a = 0; a < NACC; ++a) {
        float v[16], w[16];
        tmem_ld16(t_row + (uint32_t)(a * p.nt + c0 * 4), v);
        if (two) {
          tmem_ld16(t_row + (uint32_t)(p.nt + c0 * 4), w);
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] += w[j];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (c0 + j < nq) {
            const uint32_t off = (uint32_t)(a * nq + c0 + j) * (kTileRows * 16u);
            if (self) *reinterpret_cast<float4*>(recv + off + at) = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            else st_async4(recv_dst + off, bar_dst, &v[4 * j]);
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();                            // own sums and s_rs; also: every thread is done with TMEM
  if (warp == 1) tmem_dealloc(tmem_base, p.tmem_cols);
  {
    // peers push after waits of at most kSpinLimit polls each, so this longer wait ends after their pushes
    bool got = false;
    for (uint32_t i = 0; i < 16u * kSpinLimit && !got; ++i) got = mbar_try_wait_cluster(&recv_bar, 0);
    if (!got && lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
  }

  // ---- epilogue on finished sums: thread = weight row, four tokens per item ------------------------------------------
  const int row_l = tid & (rpr - 1), n = n0 + row_l;               // the same row in every item of a thread
  const bool n_ok = n < p.n;
  const float4* src0 = reinterpret_cast<const float4*>(recv) + row_l;
  if (EPI == PROJ_QKV) {
    sec = n / p.d;
    e = n - sec * p.d;
    h = e / p.hd;
    i2 = e - h * p.hd;
  }
  const float inv_t = EPI == PROJ_QKV ? 1.f / (float)p.t_len : 0.f;
  const size_t kv_row = (size_t)p.n_heads * p.s_max;               // cache rows per sequence
  const size_t kv_base = EPI == PROJ_QKV ? (((size_t)p.layer * p.kv_rows * p.n_heads + h) * p.s_max) * p.hd + i2 : 0;
  const int items_up = (items + 31) & ~31;                         // whole warps: the shuffles below need their lanes
  for (int idx = tid; idx < items_up; idx += n_threads) {
    const int quad = idx >> log_r, t_first = tok0 + quad * 4;
    const bool live = idx < items;
    float acc[NACC][4];
#pragma unroll
    for (int a = 0; a < NACC; ++a) {
      const float4* src = src0 + (size_t)(a * nq + (live ? quad : 0)) * kTileRows;
      float4 s = src[0];
#pragma unroll 4
      for (int r = 1; r < S; ++r) {           // rank order
        const float4 t = src[r << log_r];
        s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
      }
      acc[a][0] = s.x; acc[a][1] = s.y; acc[a][2] = s.z; acc[a][3] = s.w;
    }
    if constexpr (EPI == PROJ_ADD) {
      float xn[4], sq[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        xn[j] = xo[j] + acc[0][j];
        sq[j] = live && n_ok && t_first + j < p.m ? xn[j] * xn[j] : 0.f;
      }
      if (idx + n_threads < items) load_x(idx + n_threads);          // the next item's residual travels under this one
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int tok = t_first + j;
        const bool ok = live && n_ok && tok < p.m;
        if (ok) p.x[(size_t)tok * p.d + n] = xn[j];
        const float y = xn[j] * gsc, y2 = __shfl_xor_sync(0xffffffffu, y, 1);
        if (ok && !(lane & 1)) *reinterpret_cast<uint32_t*>(p.xg + (size_t)tok * p.d + n) = pack_bf16(y, y2);
      }
      // sums of squares over the rank's rows (over each warp's 32 of them where it has more)
      for (int o = min(16, rpr >> 1); o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < 4; ++j) sq[j] += __shfl_xor_sync(0xffffffffu, sq[j], o);
      if (live && (row_l & (min(32, rpr) - 1)) == 0) {
        const int part = (tile * (int)kTileRows + (rank << log_r) + row_l) / min(32, rpr);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (t_first + j < p.m) p.ss_out[(size_t)(t_first + j) * p.ss_out_parts + part] = sq[j];
      }
    } else if constexpr (EPI == PROJ_GATEUP) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int tok = t_first + j;
        const float rs = s_rs[quad * 4 + j < kMaxTok ? quad * 4 + j : 0];
        const float g = acc[0][j] * rs, u = acc[NACC - 1][j] * rs;
        const float y = __fdividef(g, 1.f + expf(-g)) * u, y2 = __shfl_xor_sync(0xffffffffu, y, 1);
        if (live && n_ok && tok < p.m && !(lane & 1))
          *reinterpret_cast<uint32_t*>(p.act + (size_t)tok * p.ff + n) = pack_bf16(y, y2);
      }
    } else {
      float cs[4], sn[4];
      int slot[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {                                // one round trip (mostly L1: every head reads the same)
        const int tok = min(t_first + j, p.m - 1);
        cs[j] = sec < 2 ? __ldg(p.rope_cos + (size_t)tok * (p.hd / 2) + (i2 >> 1)) : 1.f;
        sn[j] = sec < 2 ? __ldg(p.rope_sin + (size_t)tok * (p.hd / 2) + (i2 >> 1)) : 0.f;
        slot[j] = sec > 0 ? __ldg(p.slot_pos + tok) : 0;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int tok = t_first + j;
        const bool ok = live && n_ok && tok < p.m;
        const float val = acc[0][j] * s_rs[quad * 4 + j < kMaxTok ? quad * 4 + j : 0];
        const float other = __shfl_xor_sync(0xffffffffu, val, 1);      // the pair partner (row n ^ 1)
        if (ok && !(lane & 1) && slot[j] >= 0) {
          const uint32_t pk = sec < 2 ? pack_bf16(val * cs[j] - other * sn[j], val * sn[j] + other * cs[j]) : pack_bf16(val, other);
          __nv_bfloat16* dst;
          if (sec == 0) {
            dst = p.q + (size_t)tok * p.d + e;
          } else {
            const int r = (int)(((float)tok + 0.5f) * inv_t);      // tok / t_len (exact: tok is far below 2^21)
            dst = (sec == 1 ? p.kv_k : p.kv_v) + kv_base + ((size_t)r * kv_row + slot[j]) * p.hd;
          }
          *reinterpret_cast<uint32_t*>(dst) = pk;
        }
      }
    }
  }
}

template <int EPI>
cudaError_t launch_epi(const ProjPlan& pl, const Params& kp, const ProjArgs& g, cudaStream_t s) {
  auto* fn = pl.splits > 1 ? (pl.tiles_on_z ? proj_tc_kernel<EPI, true, true> : proj_tc_kernel<EPI, true, false>)
                           : (pl.tiles_on_z ? proj_tc_kernel<EPI, false, true> : proj_tc_kernel<EPI, false, false>);
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(fn), 222 * 1024);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = pl.tiles_on_z ? dim3(pl.passes, pl.splits, pl.tiles) : dim3(pl.tiles, pl.splits, pl.passes);
  cfg.blockDim = dim3(pl.threads, 1, 1);
  cfg.dynamicSmemBytes = pl.smem_bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (g.pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (pl.splits > 1) {                       // the K slices of a tile: one cluster along grid y
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = 1;
    attr[na].val.clusterDim.y = (unsigned)pl.splits;
    attr[na++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, fn, kp, *g.tm_a, g.tm_a2 ? *g.tm_a2 : *g.tm_a, *g.tm_b);
}

}  // namespace

int launch_proj(int epi, const ProjPlan& pl, const ProjArgs& g, cudaStream_t s) {
  Params kp{};
  kp.m = g.m; kp.n = g.n; kp.nt = pl.nt; kp.kb_total = pl.kb_total; kp.splits = pl.splits; kp.stages = pl.stages;
  while ((1 << kp.log_s) < pl.splits) ++kp.log_s;
  kp.alias = pl.alias; kp.tmem_cols = (uint32_t)pl.tmem_cols; kp.recv_off = (uint32_t)pl.recv_off; kp.status = g.status;
  kp.ss_in = g.ss_in; kp.ss_parts = g.ss_parts; kp.inv_d = 1.f / (float)g.d; kp.eps = g.eps;
  kp.x = g.x; kp.xg = g.xg; kp.scale = g.scale; kp.ss_out = g.ss_out; kp.ss_out_parts = epi == PROJ_ADD ? proj_ss_parts(pl) : 0; kp.d = g.d;
  kp.q = g.q; kp.kv_k = g.kv_k; kp.kv_v = g.kv_v; kp.slot_pos = g.slot_pos; kp.rope_cos = g.rope_cos;
  kp.rope_sin = g.rope_sin; kp.n_heads = g.n_heads; kp.hd = g.hd; kp.s_max = g.s_max; kp.layer = g.layer;
  kp.kv_rows = g.kv_rows; kp.t_len = g.t_len; kp.act = g.act; kp.ff = g.ff;
  kp.ahead[0] = static_cast<const uint8_t*>(g.ahead[0]); kp.ahead[1] = static_cast<const uint8_t*>(g.ahead[1]);
  kp.ahead_bytes = g.ahead[0] ? g.ahead_bytes : 0;
  cudaError_t e;
  switch (epi) {
    case PROJ_QKV: e = launch_epi<PROJ_QKV>(pl, kp, g, s); break;
    case PROJ_ADD: e = launch_epi<PROJ_ADD>(pl, kp, g, s); break;
    case PROJ_GATEUP: e = launch_epi<PROJ_GATEUP>(pl, kp, g, s); break;
    default: return VVS_ERR_INVALID_ARG;
  }
  return e == cudaSuccess ? VVS_OK : VVS_ERR_CUDA;
}

}  // namespace vvs
