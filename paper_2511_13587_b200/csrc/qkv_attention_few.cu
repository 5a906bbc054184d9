// QKV projection and attention of calls with few tokens and one to three sequences as one kernel (bf16 contexts of wide models with 64-wide
// heads whose weights stay in L2): proj_few.cu's QKV and attention_block.cu's attention, the same sums, roundings and order, bit for bit.
//
// What bounds the two as kernels of their own is the chain: behind the last CTA of QKV the wait of attention is released after 1.0 us, and q
// and the new keys come from L2 in another 0.8.  Here the six CTAs that have a head's rows -- tiles of q, k and v, two K slices each -- are a
// cluster.
// - They push the rows that they finish to the CTAs that attend with them (st.async, counted on the receiver's mbarrier): there 0.2 us after
//   the last was finished.  The cache gets its rows as before; q is nowhere else.
// - A sequence's head is shared by 6 / n_rows of the six CTAs.  The sixteen warps that attention_block.cu gives an item are dealt to them,
//   each with its slot of 32 keys, which lies over the stages, drained by then (old keys are requested into L2 before the wait and into
//   the slots behind the exchange).  XL shape, two sequences: 120 KB a CTA with 9 rows each, 152 with 14, 175 with 27 (from 10 rows on the parts
//   that one CTA folds set the size); with slots of their own 172 with 9.
// - One of these CTAs gathers the warps' parts, also by st.async, and folds them in the order of the sixteen; the others end.
// - The output projection takes more than half of an SM's shared memory then (vvs_api.cu): its CTAs would all start on the 28 SMs that this
//   kernel leaves free, three to an SM (18 layers, 18 tokens 348.0 us with what it needs, 332.5 with 116 KB; 28 tokens 358.7, 346.7; a tree
//   of 54 437.4, 423.4; one sequence of 9 tokens 344.1, 345.1).
// - Loops are rolled and code is not repeated where a layer executes it once: a rolled loop of MMAs 343.3 -> 338.8 us.
// 18 layers of the XL shape, two kernels / this one (us): guidance, 3 / 9 / 16 rows a sequence, 500 cached 355 / 334, 369 / 355, 399 / 388; 50 cached
// 344 / 327, 356 / 341, 372 / 358; trees of 20 and 32 rows, 500 cached 492 / 442, 535 / 490; without guidance, 9 rows, 570 cached 377 / 353; 24 layers
// of d_model 1024 (18 of them 328 / 306).
#include "att_mma.cuh"
#include "tc_common.cuh"
#include "vvs_internal.cuh"

namespace vvs {

using namespace tc;
using namespace proj;
using namespace attmma;

namespace {

using bf16 = __nv_bfloat16;
constexpr int kThreads = 256, kCtas = 6;              // CTAs of a cluster
constexpr int HD = 64, KS = 32, kParts = 16;          // keys of a slice; warps' parts of an item
constexpr uint32_t kRows = 64, kABytes = kRows * kBlockK * 2;
constexpr uint32_t kSlice = 2 * KS * HD * 2;          // K, then V
// Row of a part: a lane's values lie side by side, column 8 j + 2 c + e at c kSeg + 2 j + e (padded for both accesses).
constexpr int kSeg = HD / 4 + 8, kPartLd = 4 * kSeg + 4;

struct Params {
  int m, nt, kb_total, stages, group;
  uint32_t tmem_cols, recv_off, part_off, new_off;
  int32_t* status;
  const float* ss_in; int ss_parts; float inv_d, eps; int d;
  bf16* kv_k; bf16* kv_v; const int32_t* slot_pos; const float* rope_cos; const float* rope_sin;
  const int32_t* cache_len; const uint32_t* anc_mask; bf16* out;
  int n_heads, s_max, layer, kv_rows, t_len, per_item;                  // per_item: CTAs that share an item
  const uint8_t* ahead[2]; uint32_t ahead_bytes; AheadShare share;
};

__global__ void __launch_bounds__(kThreads, 1)
qkv_attention_kernel(const __grid_constant__ Params p, const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kFewStages];
  __shared__ __align__(8) uint64_t acc_bar, recv_bar, new_bar, part_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;
  __shared__ float s_rs[kFewTok];

  const int G = p.group;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int cta = (int)blockIdx.x, head = (int)blockIdx.y;         // cta: rank in the cluster
  const int sec = cta >> 1, rank = cta & 1;                        // q, k or v; K slice
  const int T = p.t_len, nq = (p.m + 3) >> 2;
  const int kb0 = (rank * p.kb_total) >> 1, nkb = (((rank + 1) * p.kb_total) >> 1) - kb0, ng = (nkb + G - 1) / G;
  const uint32_t b_bytes = (uint32_t)p.nt * kBlockK * 2u, stage_bytes = G * (kABytes + b_bytes);
  uint8_t* recv = smem + p.recv_off;                               // [quad][source rank][row] float4

  // ---- the attention item of this CTA: sequence `seq`, parts part0, part0 + per_item, .. of the sixteen, one a warp -------------
  const int seq = cta / p.per_item, part0 = cta - seq * p.per_item;
  const int gather = seq * p.per_item;                             // the CTA that folds the parts
  const int part = part0 + warp * p.per_item;
  const int groups = T > 16 ? 2 : 1, wpg = kParts / groups, grp = part / wpg, wg = part - grp * wpg;     // parts are dealt to the row groups
  const int fill = p.cache_len[seq];
  const int n_keys = fill >= 0 && fill + T <= p.s_max ? fill + T : 0, n_slices = (n_keys + KS - 1) / KS, busy = min(wpg, n_slices);
  const bool mine = part < kParts && wg < n_slices;
  const uint32_t slot = smem_u32(smem) + (uint32_t)warp * kSlice;
  const int key0 = lane >> 3, ch = lane & 7;
  const size_t cache_row = ((size_t)p.layer * p.kv_rows + seq) * p.n_heads + head;

  auto load_w = [&](int i) {
    uint8_t* st = smem + (size_t)i * stage_bytes;
    if (elect_one()) {
      mbar_expect_tx(&full_bar[i], stage_bytes);
      tma_load_3d(st, &tm_a, &full_bar[i], 0, (sec * p.n_heads + head) * (int)kRows, kb0 + i * G);
    }
  };
  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&tm_b);
      for (int i = 0; i < p.stages; ++i) mbar_init(&full_bar[i], 1);
      mbar_init(&acc_bar, 1);
      mbar_init(&recv_bar, 1);
      mbar_init(&new_bar, 1);
      mbar_init(&part_bar, 1);
      s_abort = 0;
      fence_barrier_init();
      fence_proxy_async();
    }
    __syncwarp();
    for (int i = 0; i < ng; ++i) load_w(i);                          // (before anything that waits for a load)
    if (lane == 0) {
      mbar_expect_tx(&recv_bar, (uint32_t)nq * kRows * 16u);
      mbar_expect_tx(&new_bar, (uint32_t)T * 3u * HD * 2u);
      uint32_t bytes = 0;                                          // what the peers' warps push here
      if (cta == gather)
        for (int i = 0; i < kParts; ++i)
          if (i % p.per_item && i % wpg < busy) bytes += (uint32_t)(i < wpg ? min(T, 16) : T - 16) * (HD + 2) * 4u;
      mbar_expect_tx(&part_bar, bytes);
    }
    __syncwarp();
  }
  if (warp == 2) {
    tmem_alloc(&tmem_slot, p.tmem_cols);
    tmem_relinquish();
  }
  auto request = [&](int s) {                                      // the old keys of slice s
    const int left = min(fill, n_keys) - s * KS - key0;
    const size_t at = (cache_row * p.s_max + (size_t)s * KS + key0) * HD + ch * 8;
#pragma unroll
    for (int u = 0; u < KS / 4; ++u)
      if (4 * u < left) {
        const int k = key0 + 4 * u;
        const uint32_t dst = slot + (uint32_t)k * 128u + (uint32_t)((ch ^ (k & 7)) << 4);
        cp_async16(dst, p.kv_k + at + (size_t)u * 4 * HD);
        cp_async16(dst + KS * 128u, p.kv_v + at + (size_t)u * 4 * HD);
      }
  };
  if (mine && lane < 2 && wg * KS < min(fill, n_keys)) {           // the old keys of this warp's first slice into L2
    const bf16* at = (lane ? p.kv_v : p.kv_k) + (cache_row * p.s_max + (size_t)wg * KS) * HD;
    prefetch_l2(at, (uint32_t)min(KS, min(fill, n_keys) - wg * KS) * HD * 2u);
  }
  // The warp that requests does not wait for tensor memory (as in proj_few.cu).
  if (warp == 0) {
    named_bar_arrive(1, kThreads);
    pdl_wait();
    for (int i = 0; i < ng; ++i)
      if (elect_one()) tma_load_3d(smem + (size_t)i * stage_bytes + G * kABytes, &tm_b, &full_bar[i], 0, 0, kb0 + i * G);
    named_bar_sync(2, kThreads);
  } else {
    tc_fence_before();
    named_bar_sync(1, kThreads);
    pdl_launch_dependents();  // after this CTA holds its TMEM: a dependent grid cannot take it first
    named_bar_arrive(2, kThreads);
  }
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  cluster_arrive_relaxed();      // this CTA's barriers are ready for its peers' pushes (fence_barrier_init above)

  // ---- this thread's first item of the projection's epilogue: a pair of rows and two tokens, the last warps first ----------------
  constexpr int rpr = (int)kRows / 2, log_np = 4;                  // rows of a rank, log2 of the pairs it finishes
  const int eid = (kThreads / 32 - 1 - warp) * 32 + lane;
  const int pair = (eid >> 1) & ((1 << log_np) - 1), sub = (eid & 1) * 2;
  const int items = nq << (log_np + 1);
  const int i2 = rank * rpr + 2 * pair;                            // first column inside the head
  const float inv_t = 1.f / (float)T;
  const uint32_t new_at = smem_u32(smem + p.new_off) + (uint32_t)sec * (uint32_t)T * 128u + (uint32_t)(i2 & 7) * 2u;
  float cs[2], sn[2];
  bf16* dst[2];                             // the sequence's cache
  int slots[2];                             // row of a token there; negative: none
  uint32_t to[2];                           // row and sequence of a token, -1: none
  auto prepare = [&](int idx) {
    const int t0 = (idx >> (log_np + 1)) * 4 + sub;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int tok = min(t0 + j, p.m - 1), r = (int)(((float)tok + 0.5f) * inv_t);         // tok / t_len (exact below 2^21)
      cs[j] = 1.f;
      sn[j] = 0.f;
      slots[j] = -1;
      if (sec < 2) {
        cs[j] = __ldg(p.rope_cos + (size_t)tok * (HD / 2) + (i2 >> 1));
        sn[j] = __ldg(p.rope_sin + (size_t)tok * (HD / 2) + (i2 >> 1));
      }
      if (sec > 0) {
        slots[j] = __ldg(p.slot_pos + tok);
        dst[j] = (sec == 1 ? p.kv_k : p.kv_v) + (((size_t)p.layer * p.kv_rows + r) * p.n_heads + head) * p.s_max * HD + i2;
      }
      to[j] = (uint32_t)(tok - r * T) | (uint32_t)r << 8;
      if (idx >= items || t0 + j >= p.m) {
        to[j] = ~0u;
      }
    }
  };
  if (warp == 2 && p.ahead_bytes > 0) {
    // This CTA's share of a later projection's weights, HBM -> L2, as ordinary prefetches of 32 bytes a lane: bulk requests of 4 KB, as in
    // the other kernels, stand before the activations in the unit that loads both (18 layers, 18 tokens 338.9 -> 334.0 us, 9 tokens
    // without guidance 359.8 -> 351.9; strides of 64 and 128 bytes 334.2, 335.3.  In proj_few.cu 72 tokens 508.9 -> 512.7, in all
    // kernels 288 tokens 893.8 -> 895.1.)
    const uint32_t begin = (blockIdx.y * gridDim.x + blockIdx.x) * p.share.every, end = min(begin + p.share.bytes, p.ahead_bytes);
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (p.ahead[i])
        for (uint32_t at = begin + lane * 32u; at < end; at += 32 * 32u) prefetch_l2_sector(p.ahead[i] + at);
  }
  if (warp == 1) {
    const uint32_t idesc = idesc_bf16_f32(kRows, (uint32_t)p.nt), lo0 = desc_lo_sw128(smem_u32(smem)), stage_lo = stage_bytes >> 4;
    const uint32_t b_lo = b_bytes >> 4;
    pdl_wait();
    for (int i = 0; i < ng; ++i) {
      // (a wait that ran out is reported and the loop goes on over what is there: no lane leaves the warp)
      if (!wait_or_abort(&full_bar[i], 0, &s_abort)) {
        atomicOr(p.status, VVS_DEV_TIMEOUT);
        s_abort = 1;
      }
      tc_fence_after();
      const uint32_t a_lo = lo0 + i * stage_lo;
      const int n = min(G, nkb - i * G);
#pragma unroll 1
      for (int j = 0; j < n; ++j)
        mma_bf16_k64(tmem_base, a_lo + j * (kABytes >> 4), a_lo + G * (kABytes >> 4) + j * b_lo, idesc, (uint32_t)(i + j));
    }
    mma_commit_elect(&acc_bar);
  }
  __syncwarp();
  prepare(eid);                             // (one copy of the code for all warps: what a layer executes once has to be fetched)
  if (warp >= 2) pdl_wait();
  // ---- 1/rms of the tokens, while the MMAs run: four lanes a token, lane q of them the float4 q, q + 4, .. of its row.  (The sums are those
  // of a warp that takes a float4 a lane and adds halves of itself: slots 16, 8, 4, 2 and 1 apart.)
  if (warp >= 3) {
    const int n4 = p.ss_parts >> 2, q = lane & 3;
    for (int t0 = (warp - 3) * 8; t0 < p.m; t0 += 8 * (kThreads / 32 - 3)) {
      const int t = t0 + (lane >> 2);
      const float4* row = reinterpret_cast<const float4*>(p.ss_in + (size_t)min(t, p.m - 1) * p.ss_parts);
      float4 v[8];                          // (at most 128 sums a token: plan_qkv_attention)
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = q + 4 * k < n4 ? __ldcg(row + q + 4 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
      float a[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) a[k] = (v[k].x + v[k].y) + (v[k].z + v[k].w);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < o; ++k) a[k] += a[k + o];
      a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
      a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
      if (q == 0 && t < kFewTok) s_rs[t] = rsqrtf(a[0] * p.inv_d + p.eps);
    }
  }
  uint32_t anc[2];                          // what the rows of this warp's part see of the block
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int t = grp * 16 + (lane >> 2) + 8 * i;
    anc[i] = t < T && part < kParts ? p.anc_mask[seq * T + t] : 0u;
  }
  __syncthreads();    // s_rs
  // A CTA that gave up pushes whatever its accumulator holds: its peers' waits must still end.
  if (!wait_or_abort(&acc_bar, 0, &s_abort)) {
    if (lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
    s_abort = 1;
  }
  __syncwarp();       // each lane left the wait by itself, what follows is for a whole warp at once (.aligned)
  tc_fence_after();
  cluster_wait();
  // ---- partial sums to the rank that owns the row ------------------------------------------------------------------------
  {
    const int row_t = (warp & 3) * 16 + (lane & 15), owner = row_t >> 5;
    const uint32_t at = smem_u32(recv) + (uint32_t)(rank * rpr + (row_t & (rpr - 1))) * 16u, peer = (uint32_t)(sec * 2 + owner);
    const uint32_t recv_dst = mapa(at, peer), bar_dst = mapa(smem_u32(&recv_bar), peer);
    const uint32_t t_row = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    for (int c0 = (warp >> 2) * 2; c0 < nq; c0 += 4) {
      float v[8];
      tmem_ld8(t_row + (uint32_t)(c0 * 4), v);
#pragma unroll
      for (int j = 0; j < 2; ++j)
        if (lane < 16 && c0 + j < nq) st_async4(recv_dst + (uint32_t)(c0 + j) * (kRows * 16u), bar_dst, &v[4 * j]);
    }
  }
  if (mine) request(wg);                    // over the stages, which this CTA's MMAs are done with
  cp_async_commit();
  auto wait_cluster = [&](uint64_t* bar) {
    // peers push after waits of at most kSpinLimit polls each, so these longer waits end after their pushes
    bool got = false;
    for (uint32_t i = 0; i < 16u * kSpinLimit && !got; ++i) got = mbar_try_wait_cluster(bar, 0);
    if (!got && lane == 0) atomicOr(p.status, VVS_DEV_TIMEOUT);
    __syncwarp();     // (ldmatrix and the MMAs are .aligned too)
  };
  wait_cluster(&recv_bar);
  // ---- finished sums: 1/rms, rotation, to the CTAs that attend with them; k and v into the cache ------------------------------
  for (int idx = eid; idx < items; idx += kThreads) {
    const int quad = idx >> (log_np + 1), t0 = quad * 4 + sub;
    const uint8_t* src = recv + (size_t)quad * (kRows * 16u) + (uint32_t)(2 * pair) * 16u + (uint32_t)sub * 4u;
    float acc[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float v[2];
      ld_shared_vec(src + i * 16, acc[i]);
      ld_shared_vec(src + i * 16 + rpr * 16, v);                     // rank order
      acc[i][0] += v[0];
      acc[i][1] += v[1];
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float rs = s_rs[min(t0 + j, kFewTok - 1)];
      float a = acc[0][j] * rs, b = acc[1][j] * rs;
      const float a0 = a;
      a = a0 * cs[j] - b * sn[j];         // (1, 0 for values)
      b = a0 * sn[j] + b * cs[j];
      const uint32_t word = pack_bf16(a, b);
      if (to[j] != ~0u) {
        const uint32_t t = to[j] & 255u, first = (to[j] >> 8) * (uint32_t)p.per_item;
        const uint32_t at = new_at + t * 128u + (((uint32_t)(i2 >> 3) ^ (t & 7u)) << 4);
        for (uint32_t c = first; c < first + (uint32_t)p.per_item; ++c) st_async1(mapa(at, c), mapa(smem_u32(&new_bar), c), word);
        if (sec > 0 && slots[j] >= 0) *reinterpret_cast<uint32_t*>(dst[j] + (size_t)slots[j] * HD) = word;
      }
    }
    if (idx + kThreads < items) prepare(idx + kThreads);
  }
  tc_fence_before();

  // ---- attention: this warp's part of the item ------------------------------------------------------------------------------
  const uint32_t new_s = smem_u32(smem + p.new_off);                 // q, k, v of the sequence's block rows
  auto patch = [&](int s) {                                          // the block's own keys of slice s
    const int k_lo = max(fill, s * KS), n = min(n_keys, (s + 1) * KS) - k_lo;
    for (int at = lane; at < n * 16; at += 32) {
      const int t = k_lo + (at >> 4) - fill, k = k_lo + (at >> 4) - s * KS, is_v = (at >> 3) & 1, piece = at & 7;
      const uint4 v = *reinterpret_cast<const uint4*>(smem + p.new_off + (size_t)((1 + is_v) * T + t) * 128 + ((piece ^ (t & 7)) << 4));
      *reinterpret_cast<uint4*>(smem + (size_t)warp * kSlice + is_v * KS * 128 + k * 128 + ((piece ^ (k & 7)) << 4)) = v;
    }
  };
  const float sl2 = rsqrtf((float)HD) * 1.4426950408889634f;
  const int g = lane >> 2, c = lane & 3;
  const int ld_t = min(T, 16);                                       // rows of a part
  float* parts_o = reinterpret_cast<float*>(smem + p.part_off);      // over the stages too: [part][ld_t][kPartLd]
  float* parts_ml = parts_o + kParts * ld_t * kPartLd;               // [part][ld_t][2]
  AttState<HD> st;
  st.m[0] = st.m[1] = -CUDART_INF_F;
  st.l[0] = st.l[1] = 0.f;
#pragma unroll
  for (int j = 0; j < HD / 8; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) st.o[j][e] = 0.f;
  wait_cluster(&new_bar);
  if (mine) {
    uint32_t qa[HD / 16][4];
#pragma unroll
    for (int kk = 0; kk < HD / 16; ++kk) {
      const int row = min(grp * 16 + (lane & 15), T - 1), cc = 2 * kk + (lane >> 4);       // (rows past the block: not stored)
      ldsm4(new_s + row * 128 + (((cc & 7) ^ (row & 7)) << 4), qa[kk][0], qa[kk][1], qa[kk][2], qa[kk][3]);
    }
#pragma unroll 1
    for (int s = wg; s < n_slices; s += wpg) {
      patch(s);
      cp_async_wait<0>();
      __syncwarp();
      const int left = n_keys - s * KS, old = fill - s * KS;
      const uint32_t vmem = 0xffffffffu >> (32 - min(left, KS)), vold = old > 0 ? 0xffffffffu >> (32 - min(old, KS)) : 0u;
      uint32_t vis[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const uint32_t own = old >= KS ? 0u : old >= 0 ? anc[e] << old : anc[e] >> (-old);
        vis[e] = (vold | own) & vmem;
      }
      att_keys<HD, KS / 16, true>(st, qa, slot, slot + KS * 128u, lane, sl2, vis, vmem);
      __syncwarp();
      if (s + wpg < n_slices) request(s + wpg);
      cp_async_commit();
    }
    // its (output, maximum, normaliser) to the CTA that folds them
    const uint32_t o_to = mapa(smem_u32(parts_o), (uint32_t)gather), ml_to = mapa(smem_u32(parts_ml), (uint32_t)gather);
    const uint32_t bar_to = mapa(smem_u32(&part_bar), (uint32_t)gather);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int row = g + 8 * i;
      float l = st.l[i];
      l += __shfl_xor_sync(0xffffffffu, l, 1);
      l += __shfl_xor_sync(0xffffffffu, l, 2);
      if (grp * 16 + row < T) {
        const uint32_t at = (uint32_t)((part * ld_t + row) * kPartLd + kSeg * c) * 4u;
#pragma unroll
        for (int j = 0; j < HD / 8; j += 2) {
          const float v[4] = {st.o[j][2 * i], st.o[j][2 * i + 1], st.o[j + 1][2 * i], st.o[j + 1][2 * i + 1]};
          if (cta == gather) *reinterpret_cast<float4*>(smem + p.part_off + at + 8 * j) = make_float4(v[0], v[1], v[2], v[3]);
          else st_async4(o_to + at + 8u * j, bar_to, v);
        }
        if (c == 0) {
          if (cta == gather) *reinterpret_cast<float2*>(parts_ml + (part * ld_t + row) * 2) = make_float2(st.m[i] * sl2, l);
          else st_async2(ml_to + (uint32_t)(part * ld_t + row) * 8u, bar_to, st.m[i] * sl2, l);
        }
      }
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  if (warp == 2) tmem_dealloc(tmem_base, p.tmem_cols);
  if (cta != gather) return;
  wait_cluster(&part_bar);
  // ---- parts folded in their order ---------------------------------------------------------------------------------------------
  {
    // weights of the parts of each row, sixteen lanes a row; a part past the last one gets none
#pragma unroll 1
    for (int idx = tid; idx < (T + 1) / 2 * 32; idx += kThreads) {   // (whole warps: the second half of the last one may have no row)
      const int t = min(idx >> 4, T - 1), w = idx & 15, row = groups == 2 ? t & 15 : t;
      float2* ml = reinterpret_cast<float2*>(parts_ml) + ((groups == 2 ? (t >> 4) * wpg : 0) + min(w, wpg - 1)) * ld_t + row;
      const float mine = w < busy ? ml->x : -CUDART_INF_F;
      float m = mine;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (w < busy && idx < T * kParts) ml->x = ex2(mine - (m == -CUDART_INF_F ? 0.f : m));
    }
    __syncthreads();
  }
  for (int idx = tid; idx < T * 16; idx += kThreads) {               // a row's columns 16 jj + 2 c and 16 jj + 8 + 2 c, two each
    const int t = idx >> 4, c4 = idx & 3, jj = (idx >> 2) & 3;
    const int part_t = groups == 2 ? (t >> 4) * wpg : 0, row = groups == 2 ? t & 15 : t;
    const float* o_src = parts_o + (size_t)(part_t * ld_t + row) * kPartLd + c4 * kSeg + 4 * jj;
    const float2* ml = reinterpret_cast<const float2*>(parts_ml) + (part_t * ld_t + row);
    float l = 0.f, o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 5
    for (int w = 0; w < busy; ++w) {
      const float2 x = ml[w * ld_t];                                 // (weight, normaliser)
      l += x.y * x.x;
      const float4 y = *reinterpret_cast<const float4*>(o_src + (size_t)w * ld_t * kPartLd);
      o[0] += y.x * x.x; o[1] += y.y * x.x; o[2] += y.z * x.x; o[3] += y.w * x.x;
    }
    const float inv = l > 0.f ? 1.f / l : 0.f;                // a sequence that failed its cache check gives zeros
    bf16* out = p.out + (size_t)(seq * T + t) * p.d + head * HD + 16 * jj + 2 * c4;
    *reinterpret_cast<uint32_t*>(out) = pack2(o[0] * inv, o[1] * inv);
    *reinterpret_cast<uint32_t*>(out + 8) = pack2(o[2] * inv, o[3] * inv);
  }
}

cudaError_t launch(const QkvAttentionPlan& pl, const Params& kp, const ProjArgs& g, cudaStream_t s) {
  auto* fn = qkv_attention_kernel;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(fn), kFewSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kCtas, g.n_heads, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = pl.smem_bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCtas;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g.pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, fn, kp, *g.tm_a, *g.tm_b);
}

}  // namespace

int launch_qkv_attention(const QkvAttentionPlan& pl, const ProjArgs& g, const AttentionBlockArgs& at, cudaStream_t s) {
  Params p{};
  p.m = g.m; p.nt = pl.proj.nt; p.kb_total = pl.proj.kb_total; p.stages = pl.proj.stages; p.group = pl.proj.group;
  p.tmem_cols = (uint32_t)pl.proj.tmem_cols; p.recv_off = (uint32_t)pl.recv_off; p.part_off = (uint32_t)pl.part_off; p.new_off = (uint32_t)pl.new_off;
  p.status = g.status; p.ss_in = g.ss_in; p.ss_parts = g.ss_parts; p.inv_d = 1.f / (float)g.d; p.eps = g.eps; p.d = g.d;
  p.kv_k = g.kv_k; p.kv_v = g.kv_v; p.slot_pos = g.slot_pos; p.rope_cos = g.rope_cos; p.rope_sin = g.rope_sin;
  p.cache_len = at.cache_len; p.anc_mask = at.anc_mask; p.out = at.out;
  p.n_heads = g.n_heads; p.s_max = g.s_max; p.layer = g.layer; p.kv_rows = g.kv_rows; p.t_len = g.t_len; p.per_item = pl.per_item;
  p.ahead[0] = static_cast<const uint8_t*>(g.ahead[0]); p.ahead[1] = static_cast<const uint8_t*>(g.ahead[1]);
  p.ahead_bytes = g.ahead[0] ? g.ahead_bytes : 0;
  p.share = ahead_share(p.ahead_bytes, (uint32_t)(kCtas * g.n_heads));
  const cudaError_t e = launch(pl, p, g, s);
  return e == cudaSuccess ? VVS_OK : VVS_ERR_CUDA;
}

}  // namespace vvs
