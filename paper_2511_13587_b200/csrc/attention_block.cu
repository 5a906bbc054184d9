// Block-vs-cache attention of the decoder (bf16 contexts; Alg. 2 line 9): the T block rows of a (sequence, head)
// against the cached keys [0, fill) and, under the ancestor mask, the block's own keys, which the QKV projection has
// just written to slots fill .. fill + T - 1.
//
// One CTA per (sequence, head) -- or a cluster of S CTAs when there are few of them and the cache may be long
// (attention_split, launch_plans.h).  Every warp
// owns the slices w, w + W, ... of 16 or 32 keys and streams them through a ring of its own (cp.async, 16-byte pieces, D
// slices deep): no barrier inside the loop.  Slices of old keys are requested BEFORE griddepcontrol.wait, while the
// QKV projection is still running; after the wait only q (registers) and the one to three slices that hold new keys
// travel.  Online softmax per warp, then one merge through shared memory in warp order (and rank order), so the
// result does not depend on timing.
//
// What bounds it: with few items the dependency chain (wait, q from L2, two or three slices, merge), which is why an
// item gets as many warps as it has slices to deal; with many items the instructions a warp executes one after the other (7.4 cycles
// each; half of them were per item, not per slice).  Hence no masks on slices of old keys only, scaling and subtraction as one
// FMA, copies and merge with addresses of one add each, and the next item's first slices requested before the merge, whose
// buffer lies over the last slot of the rings only.  XL shape, 16 images (288 tokens, 640 items) 1803 -> 1724 us a step, fills of 300 to 575
// 1946 -> 1848; 8 images 1384 -> 1294, 4 images 1006 -> 958; 5 images of 27 rows each 1721 -> 1596; d_model 2048, 16 images of 4 rows
// 1800 -> 1739; one image 708 -> 702 (a cache filled to 570: 756 -> 761), a tree of 27 rows 872 -> 865.
#include "att_mma.cuh"
#include "tc_common.cuh"
#include "vvs_internal.cuh"

namespace vvs {

using namespace attmma;

namespace {

using bf16 = __nv_bfloat16;
constexpr int kMaxT = 32;      // block rows per sequence

// Shared memory: the rings of the W warps, [slot][warp]; the merge buffer lies over the last slot of them; then, in a cluster,
// the states of ranks 1 .. S-1 (written by them into rank 0).  A slice is 16 NS keys.
template <int HD, int NMT, int W, int D, int NS, bool MANY>
struct Smem {
  static constexpr int kSlice = 64 * HD * NS;                 // K, then V
  // Row of the merge buffer.  Sixteen warps: a lane's values of a row lie side by side, column 8 j + 2 c + e at c kSeg + 2 j + e, so that it
  // stores them as float4 (padded for both accesses; 18 layers of the XL shape, 18 tokens 359.0 -> 358.1 us, a tree of 54 465.4 -> 463.1).
  static constexpr bool kSide = HD == 64 && W == 16;
  static constexpr int kSeg = HD / 4 + 8, kLd = kSide ? 4 * kSeg + 4 : HD + 8;
  static constexpr int kMerge = W * NMT * 16 * (kLd + 2) * 4;
  static constexpr int kRing = D * W * kSlice, kMergeAt = MANY ? (D - 1) * W * kSlice : 0;
  static constexpr int kMain = kRing > kMergeAt + kMerge ? kRing : kMergeAt + kMerge;
  static constexpr int kQ = 32 * HD * 2;                      // the item's q: 64-column tiles, 128-byte swizzled
  static int bytes(int t_len, int s) { return kMain + kQ + (s - 1) * t_len * (HD + 2) * 4; }
};

template <int HD, int NMT, int W, int D, int NS, bool MANY>
__global__ void __launch_bounds__(32 * W) attention_block_kernel(AttentionBlockArgs a) {
  using L = Smem<HD, NMT, W, D, NS, MANY>;
  constexpr int NC = HD / 64, NJ = HD / 8, KS = 16 * NS;
  constexpr uint32_t kChunk = NS * 2048u;
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t x_bar;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, c = lane & 3;
  const int T = a.t_len, S = (int)gridDim.z, rank = (int)blockIdx.z;
  // warps are dealt to the m-tiles in groups when a warp holds one m-tile and the block has two
  const int groups = (NMT == 1 && T > 16) ? 2 : 1;
  const int wpg = W / groups, grp = warp / wpg, wg = warp - grp * wpg;
  const int first = rank * wpg + wg, stride = S * wpg;
  const uint32_t ring = tc::smem_u32(smem) + (uint32_t)warp * L::kSlice;

  if (S > 1) {
    if (tid == 0) {
      tc::mbar_init(&x_bar, 1);
      tc::fence_barrier_init();
      tc::mbar_expect_tx(&x_bar, rank == 0 ? (uint32_t)((S - 1) * T * (HD + 2) * 4) : 0u);
    }
    __syncwarp();
    tc::cluster_arrive();
  }
  const int n_items = a.n_heads * a.n_rows, G = (int)gridDim.x;
  // 16-byte pieces of a slice: this lane's first key and chunk; a step of kStep keys keeps the chunk and changes the swizzle by
  // a constant
  constexpr int kPer = HD / 8, kStep = 32 / kPer;
  const int key0 = lane / kPer, ch = lane % kPer;
  const uint32_t piece = (uint32_t)(ch >> 3) * kChunk + key0 * 128, swz = (uint32_t)((ch & 7) ^ key0) << 4;
  struct Item {
    int h, r, fill, n_keys, n_old, n_slices;                    // n_old: slices that hold old keys only
    const bf16* kp; const bf16* vp;                             // this lane's pieces of the first keys
  };
  // More items than the GPU holds CTAs: the grid is one wave, and its CTAs walk the list forth and back (longest first).
  auto item_of = [&](int k) { return k * G + ((k & 1) ? G - 1 - (int)blockIdx.x : (int)blockIdx.x); };
  auto locate = [&](int item, Item& it) {
    const int rk = item / a.n_heads;
    it.h = item - rk * a.n_heads;
    it.r = a.seq_order[rk];
    it.fill = a.cache_len[it.r];
    const bool ok = it.fill >= 0 && it.fill + T <= a.s_max;
    const size_t at = (((size_t)(a.layer * a.kv_rows + it.r) * a.n_heads + it.h) * a.s_max + key0) * HD + ch * 8;
    it.kp = a.kv_k + at;
    it.vp = a.kv_v + at;
    it.n_keys = ok ? it.fill + T : 0;
    it.n_old = ok ? it.fill / KS : 0;
    it.n_slices = (it.n_keys + KS - 1) / KS;
  };
  auto request = [&](const Item& it, int i) {                   // slice i of this warp into its ring slot
    const int s = first + i * stride, rows = it.n_keys - s * KS - key0;
    const uint32_t dst = ring + (uint32_t)(i % D) * (W * L::kSlice) + piece;
    const bf16* ks = it.kp + (size_t)s * (KS * HD);
    const bf16* vs = it.vp + (size_t)s * (KS * HD);
#pragma unroll
    for (int u = 0; u < KS / kStep; ++u)
      if (u * kStep < rows) {
        const uint32_t at = dst + u * kStep * 128 + (swz ^ (uint32_t)(((u * kStep) & 7) << 4));
        tc::cp_async16(at, ks + u * kStep * HD);
        tc::cp_async16(at + NC * kChunk, vs + u * kStep * HD);
      }
  };
  uint32_t anc[NMT][2], qa[NMT][HD / 16][4];
  auto load_anc = [&](const Item& it) {
#pragma unroll
    for (int mi = 0; mi < NMT; ++mi)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int t = (grp + mi) * 16 + g + 8 * i;
        anc[mi][i] = t < T ? a.anc_mask[it.r * T + t] : 0u;
      }
  };
  // q goes through shared memory, each piece read from L2 by one thread: as fragments, by every warp for itself, it took 1.2 us
  // of a CTA of 16 warps (one image 699 -> 687 us a step, a tree of 27 rows 863 -> 855, 5 images of 27 rows 1600 -> 1572, d_model 2048, 4
  // images 1127 -> 1112).  (Rows past the block hold whatever lies there; their results are not stored.)
  constexpr int kQP = (32 * kPer + 32 * W - 1) / (32 * W);      // pieces of a thread
  const uint32_t q_smem = tc::smem_u32(smem) + L::kMain;
  uint4 qv[kQP];
  auto load_q = [&](const Item& it) {
#pragma unroll
    for (int u = 0; u < kQP; ++u) {
      const int t = (tid + u * 32 * W) / kPer;                  // (the chunk is the same every time)
      if (t < T) qv[u] = __ldcg(reinterpret_cast<const uint4*>(a.q + (size_t)(it.r * T + t) * a.d + it.h * HD + ch * 8));
    }
  };
  auto store_q = [&]() {
#pragma unroll
    for (int u = 0; u < kQP; ++u) {
      const int t = (tid + u * 32 * W) / kPer;
      if (t < T)
        *reinterpret_cast<uint4*>(smem + L::kMain + (ch >> 3) * 4096 + t * 128 + (((ch & 7) ^ (t & 7)) << 4)) = qv[u];
    }
  };
  auto take_q = [&]() {
#pragma unroll
    for (int mi = 0; mi < NMT; ++mi)
#pragma unroll
      for (int kk = 0; kk < HD / 16; ++kk) {
        const int row = (grp + mi) * 16 + (lane & 15), cc = 2 * kk + (lane >> 4);
        ldsm4(q_smem + (cc >> 3) * 4096 + row * 128 + (((cc & 7) ^ (row & 7)) << 4), qa[mi][kk][0], qa[mi][kk][1], qa[mi][kk][2],
              qa[mi][kk][3]);
      }
  };
  const float sl2 = rsqrtf((float)HD) * 1.4426950408889634f;

  // ---- the first item: slices of old keys before the wait ---------------------------------------------------------------
  Item it;
  locate(item_of(0), it);                                       // (the grid has no more CTAs than items)
#pragma unroll
  for (int i = 0; i < D; ++i) {
    if (first + i * stride < it.n_old) request(it, i);
    tc::cp_async_commit();
  }
  tc::pdl_launch_dependents();                  // the projection after this kernel may start fetching its weights
  load_anc(it);
  tc::pdl_wait();
  load_q(it);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const int s = first + i * stride;
    if (s >= it.n_old && s < it.n_slices) request(it, i);
  }
  tc::cp_async_commit();
  store_q();
  __syncthreads();

#pragma unroll 1
  for (int k = 0;; ++k) {
    const int next_item = item_of(k + 1);
    const bool more = MANY && next_item < n_items;
    Item nx;
    if (more) locate(next_item, nx);
    take_q();
    AttState<HD> st[NMT];
#pragma unroll
    for (int mi = 0; mi < NMT; ++mi) {
      st[mi].m[0] = st[mi].m[1] = -CUDART_INF_F;
      st[mi].l[0] = st[mi].l[1] = 0.f;
#pragma unroll
      for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) st[mi].o[j][e] = 0.f;
    }
#pragma unroll 1
    for (int i = 0; first + i * stride < it.n_slices; ++i) {
      const int s = first + i * stride;
      const uint32_t k_base = ring + (uint32_t)(i % D) * (W * L::kSlice), v_base = k_base + NC * kChunk;
      // groups so far: D for the first slices, one more, one per iteration; slice i is in one of the oldest i + 2 of them
      // unless it was requested after the wait
      if (MANY && s < it.n_old) {
        tc::cp_async_wait<D - 1>();
        __syncwarp();
        const uint32_t all[2] = {0u, 0u};
#pragma unroll
        for (int mi = 0; mi < NMT; ++mi) att_keys<HD, NS, false>(st[mi], qa[mi], k_base, v_base, lane, sl2, all, 0u);
      } else {
        if (MANY || s >= it.n_old) tc::cp_async_wait<0>(); else tc::cp_async_wait<D - 1>();
        __syncwarp();
        const int left = it.n_keys - s * KS, old = it.fill - s * KS;      // valid keys of the slice (at least one); old ones among them
        const uint32_t vmem = 0xffffffffu >> (32 - min(left, KS)), vold = old > 0 ? 0xffffffffu >> (32 - min(old, KS)) : 0u;
#pragma unroll
        for (int mi = 0; mi < NMT; ++mi) {
          uint32_t vis[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const uint32_t own = old >= KS ? 0u : old >= 0 ? anc[mi][e] << old : anc[mi][e] >> (-old);
            vis[e] = (vold | own) & vmem;
          }
          att_keys<HD, NS, true>(st[mi], qa[mi], k_base, v_base, lane, sl2, vis, vmem);
        }
      }
      __syncwarp();                                             // every lane is done with the ring slot
      if (first + (i + D) * stride < it.n_slices) request(it, i + D);
      tc::cp_async_commit();
    }
    // ---- this warp's part of the next item: all slots but the last, over which the merge buffer lies --
    if (more) {
#pragma unroll
      for (int i = 0; i < D - 1; ++i) {
        if (first + i * stride < nx.n_slices) request(nx, i);
        tc::cp_async_commit();
      }
    }
    // ---- merge: every warp that had keys leaves (max, normaliser, output) of its rows, the CTA folds them in warp order --
    const int busy = min(wpg, max(it.n_slices - rank * wpg, 0));
    __syncthreads();                                            // the last slots have drained everywhere
    float* s_o = reinterpret_cast<float*>(smem + L::kMergeAt);  // [W][NMT * 16][kLd]
    float* s_ml = s_o + W * NMT * 16 * L::kLd;                  // [W][NMT * 16][2]
    if (wg < busy) {
#pragma unroll
      for (int mi = 0; mi < NMT; ++mi)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int row = mi * 16 + g + 8 * i;
          float l = st[mi].l[i];
          l += __shfl_xor_sync(0xffffffffu, l, 1);
          l += __shfl_xor_sync(0xffffffffu, l, 2);
          if ((grp + mi) * 16 + g + 8 * i < T) {
            float* dst = s_o + (size_t)(warp * NMT * 16 + row) * L::kLd + (L::kSide ? L::kSeg : 2) * c;
            if constexpr (L::kSide) {
#pragma unroll
              for (int j = 0; j < NJ; j += 2)
                *reinterpret_cast<float4*>(dst + 2 * j) =
                    make_float4(st[mi].o[j][2 * i], st[mi].o[j][2 * i + 1], st[mi].o[j + 1][2 * i], st[mi].o[j + 1][2 * i + 1]);
            } else {
#pragma unroll
              for (int j = 0; j < NJ; ++j) *reinterpret_cast<float2*>(dst + 8 * j) = make_float2(st[mi].o[j][2 * i], st[mi].o[j][2 * i + 1]);
            }
            if (c == 0) *reinterpret_cast<float2*>(s_ml + (warp * NMT * 16 + row) * 2) = make_float2(HD == 128 ? st[mi].m[i] : st[mi].m[i] * sl2, l);
          }
        }
    }
    const int h = it.h, r = it.r;
    if (more) {
      it = nx;
      load_anc(it);
      load_q(it);
    }
    __syncthreads();
    if (S > 1) tc::cluster_wait();   // rank 0's barrier is ready
    float* xbuf = reinterpret_cast<float*>(smem + L::kMain + L::kQ);    // [S - 1][T][HD + 2]
    const uint32_t x_bar0 = S > 1 ? tc::mapa(tc::smem_u32(&x_bar), 0) : 0u;
    const uint32_t xbuf0 = S > 1 ? tc::mapa(tc::smem_u32(xbuf), 0) : 0u;
    bool waited = S == 1;
    constexpr int CP = W > 4 ? 2 : 8;                          // columns per item of the merge
    for (int idx = tid; idx < T * (HD / CP); idx += 32 * W) {
      const int t = idx / (HD / CP), cp = idx - t * (HD / CP);
      const int grp_t = groups == 2 ? t >> 4 : 0, row = groups == 2 ? t & 15 : t;
      const float* o_src = s_o + (size_t)(grp_t * wpg * NMT * 16 + row) * L::kLd + (L::kSide ? (cp & 3) * L::kSeg + 2 * (cp >> 2) : CP * cp);
      const float2* ml = reinterpret_cast<const float2*>(s_ml) + (grp_t * wpg * NMT * 16 + row);
      float m = -CUDART_INF_F;
#pragma unroll 4
      for (int w = 0; w < busy; ++w) m = fmaxf(m, ml[w * NMT * 16].x);
      const float m_safe = m == -CUDART_INF_F ? 0.f : m;
      float l = 0.f, o[CP];
#pragma unroll
      for (int e = 0; e < CP; ++e) o[e] = 0.f;
#pragma unroll 4
      for (int w = 0; w < busy; ++w) {
        const float2 x = ml[w * NMT * 16];
        const float f = ex2(x.x - m_safe);
        l += x.y * f;
        const float* v = o_src + (size_t)w * NMT * 16 * L::kLd;
        if constexpr (CP == 2) {
          const float2 y = *reinterpret_cast<const float2*>(v);
          o[0] += y.x * f;
          o[1] += y.y * f;
        } else {
#pragma unroll
          for (int e = 0; e < CP; e += 4) {
            const float4 y = *reinterpret_cast<const float4*>(v + e);
            o[e] += y.x * f; o[e + 1] += y.y * f; o[e + 2] += y.z * f; o[e + 3] += y.w * f;
          }
        }
      }
      bf16* out = a.out + (size_t)(r * T + t) * a.d + h * HD + CP * cp;
      if constexpr (CP == 2) {
        if (rank > 0) {
          const uint32_t dst = xbuf0 + (uint32_t)(((rank - 1) * T + t) * (HD + 2)) * 4u;
          tc::st_async2(dst + (uint32_t)cp * 8u, x_bar0, o[0], o[1]);
          if (cp == 0) tc::st_async2(dst + HD * 4u, x_bar0, m, l);
          continue;
        }
        if (!waited) {
          // the peers' loops hold no unbounded wait; the limit only guards against a CTA that never runs
          bool got = false;
          for (uint32_t i = 0; i < 4u * tc::kSpinLimit && !got; ++i) got = tc::mbar_try_wait_cluster(&x_bar, 0);
          if (!got) atomicOr(a.status, VVS_DEV_TIMEOUT);
          waited = true;
        }
        for (int q = 0; q < S - 1; ++q) {
          const float* x = xbuf + (size_t)(q * T + t) * (HD + 2);
          const float mo = x[HD], lo = x[HD + 1];
          const float m_new = fmaxf(m, mo), ms = m_new == -CUDART_INF_F ? 0.f : m_new;
          const float aa = ex2(m - ms), bb = ex2(mo - ms);
          m = m_new;
          l = l * aa + lo * bb;
          o[0] = o[0] * aa + x[2 * cp] * bb;
          o[1] = o[1] * aa + x[2 * cp + 1] * bb;
        }
      }
      const float inv = l > 0.f ? 1.f / l : 0.f;                // a sequence that failed its cache check gives zeros
      if constexpr (CP == 2) {
        *reinterpret_cast<uint32_t*>(out) = pack2(o[0] * inv, o[1] * inv);
      } else {
        *reinterpret_cast<uint4*>(out) = make_uint4(pack2(o[0] * inv, o[1] * inv), pack2(o[2] * inv, o[3] * inv),
                                                    pack2(o[4] * inv, o[5] * inv), pack2(o[6] * inv, o[7] * inv));
      }
    }
    if (!more) break;
    store_q();
    __syncthreads();                                            // q; the merge is done with the last slots
    if (first + (D - 1) * stride < it.n_slices) request(it, D - 1);
    tc::cp_async_commit();
    tc::cp_async_commit();                                      // (as many groups as the first item has)
  }
}

template <int HD, int NMT, int W, int D, int NS, bool MANY>
int launch_variant(const AttentionBlockArgs& a, int split, int per_sm, cudaStream_t s) {
  using L = Smem<HD, NMT, W, D, NS, MANY>;
  const void* fn = reinterpret_cast<const void*>(attention_block_kernel<HD, NMT, W, D, NS, MANY>);
  if (ensure_dynamic_smem(fn, L::bytes(kMaxT, split)) != cudaSuccess) return VVS_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  int ctas = a.n_heads * a.n_rows;
  if (split == 1 && ctas > per_sm * a.n_sms) ctas = per_sm * a.n_sms;
  cfg.gridDim = dim3(ctas, 1, split);
  cfg.blockDim = dim3(32 * W, 1, 1);
  cfg.dynamicSmemBytes = L::bytes(a.t_len, split);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (a.pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (split > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = 1;
    attr[na].val.clusterDim.y = 1;
    attr[na++].val.clusterDim.z = (unsigned)split;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, attention_block_kernel<HD, NMT, W, D, NS, MANY>, a) == cudaSuccess ? VVS_OK : VVS_ERR_CUDA;
}

}  // namespace

// CTAs per item: attention_split (launch_plans.h).  Warps per item by how many items there are: with few, one item's slices over
// many warps (XL shape, one image: 16 warps with a slot of 32 keys each 702 us a step, with two of 16 keys 721, 14 warps 698 but 886
// where they are dealt to two row groups (16: 863), 8 warps with two slots 713); with many, small CTAs: four warps with three slots of 16 keys,
// three CTAs per SM (16 images 1724, 8 images 1294, 4 images 958; four CTAs per SM with two slots 1716, 1329 and 1021; three with two slots
// of 32 keys 1766, 1294 and 959), two m-tiles a warp beyond 16 rows (5 images of 27 rows, two slots of 32 keys 1596, three of 16 keys 1624).
// Heads of 128 (see att_keys): up to two items per SM take eight warps, more take four, since the warps' shares of the keys decide in
// which order the sums are taken (224 items would take 1378 us a step with four, 1398 with eight).
int launch_attention_block(const AttentionBlockArgs& a, cudaStream_t s) {
  if (a.t_len > kMaxT) return VVS_ERR_SHAPE;
  const long long items = (long long)a.n_heads * a.n_rows;
  const int split = attention_split(a.hd, items, a.s_max, a.n_sms);
  if (a.hd == 64) {
    if (items <= a.n_sms) return launch_variant<64, 1, 16, 1, 2, false>(a, split, 1, s);
    return a.t_len > 16 ? launch_variant<64, 2, 4, 2, 2, true>(a, split, 2, s) : launch_variant<64, 1, 4, 3, 1, true>(a, split, 3, s);
  }
  if (a.hd == 128)
    return items <= 2LL * a.n_sms ? launch_variant<128, 1, 8, 2, 1, true>(a, split, 1, s) : launch_variant<128, 1, 4, 3, 1, true>(a, split, 2, s);
  return VVS_ERR_SHAPE;
}

}  // namespace vvs
