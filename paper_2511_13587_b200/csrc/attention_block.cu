// Block-vs-cache attention of the decoder (bf16 contexts; Alg. 2 line 9): the T block rows of a (sequence, head)
// against the cached keys [0, fill) and, under the ancestor mask, the block's own keys, which the QKV projection has
// just written to slots fill .. fill + T - 1.
//
// One CTA per (sequence, head) -- or a cluster of S CTAs when there are few of them and the cache may be long
// (attention_split, launch_plans.h).  Every warp
// owns the 16-key slices w, w + W, ... and streams them through a ring of its own (cp.async, 16-byte pieces, D
// slices deep): no barrier inside the loop.  Slices of old keys are requested BEFORE griddepcontrol.wait, while the
// QKV projection is still running; after the wait only q (registers) and the one to three slices that hold new keys
// travel.  Online softmax per warp, then one merge through shared memory in warp order (and rank order), so the
// result does not depend on timing.
//
// What bounds it: with few items the dependency chain (wait, q from L2, two or three slices, merge), which is why an
// item gets as many warps as it has slices to deal; with many items the K / V stream.
#include "att_mma.cuh"
#include "tc_common.cuh"
#include "vvs_internal.cuh"

namespace vvs {

using namespace attmma;

namespace {

using bf16 = __nv_bfloat16;
constexpr int kMaxT = 32;      // block rows per sequence

__device__ __forceinline__ void st_async2(uint32_t addr, uint32_t bar, float a, float b) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];"
               ::"r"(addr), "f"(a), "f"(b), "r"(bar) : "memory");
}

// shared memory: rings of the W warps, over which the merge buffers lie afterwards; then, in a cluster, the states of
// ranks 1 .. S-1 (written by them into rank 0)
template <int HD, int NMT, int W, int D>
struct Smem {
  static constexpr int kSlice = 64 * HD;                      // 16 keys, K and V
  static constexpr int kRing = W * D * kSlice;
  static constexpr int kLd = HD + 8;                          // padded row of the merge buffer
  static constexpr int kMerge = W * NMT * 16 * (kLd + 2) * 4;
  static constexpr int kMain = kRing > kMerge ? kRing : kMerge;
  static int bytes(int t_len, int s) { return kMain + (s - 1) * t_len * (HD + 2) * 4; }
};

template <int HD, int NMT, int W, int D>
__global__ void __launch_bounds__(32 * W) attention_block_kernel(AttentionBlockArgs a) {
  using L = Smem<HD, NMT, W, D>;
  constexpr int NC = HD / 64, NJ = HD / 8;
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t x_bar;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, c = lane & 3;
  const int T = a.t_len, S = (int)gridDim.z, rank = (int)blockIdx.z;
  // warps are dealt to the m-tiles in groups when a warp holds one m-tile and the block has two
  const int groups = (NMT == 1 && T > 16) ? 2 : 1;
  const int wpg = W / groups, grp = warp / wpg, wg = warp - grp * wpg;
  const int first = rank * wpg + wg, stride = S * wpg;
  const uint32_t ring = tc::smem_u32(smem) + (uint32_t)(warp * D) * L::kSlice;

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
  // More items than the GPU holds CTAs: the grid is one wave, and its CTAs walk the list forth and back (longest first).
#pragma unroll 1
  for (int k = 0;; ++k) {
    const int item = k * G + ((k & 1) ? G - 1 - (int)blockIdx.x : (int)blockIdx.x);
    if (item >= n_items) break;
    const int h = item % a.n_heads, r = a.seq_order[item / a.n_heads];
    const int fill = a.cache_len[r];
    const bool ok = fill >= 0 && fill + T <= a.s_max;
    const size_t row_base = ((size_t)(a.layer * a.kv_rows + r) * a.n_heads + h) * a.s_max;
    const bf16* kp = a.kv_k + row_base * HD;
    const bf16* vp = a.kv_v + row_base * HD;
    const int n_keys = ok ? fill + T : 0;
    const int n_old = ok ? fill >> 4 : 0;                       // slices that hold old keys only
    const int n_slices = (n_keys + 15) >> 4;
    if (k > 0) __syncthreads();                                 // the merge of the item before is done with the rings
    auto request = [&](int i) {                                 // slice i of this warp into its ring slot
      const int s = first + i * stride;
      const uint32_t dst0 = ring + (uint32_t)(i % D) * L::kSlice;
      const int rows = min(16, n_keys - s * 16);
      constexpr int per_row = HD / 8;                           // 16-byte pieces
#pragma unroll
      for (int u = 0; u < 2 * 16 * per_row / 32; ++u) {
        const int idx = lane + u * 32, which = idx / (16 * per_row), rem = idx - which * 16 * per_row;
        const int key = rem / per_row, ch = rem - key * per_row;
        if (key < rows)
          tc::cp_async16(dst0 + (uint32_t)(which * NC + (ch >> 3)) * 2048u + key * 128 + (((ch & 7) ^ (key & 7)) << 4),
                     (which ? vp : kp) + (size_t)(s * 16 + key) * HD + ch * 8);
      }
    };
#pragma unroll
    for (int i = 0; i < D; ++i) {
      if (first + i * stride < n_old) request(i);
      tc::cp_async_commit();
    }
    if (k == 0) tc::pdl_launch_dependents();      // the projection after this kernel may start fetching its weights
    uint32_t anc[NMT][2];
#pragma unroll
    for (int mi = 0; mi < NMT; ++mi)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int t = (grp + mi) * 16 + g + 8 * i;
        anc[mi][i] = t < T ? a.anc_mask[r * T + t] : 0u;
      }
    if (k == 0) tc::pdl_wait();
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const int s = first + i * stride;
      if (s >= n_old && s < n_slices) request(i);
    }
    tc::cp_async_commit();
    uint32_t qa[NMT][HD / 16][4];
#pragma unroll
    for (int mi = 0; mi < NMT; ++mi) {
      const int t0 = (grp + mi) * 16 + g, t1 = t0 + 8;
      const bf16* q0 = a.q + (size_t)(r * T + t0) * a.d + h * HD + 2 * c;
      const bf16* q1 = q0 + (size_t)8 * a.d;
#pragma unroll
      for (int kk = 0; kk < HD / 16; ++kk) {
        qa[mi][kk][0] = t0 < T ? __ldcg(reinterpret_cast<const unsigned*>(q0 + 16 * kk)) : 0u;
        qa[mi][kk][1] = t1 < T ? __ldcg(reinterpret_cast<const unsigned*>(q1 + 16 * kk)) : 0u;
        qa[mi][kk][2] = t0 < T ? __ldcg(reinterpret_cast<const unsigned*>(q0 + 16 * kk + 8)) : 0u;
        qa[mi][kk][3] = t1 < T ? __ldcg(reinterpret_cast<const unsigned*>(q1 + 16 * kk + 8)) : 0u;
      }
    }
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
    const float sl2 = rsqrtf((float)HD) * 1.4426950408889634f;

#pragma unroll 1
    for (int i = 0; first + i * stride < n_slices; ++i) {
      const int s = first + i * stride;
      // groups so far: D before the wait, one after it, one per iteration; slice i is in one of the oldest i + 2 of them
      // unless it was requested after the wait
      if (s >= n_old) tc::cp_async_wait<0>(); else tc::cp_async_wait<D - 1>();
      __syncwarp();
      const uint32_t k_base = ring + (uint32_t)(i % D) * L::kSlice, v_base = k_base + NC * 2048u;
      const int left = n_keys - s * 16, old = fill - s * 16;    // valid keys of the slice; old ones among them
      const uint32_t vmem = left >= 16 ? 0xffffu : ((1u << left) - 1u);
      const uint32_t vold = old >= 16 ? 0xffffu : old > 0 ? ((1u << old) - 1u) : 0u;
#pragma unroll
      for (int mi = 0; mi < NMT; ++mi) {
        uint32_t vis[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const uint32_t own = old >= 16 ? 0u : old >= 0 ? anc[mi][e] << old : anc[mi][e] >> (-old);
          vis[e] = (vold | own) & vmem;
        }
        att_slice<HD>(st[mi], qa[mi], k_base, v_base, 2048u, 0, lane, sl2, vis, vmem);
      }
      __syncwarp();                                             // every lane is done with the ring slot
      if (first + (i + D) * stride < n_slices) request(i + D);
      tc::cp_async_commit();
    }
    tc::cp_async_wait<0>();
    // ---- merge: every warp leaves (max, normaliser, output) of its rows, the CTA folds them in warp order --
    __syncthreads();                                            // the rings have drained everywhere
    float* s_o = reinterpret_cast<float*>(smem);                // [W][NMT * 16][kLd]
    float* s_ml = s_o + W * NMT * 16 * L::kLd;                  // [W][NMT * 16][2]
#pragma unroll
    for (int mi = 0; mi < NMT; ++mi)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int row = mi * 16 + g + 8 * i;
        float l = st[mi].l[i];
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        if ((grp + mi) * 16 + g + 8 * i < T) {
          float* dst = s_o + (size_t)(warp * NMT * 16 + row) * L::kLd + 2 * c;
#pragma unroll
          for (int j = 0; j < NJ; ++j) *reinterpret_cast<float2*>(dst + 8 * j) = make_float2(st[mi].o[j][2 * i], st[mi].o[j][2 * i + 1]);
          if (c == 0) {
            s_ml[(warp * NMT * 16 + row) * 2] = st[mi].m[i];
            s_ml[(warp * NMT * 16 + row) * 2 + 1] = l;
          }
        }
      }
    __syncthreads();
    if (S > 1) tc::cluster_wait();   // rank 0's barrier is ready
    float* xbuf = reinterpret_cast<float*>(smem + L::kMain);    // [S - 1][T][HD + 2]
    const uint32_t x_bar0 = S > 1 ? tc::mapa(tc::smem_u32(&x_bar), 0) : 0u;
    const uint32_t xbuf0 = S > 1 ? tc::mapa(tc::smem_u32(xbuf), 0) : 0u;
    bool waited = S == 1;
    for (int idx = tid; idx < T * (HD / 2); idx += 32 * W) {
      const int t = idx / (HD / 2), cp = idx - t * (HD / 2);
      const int grp_t = groups == 2 ? t >> 4 : 0, row = groups == 2 ? t & 15 : t;
      const float* o_src = s_o + (size_t)(grp_t * wpg * NMT * 16 + row) * L::kLd + 2 * cp;
      const float* ml = s_ml + (grp_t * wpg * NMT * 16 + row) * 2;
      float m = -CUDART_INF_F;
#pragma unroll 4
      for (int w = 0; w < wpg; ++w) m = fmaxf(m, ml[w * NMT * 32]);
      const float m_safe = m == -CUDART_INF_F ? 0.f : m;
      float l = 0.f, o0 = 0.f, o1 = 0.f;
#pragma unroll 4
      for (int w = 0; w < wpg; ++w) {
        const float f = ex2(ml[w * NMT * 32] - m_safe);
        const float2 v = *reinterpret_cast<const float2*>(o_src + (size_t)w * NMT * 16 * L::kLd);
        l += ml[w * NMT * 32 + 1] * f;
        o0 += v.x * f;
        o1 += v.y * f;
      }
      if (rank > 0) {
        const uint32_t dst = xbuf0 + (uint32_t)(((rank - 1) * T + t) * (HD + 2)) * 4u;
        st_async2(dst + (uint32_t)cp * 8u, x_bar0, o0, o1);
        if (cp == 0) st_async2(dst + HD * 4u, x_bar0, m, l);
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
        o0 = o0 * aa + x[2 * cp] * bb;
        o1 = o1 * aa + x[2 * cp + 1] * bb;
      }
      const float inv = l > 0.f ? 1.f / l : 0.f;                // a sequence that failed its cache check gives zeros
      *reinterpret_cast<uint32_t*>(a.out + (size_t)(r * T + t) * a.d + h * HD + 2 * cp) = pack2(o0 * inv, o1 * inv);
    }
  }
}

template <int HD, int NMT, int W, int D>
int launch_variant(const AttentionBlockArgs& a, int split, int per_sm, cudaStream_t s) {
  using L = Smem<HD, NMT, W, D>;
  const void* fn = reinterpret_cast<const void*>(attention_block_kernel<HD, NMT, W, D>);
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
  return cudaLaunchKernelEx(&cfg, attention_block_kernel<HD, NMT, W, D>, a) == cudaSuccess ? VVS_OK : VVS_ERR_CUDA;
}

}  // namespace

// CTAs per item: attention_split (launch_plans.h).  Warps per item by how many items there are: with few, one item's slices over many warps (XL shape, step of 18 tokens
// with 16, 8 and 4 warps 962, 1004 and 1013 us; 54 tokens, two row groups of 8 warps 1184, of 4 warps 1286, four warps
// with two m-tiles each 1272); with many, small CTAs (288 tokens, 640 items: 4 warps, three CTAs per SM 1.88 ms, 8 warps
// 2.07 ms).  The item loop let the compiler keep addresses in registers: 160 instead of 128 a thread, three CTAs per SM
// instead of four, and all the same 1.97 -> 1.88 ms (7B shape 3.13 -> 3.08 ms).
int launch_attention_block(const AttentionBlockArgs& a, cudaStream_t s) {
  if (a.t_len > kMaxT) return VVS_ERR_SHAPE;
  const long long items = (long long)a.n_heads * a.n_rows;
  const bool few = items <= a.n_sms, some = items <= 2LL * a.n_sms;
  const int split = attention_split(a.hd, items, a.s_max, a.n_sms);
  if (a.hd == 64) {
    if (few) return launch_variant<64, 1, 16, 2>(a, split, 1, s);
    if (a.t_len > 16) return launch_variant<64, 2, 4, 3>(a, split, 2, s);
    return some ? launch_variant<64, 1, 8, 3>(a, split, 2, s) : launch_variant<64, 1, 4, 3>(a, split, 3, s);
  }
  if (a.hd == 128) return some ? launch_variant<128, 1, 8, 2>(a, split, 1, s) : launch_variant<128, 1, 4, 3>(a, split, 2, s);
  return VVS_ERR_SHAPE;
}

}  // namespace vvs
