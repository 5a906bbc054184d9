// Verification of a candidate TREE (the drafter of the paper proposes a token tree, Sec. 5):
// multi-round speculative sampling over the children of the current node, which are taken to be
// independent draws from the drafter's distribution q at that node.  A child x passes iff
// u < min(1, p_res(x) / q(x)); a rejection replaces p_res by norm(max(0, p_res - q)); when no
// child is left the next token is drawn from the last residual.  A chain-shaped tree reduces to
// the chain rule of Sec. 2 bit for bit: the first residual is the float32 difference of the two
// float32 rows, later rounds (which a chain never reaches) work in float64.
// Relaxed mode: the numerator is the pooled mass of x and its neighbours in the current p_res
// (the chain's relaxed rule with p_res in the place of p); with the adjusted-residual flag a
// rejection subtracts q from p_res after the pooled neighbours' mass has been moved onto x.
//
// One CTA per image, or a cluster of S for larger codebooks (tree_walk_parts, launch_plans.h), each with a contiguous part of
// the codes; the walk is sequential over tree depth and siblings and every CTA takes it, each residual update and the final
// inverse-CDF draw are passes over the parts whose sums are exchanged through distributed shared memory and added in rank
// order, so a call repeats bit for bit on the same probabilities.  What bounds it: the chain of tests and passes; a cluster
// pays one barrier per rejection and two for the draw, a pass of 16384 codes on one SM (float64 units and loads) 7 us.
// 26 nodes, most rejected, before with one CTA each / now: 4 images x 4096 codes 23.8 / 23.1 us, x 16384 67.6 / 24.2, 8 images
// x 32768 123 / 30; most accepted 11.3 / 11.2, 19.8 / 13.3, 45.2 / 13.8.
#include <math_constants.h>

#include "tc_common.cuh"
#include "vvs_internal.cuh"

namespace vvs {

namespace {

constexpr int kTreeThreads = 1024;

__device__ __forceinline__ double tw_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double tw_warp_scan(double v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Longest distance-ordered prefix of neighbour entries 1 .. kk-1 whose cumulative mass stays
// <= delta (one warp; the pooled mass in every lane, the first entry not pooled in *j_end).
template <typename F>
__device__ __forceinline__ double tw_pooled_prefix(int kk, double delta, int lane, F pn_of, int* j_end) {
  double cum = 0.0;
  int end = kk;
  for (int j0 = 1; j0 < kk; j0 += 32) {
    const int j = j0 + lane;
    const double pn = (j < kk) ? pn_of(j) : 0.0;
    const double tot = cum + tw_warp_scan(pn, lane);
    const unsigned over = __ballot_sync(0xffffffffu, (j < kk) && (tot > delta));
    if (over) {
      const int first = __ffs(over) - 1;
      const double prev = __shfl_sync(0xffffffffu, tot, first > 0 ? first - 1 : 0);
      if (first > 0) cum = prev;
      end = j0 + first;
      break;
    }
    cum = __shfl_sync(0xffffffffu, tot, 31);
  }
  *j_end = end;
  return cum;
}

// Sum over the block, the same value in every thread (two barriers).
__device__ double tw_block_sum(double v, double* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = tw_warp_sum(v);
  __syncthreads();
  if (lane == 0) s_warp[warp] = v;
  __syncthreads();
  double tot = 0.0;
  for (int w = 0; w < kTreeThreads / 32; ++w) tot += s_warp[w];
  return tot;
}

// The sum of the CTAs' values at *slot, in rank order.  Consecutive calls take two slots in turn: a CTA that writes a slot
// again has met every reader of it at the barrier of the call between.  The barrier also publishes what the CTAs have
// written to global memory.
__device__ __forceinline__ double tw_exchange(double v, double* slot, int S) {
  if (threadIdx.x == 0) *slot = v;
  tc::cluster_sync();
  double tot = 0.0;
  for (int r = 0; r < S; ++r) tot += tc::ld_cluster_f64(slot, (uint32_t)r);
  return tot;
}

// CLUSTER: several CTAs per image; else one, which needs none of the barriers and exchanges between them.
template <bool CLUSTER>
__global__ void __launch_bounds__(kTreeThreads) tree_walk_kernel(TreeParams p) {
  __shared__ double s_warp[kTreeThreads / 32], s_slot[2];
  __shared__ int s_child[32];
  __shared__ int s_n, s_pass, s_first, s_last, s_jend;
  __shared__ double s_mass;
  const int b = blockIdx.y, S = CLUSTER ? (int)gridDim.x : 1, rank = CLUSTER ? (int)blockIdx.x : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int F = p.n_forced, K = p.n_draft_max, T = p.t_len, V = p.vocab;
  const int32_t* par = p.parent + (size_t)b * T;
  double* buf[2] = {p.res + (size_t)b * V, p.res + ((size_t)p.n_images + b) * V};

  const int part = (V + S - 1) / S, r0 = min(V, rank * part), r1 = min(V, r0 + part);   // this CTA's codes
  int turn = 0;
  auto residual_at = [](const double* r) { return CLUSTER ? __ldcg(r) : *r; };          // (another CTA's part, maybe)
  if (rank == 0 && tid == 0) {
    for (int i = 0; i <= K; ++i)
      if (p.margins) p.margins[(size_t)b * (K + 1) + i] = CUDART_INF_F;
    for (int i = 0; i < K; ++i) {
      if (p.accept_mask) p.accept_mask[(size_t)b * K + i] = 0;
      p.accept_path[(size_t)b * K + i] = -1;
    }
  }
  int cur = F - 1, n_acc = 0;
  int src = -1;                 // -1: sample from the float32 row of `cur`; else from buf[src]
  const float* prow = nullptr;
#pragma unroll 1
  for (int level = 0; level <= K; ++level) {
    __syncthreads();
    if (tid == 0) {
      int n = 0;
      for (int c = F; c < T; ++c)
        if (par[c] == cur) s_child[n++] = c;
      s_n = n;
    }
    __syncthreads();
    const int n_child = s_n;
    prow = p.probs + ((size_t)b * T + cur) * V;
    src = -1;
    if (n_child == 0) break;                      // leaf: the bonus token comes from its own row
    bool first_round = true;
    double z = 1.0;
    int accepted = -1;
#pragma unroll 1
    for (int ci = 0; ci < n_child; ++ci) {
      const int c = s_child[ci], i = c - F;
      const float* qrow = p.draft_probs + ((size_t)b * K + i) * V;
      const int x = p.drafts[(size_t)b * p.drafts_ld + i] - p.vocab_offset;
      const bool x_ok = x >= 0 && x < V;
      if (warp == 0) {
        int pass = 0;
        if (!x_ok) {
          if (lane == 0) atomicOr(p.status, VVS_DEV_BAD_TOKEN);
        } else {
          double px = first_round ? (double)prow[x] : residual_at(buf[src] + x) / z;
          int j_end = 1;
          if (p.relaxed) {
            const int beg = p.row_ptr[x], len = p.row_ptr[x + 1] - beg;
            if (len < 1 && lane == 0) atomicOr(p.status, VVS_DEV_BAD_NEIGHBOUR);
            const int kk = min(p.nbr_k, len);
            const double* cur_res = first_round ? nullptr : buf[src];
            px += tw_pooled_prefix(kk, (double)p.delta, lane, [&](int j) {
              const int cc = p.col[beg + j];
              if (cc < 0 || cc >= V) return 0.0;
              return cur_res ? residual_at(cur_res + cc) / z : (double)prow[cc]; }, &j_end);
          }
          const double qx = (double)qrow[x];
          const double ratio = qx > 0.0 ? fmin(1.0, px / qx) : (px > 0.0 ? 1.0 : 0.0);
          const double u = (double)p.uniforms[(size_t)b * (K + 1) + i];
          if (rank == 0 && lane == 0 && p.margins) p.margins[(size_t)b * (K + 1) + i] = (float)fabs(u - ratio);
          pass = u < ratio ? 1 : 0;
          if (lane == 0) {
            s_mass = px;
            s_jend = j_end;
          }
        }
        if (lane == 0) s_pass = pass;
      }
      __syncthreads();
      if (s_pass) {
        // the next level's first residual may go where a slower CTA is still reading this one's; a rejection writes the other
        // buffer, whose readers have all met at the exchange before
        if (CLUSTER && src >= 0) tc::cluster_sync();
        accepted = c;
        break;
      }
      if (!x_ok) {
        __syncthreads();                          // s_pass is written again
        continue;
      }
      // rejected: residual of this round
      double* dst = buf[src < 0 ? 0 : (src ^ 1)];
      double local = 0.0;
      if (first_round) {
        for (int v = r0 + tid; v < r1; v += kTreeThreads) {
          const double r = (double)fmaxf(0.f, __fsub_rn(prow[v], qrow[v]));
          dst[v] = r;
          local += r;
        }
      } else {
        const double* cur_res = buf[src];
        for (int v = r0 + tid; v < r1; v += kTreeThreads) {
          const double r = fmax(0.0, __dsub_rn(cur_res[v] / z, (double)qrow[v]));
          dst[v] = r;
          local += r;
        }
      }
      if (p.adjusted) {
        // adjusted target of the rejected child: its pooled neighbours carry no mass, the child
        // carries the pooled mass; the touched entries are rewritten and the sum is taken again
        __syncthreads();
        const int beg = p.row_ptr[x];
        const int j_end = s_jend;
        for (int j = 1 + tid; j < j_end; j += kTreeThreads) {
          const int cc = p.col[beg + j];
          if (cc >= r0 && cc < r1) dst[cc] = 0.0;
        }
        __syncthreads();
        if (tid == 0 && x >= r0 && x < r1)
          dst[x] = first_round ? (double)fmaxf(0.f, __fsub_rn((float)s_mass, qrow[x]))
                               : fmax(0.0, __dsub_rn(s_mass, (double)qrow[x]));
        __syncthreads();
        local = 0.0;
        for (int v = r0 + tid; v < r1; v += kTreeThreads) local += dst[v];
      }
      double z_new = tw_block_sum(local, s_warp);
      if (CLUSTER) z_new = tw_exchange(z_new, &s_slot[turn], S);
      turn ^= 1;
      if (z_new > 0.0) {                          // else p_res == q numerically: keep p_res
        src = src < 0 ? 0 : (src ^ 1);
        z = z_new;
        first_round = false;
      }
    }
    if (accepted < 0) break;
    if (rank == 0 && tid == 0) {
      p.accept_path[(size_t)b * K + n_acc] = accepted;
      if (p.accept_mask) p.accept_mask[(size_t)b * K + (accepted - F)] = 1;
    }
    ++n_acc;
    cur = accepted;
  }
  __syncthreads();

  // ---- inverse-CDF draw from the un-normalised source, ascending index ----
  const int seg = (part + kTreeThreads - 1) / kTreeThreads;
  const int v0 = min(r1, r0 + tid * seg), v1 = min(r1, v0 + seg);
  const double* dsrc = src < 0 ? nullptr : buf[src];
  if (tid == 0) {
    s_first = 0x7fffffff;
    s_last = -1;
  }
  double local = 0.0;
  int nz = -1;                                    // last code of this thread that carries mass
  for (int v = v0; v < v1; ++v) {
    const double r = dsrc ? dsrc[v] : (double)prow[v];
    local += r;
    if (r > 0.0) nz = v;
  }
  double incl = tw_warp_scan(local, lane);
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (nz >= 0) atomicMax(&s_last, nz);
  double before = 0.0, total = 0.0;               // mass ahead of this warp, in front of the CTA's part at first
  for (int w = 0; w < kTreeThreads / 32; ++w) {
    const double t = s_warp[w];
    if (w < warp) before += t;
    total += t;
  }
  // the part that holds the sample point, by the parts' sums in rank order: the first whose end lies beyond it
  const double u = (double)p.uniforms[(size_t)b * (K + 1) + K];
  double target = u * total;
  int last, owner = 0;
  if (CLUSTER) {
    if (tid == 0) s_slot[turn] = total;
    tc::cluster_sync();                            // s_last is complete too
    double sum = 0.0, part_sum[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) part_sum[r] = r < S ? tc::ld_cluster_f64(&s_slot[turn], (uint32_t)r) : 0.0;
#pragma unroll
    for (int r = 0; r < 8; ++r) sum += part_sum[r];
    target = u * sum;
    total = sum;
    owner = -1;
    last = -1;
    double ahead = 0.0;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      if (r == rank) before += ahead;
      ahead += part_sum[r];
      if (owner < 0 && ahead > target) owner = r;
    }
    if (owner < 0)                                // the point rounds to the end: the last code with mass, wherever it is
      for (int r = 0; r < S; ++r) last = max(last, tc::ld_cluster_s32(&s_last, (uint32_t)r));
    else
      last = s_last;
    tc::cluster_arrive();     // (waited for at the end)
  }
  const double excl = before + incl - local;
  if (owner == rank) {
    double c = excl;
    for (int v = v0; v < v1; ++v) {
      c += dsrc ? dsrc[v] : (double)prow[v];
      if (c > target) {
        atomicMin(&s_first, v);
        break;
      }
    }
  }
  __syncthreads();                                // s_first; s_last too where there is one CTA
  if (!CLUSTER) last = s_last;
  // (in the part that holds the point its own last code with mass, should the sums of its threads round to less)
  const int pick = owner == rank && s_first != 0x7fffffff ? s_first : last;
  if ((owner == rank || owner < 0) && pick >= v0 && pick < v1) {
    double c = excl;
    for (int v = v0; v < pick; ++v) c += dsrc ? dsrc[v] : (double)prow[v];
    const double hi = c + (dsrc ? dsrc[pick] : (double)prow[pick]);
    p.next_token[b] = p.vocab_offset + pick;
    if (p.margins) p.margins[(size_t)b * (K + 1) + K] = (float)(fmin(fabs(target - c), fabs(hi - target)) / total);
  }
  if (rank == 0 && tid == 0) {
    if (owner == rank ? pick < 0 : owner < 0 && last < 0) {     // an all-zero source: no token can be drawn
      p.next_token[b] = -1;
      atomicOr(p.status, VVS_DEV_BAD_ARG);
    }
    p.accept_len[b] = n_acc;
    for (int c = 0; c < p.n_cfg; ++c) {
      const int r = c * p.n_images + b;
      if (p.new_len && p.cache_len) p.new_len[r] = p.cache_len[r] + F + n_acc;
      if (p.n_commit) p.n_commit[r] = F + n_acc;
    }
  }
  if (CLUSTER) tc::cluster_wait();   // nobody leaves while it may be read
}

// K/V of the accepted nodes move from their block slots fill + node to fill + F + i (i-th
// accepted node): the cache is contiguous again and the rejected branches fall behind new_len.
// node_i >= F + i and the nodes ascend, so moving in path order never overwrites a later source.
template <typename T>
__global__ void tree_commit_kernel(T* __restrict__ kv_k, T* __restrict__ kv_v, const int32_t* __restrict__ cache_len,
                                   const int32_t* __restrict__ accept_len, const int32_t* __restrict__ accept_path,
                                   int n_heads, int hd, int s_max, int kv_rows, int n_images, int n_forced,
                                   int n_draft_max) {
  const int h = blockIdx.x, r = blockIdx.y, layer = blockIdx.z;
  const int b = r % n_images;
  const int fill = cache_len[r];
  if (fill < 0 || fill + n_forced + n_draft_max > s_max) return;
  const int n = accept_len[b];
  const int vecs = hd * (int)sizeof(T) / 16;          // 16-byte vectors per row
  T* base = (threadIdx.x < (unsigned)vecs ? kv_k : kv_v) + (((size_t)layer * kv_rows + r) * n_heads + h) * s_max * hd;
  const int vec = threadIdx.x < (unsigned)vecs ? threadIdx.x : threadIdx.x - vecs;
  if (vec >= vecs) return;
  for (int i = 0; i < n; ++i) {
    const int node = accept_path[(size_t)b * n_draft_max + i];
    if (node < n_forced + i || node >= n_forced + n_draft_max || node == n_forced + i) continue;
    const uint4 val = reinterpret_cast<const uint4*>(base + (size_t)(fill + node) * hd)[vec];
    reinterpret_cast<uint4*>(base + (size_t)(fill + n_forced + i) * hd)[vec] = val;
  }
}

}  // namespace

void launch_tree_walk(const TreeParams& p, int n_sms, cudaStream_t s) {
  const int S = tree_walk_parts(p.vocab, p.n_images, n_sms);
  if (S == 1) {
    tree_walk_kernel<false><<<dim3(1, p.n_images), kTreeThreads, 0, s>>>(p);
    return;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(S, p.n_images, 1);
  cfg.blockDim = dim3(kTreeThreads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, tree_walk_kernel<true>, p);   // (the caller reads cudaGetLastError)
}

void launch_tree_commit(void* kv_k, void* kv_v, const int32_t* cache_len, const int32_t* accept_len,
                        const int32_t* accept_path, const vvs_model_desc& md, int kv_rows, int n_images, int n_cfg,
                        int n_forced, int n_draft_max, cudaStream_t s) {
  if (md.n_layers < 1) return;
  using T = __nv_bfloat16;
  const int vecs = md.head_dim * (int)sizeof(T) / 16;
  dim3 grid(md.n_heads, n_images * n_cfg, md.n_layers);
  tree_commit_kernel<T><<<grid, 2 * vecs, 0, s>>>(static_cast<T*>(kv_k), static_cast<T*>(kv_v), cache_len, accept_len,
                                                  accept_path, md.n_heads, md.head_dim, md.s_max, kv_rows, n_images,
                                                  n_forced, n_draft_max);
}

}  // namespace vvs
