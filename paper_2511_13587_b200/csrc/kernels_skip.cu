// Dynamic verification-skipping decision (paper Sec. 4.4, Eq. 2, Alg. 1): for each image, the
// cosine similarity of the latent codebook embeddings of its down-sampled candidate token paths,
// weighted over depth by alpha^l, against a threshold; never two skipped steps in a row.
// One CTA per image.  The work is tiny (tens of paths, a few levels, an 8..256-dim codebook): the
// kernel is latency-bound, its cost is one dependent chain of L2 loads.
#include "vvs_internal.cuh"

namespace vvs {

namespace {

constexpr int kSkipThreads = 256;
constexpr int kSkipMaxKept = 64;    // paths kept after down-sampling
constexpr int kSkipMaxDepth = 16;

// S^(l), the mean cosine over all unordered pairs of kept paths, from unit vectors u_i = E[c_i] / |E[c_i]|:
// sum over pairs of u_i . u_j = (|sum_i u_i|^2 - n) / 2 with n the number of paths that have one -- linear in the
// number of paths.  Two rounds of loads (all norms at once, then a warp per level for the sums, from L1); sums in
// float64 in a fixed order.  16 images of 24 paths of depth 5: 8.7 us under ncu with the pairs written out, one level
// after the other.
__global__ void __launch_bounds__(kSkipThreads)
skip_decide_kernel(const int32_t* __restrict__ paths, const int32_t* __restrict__ path_len,
                   const float* __restrict__ codebook, const uint8_t* __restrict__ last_verified,
                   int n_paths, int max_len, int vocab, int dim, int lanes, int stride, float alpha, float threshold,
                   uint8_t* __restrict__ decision, float* __restrict__ sim, int32_t* status) {
  __shared__ double s_inv[kSkipMaxKept * kSkipMaxDepth];   // 1 / |E[c_i[l]]|, 0 where the cosine counts 0
  __shared__ int s_tok[kSkipMaxKept * kSkipMaxDepth];      // -1 for a token outside the codebook
  __shared__ double s_level[kSkipMaxDepth];
  __shared__ int s_depth;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int32_t* pb = paths + (size_t)b * n_paths * max_len;
  const int n_keep = (n_paths + stride - 1) / stride;
  grid_dep_launch();
  grid_dep_wait();
  if (warp == 0) {
    int depth = max_len;
    if (path_len)
      for (int i = lane; i < n_keep; i += 32) depth = min(depth, path_len[(size_t)b * n_paths + i * stride]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) depth = min(depth, __shfl_xor_sync(0xffffffffu, depth, o));
    if (lane == 0) s_depth = depth < 0 ? 0 : depth;
  }
  const bool verified = last_verified ? last_verified[b] != 0 : true;
  // norms of every (path, level): `lanes` lanes each (a power of two), levels beyond the depth are computed in vain
  // rather than waited for
  const int n_items = n_keep * max_len, per = kSkipThreads / lanes, sub = tid & (lanes - 1);
  for (int base = 0; base < n_items; base += per) {
    const int t = base + tid / lanes;
    const int i = t / max_len, l = t - i * max_len;
    int tok = -1;
    if (t < n_items) tok = pb[(size_t)(i * stride) * max_len + l];
    const bool ok = tok >= 0 && tok < vocab;
    double nn = 0.0;
    if (ok) {
      const float* e = codebook + (size_t)tok * dim;
      for (int d = sub; d < dim; d += lanes) nn += (double)e[d] * (double)e[d];
    }
    for (int o = lanes >> 1; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
    if (t < n_items && sub == 0) {
      s_tok[i * kSkipMaxDepth + l] = ok ? tok : -1;
      s_inv[i * kSkipMaxDepth + l] = nn > 0.0 ? 1.0 / sqrt(nn) : 0.0;
    }
  }
  __syncthreads();
  const int depth = s_depth;
  if (!verified || depth == 0 || n_keep < 2) {              // Alg. 1 guard and the degenerate cases
    if (tid == 0) {
      const float s = (!verified || depth == 0) ? 0.f : 1.f;
      sim[b] = s;
      decision[b] = (verified && s >= threshold) ? 1 : 0;
    }
    return;
  }
  const double n_pairs = 0.5 * n_keep * (n_keep - 1);
  for (int l = warp; l < depth; l += kSkipThreads / 32) {
    // lane = (path phase, dimension): the phases are added by shuffles, then squared
    const int phases = 32 / lanes, ph = lane / lanes, ds = lane & (lanes - 1);
    double sq = 0.0;
    for (int d0 = 0; d0 < dim; d0 += lanes) {
      const int d = d0 + ds;
      double u = 0.0;
      if (d < dim)
        for (int i = ph; i < n_keep; i += phases) {
          const double inv = s_inv[i * kSkipMaxDepth + l];
          if (inv > 0.0) u += inv * (double)codebook[(size_t)s_tok[i * kSkipMaxDepth + l] * dim + d];
        }
      for (int o = lanes; o < 32; o <<= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
      sq += u * u;
    }
    for (int o = lanes >> 1; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    int n = 0;
    bool bad = false;
    for (int i = lane; i < n_keep; i += 32) {
      n += s_inv[i * kSkipMaxDepth + l] > 0.0 ? 1 : 0;
      bad |= s_tok[i * kSkipMaxDepth + l] < 0;
    }
    n = __reduce_add_sync(0xffffffffu, n);
    if (bad) atomicOr(status, VVS_DEV_BAD_TOKEN);
    if (lane == 0) s_level[l] = n < 2 ? 0.0 : 0.5 * (sq - (double)n) / n_pairs;
  }
  __syncthreads();
  if (tid == 0) {
    double wsum = 0.0, w = 1.0, s = 0.0;
    for (int l = 0; l < depth; ++l) {
      s += w * s_level[l];
      wsum += w;
      w *= (double)alpha;
    }
    s /= wsum;
    sim[b] = (float)s;
    decision[b] = s >= (double)threshold ? 1 : 0;
  }
}

// Unverified token selection with truncation (Sec. 4.2, Eq. 3): one warp per image.
__global__ void select_unverified_kernel(const int32_t* __restrict__ paths, const int32_t* __restrict__ path_len,
                                         const float* __restrict__ uniforms, int n_paths, int max_len,
                                         int32_t* __restrict__ out_path, int32_t* __restrict__ out_gamma,
                                         int32_t* __restrict__ out_tokens, int32_t* status) {
  const int b = blockIdx.x, lane = threadIdx.x;
  grid_dep_launch();
  grid_dep_wait();
  long long total = 0;
  bool bad = false;
  for (int i = lane; i < n_paths; i += 32) {
    const int len = path_len ? path_len[(size_t)b * n_paths + i] : max_len;
    bad |= len < 0 || len > max_len;
    total += len < 0 ? 0 : (len > max_len ? max_len : len);
  }
  for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, VVS_DEV_BAD_ARG);
  int idx = (int)floorf(uniforms[b] * (float)n_paths);
  idx = idx < 0 ? 0 : (idx > n_paths - 1 ? n_paths - 1 : idx);
  int len_s = path_len ? path_len[(size_t)b * n_paths + idx] : max_len;
  len_s = len_s < 0 ? 0 : (len_s > max_len ? max_len : len_s);
  const int mean_floor = (int)(total / n_paths);
  const int gamma = len_s < mean_floor ? len_s : mean_floor;
  if (lane == 0) {
    out_path[b] = idx;
    out_gamma[b] = gamma;
  }
  for (int t = lane; t < max_len; t += 32)
    out_tokens[(size_t)b * max_len + t] = t < gamma ? paths[((size_t)b * n_paths + idx) * max_len + t] : -1;
}

}  // namespace

int launch_select_unverified(const int32_t* paths, const int32_t* path_len, const float* uniforms, int n_images,
                             int n_paths, int max_len, int32_t* out_path, int32_t* out_gamma, int32_t* out_tokens,
                             int32_t* status, cudaStream_t s) {
  return launch_kernel(select_unverified_kernel, dim3(n_images), dim3(32), 0, true, s, paths, path_len, uniforms, n_paths, max_len,
                       out_path, out_gamma, out_tokens, status) == cudaSuccess ? VVS_OK : VVS_ERR_CUDA;
}

int launch_skip_decide(const int32_t* paths, const int32_t* path_len, const float* codebook,
                       const uint8_t* last_verified, int n_images, int n_paths, int max_len, int vocab, int dim,
                       int stride, float alpha, float threshold, uint8_t* decision, float* sim, int32_t* status,
                       cudaStream_t s) {
  if ((n_paths + stride - 1) / stride > kSkipMaxKept || max_len > kSkipMaxDepth) return VVS_ERR_SHAPE;
  int lanes = 1;                                            // per embedding: the largest power of two within a row and a warp
  while (lanes < 32 && lanes * 2 <= dim) lanes *= 2;
  return launch_kernel(skip_decide_kernel, dim3(n_images), dim3(kSkipThreads), 0, true, s, paths, path_len, codebook, last_verified,
                       n_paths, max_len, vocab, dim, lanes, stride, alpha, threshold, decision, sim, status) == cudaSuccess
             ? VVS_OK : VVS_ERR_CUDA;
}

}  // namespace vvs
