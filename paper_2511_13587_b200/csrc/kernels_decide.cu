// Decision stage of the verify step (paper Sec. 2): acceptance test per drafted token, accepted
// prefix, residual / bonus sample.  Works on softmax statistics plus gathered logits, so the
// same kernels serve the generic path (full logits in scratch) and the fused LM-head path
// (logits never written out).
#include <math_constants.h>

#include "tc_common.cuh"
#include "vvs_internal.cuh"

namespace vvs {

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_incl_scan_d(double v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    double t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Relaxed numerator (Sec. 2): the longest distance-ordered prefix of neighbour entries 1 .. kk-1
// whose cumulative mass stays <= delta.  One warp; pn(j) gives the mass of entry j.  Returns the
// pooled mass (the same value in every lane) and the first entry NOT pooled in *j_end.
template <typename F>
__device__ __forceinline__ double pooled_prefix(int kk, double delta, int lane, F pn_of, int* j_end) {
  double cum = 0.0;
  int end = kk;
  for (int j0 = 1; j0 < kk; j0 += 32) {
    const int j = j0 + lane;
    const double pn = (j < kk) ? pn_of(j) : 0.0;
    const double tot = cum + warp_incl_scan_d(pn, lane);
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

// ---------------------------------------------------------------------------------------------
// Combine per-tile softmax partials: M = max_t m_t, S = sum_t s_t exp(m_t - M), fixed order.
__global__ void finalize_stats_kernel(const float* __restrict__ part_m, const float* __restrict__ part_s,
                                      float* __restrict__ stat_m, float* __restrict__ stat_inv,
                                      int n_tiles, int n_rows) {
  int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  int lane = threadIdx.x & 31;
  if (row >= n_rows) return;
  float mx = -CUDART_INF_F;
  for (int t = lane; t < n_tiles; t += 32) mx = fmaxf(mx, part_m[(size_t)row * n_tiles + t]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  float sum = 0.f;
  for (int t = lane; t < n_tiles; t += 32)
    sum += part_s[(size_t)row * n_tiles + t] * expf(part_m[(size_t)row * n_tiles + t] - mx);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) {
    stat_m[row] = mx;
    stat_inv[row] = 1.f / sum;
  }
}

void launch_finalize_stats(const Workspace& ws, int n_tiles, int n_rows, cudaStream_t s) {
  finalize_stats_kernel<<<(n_rows + 3) / 4, 128, 0, s>>>(ws.part_m, ws.part_s, ws.stat_m, ws.stat_inv,
                                                         n_tiles, n_rows);
}

// ---------------------------------------------------------------------------------------------
// Generic path: pull the logits of each drafted token and of its neighbours out of the
// materialised logits.  grid (K, B).
__global__ void gather_logits_kernel(const float* __restrict__ logits, float* __restrict__ l_tok,
                                     float* __restrict__ l_nbr, DecideParams p, int32_t* status) {
  int i = blockIdx.x, b = blockIdx.y;
  int K = p.n_draft_max, V = p.vocab;
  int x = p.drafts[(size_t)b * p.drafts_ld + i] - p.vocab_offset;
  if (x < 0 || x >= V) return;  // reported by the acceptance kernel
  const float* row = logits + ((size_t)b * p.rows_per_seq + p.first_row + i) * V;
  if (threadIdx.x == 0) l_tok[b * K + i] = row[x];
  if (p.mode != VVS_MODE_RELAXED || p.nbr_k <= 1) return;
  int beg = p.row_ptr[x], len = p.row_ptr[x + 1] - beg;
  int kk = min(p.nbr_k, len);
  float* dst = l_nbr + ((size_t)b * K + i) * p.kmax;
  for (int j = 1 + threadIdx.x; j < kk; j += blockDim.x) {
    int c = p.col[beg + j];
    bool ok = c >= 0 && c < V;
    if (!ok) atomicOr(status, VVS_DEV_BAD_NEIGHBOUR);
    dst[j] = ok ? row[c] : -CUDART_INF_F;
  }
}

void launch_gather_logits(const float* logits, const Workspace& ws, const DecideParams& p, cudaStream_t s) {
  if (p.n_draft_max == 0) return;
  dim3 grid(p.n_draft_max, p.n_images);
  gather_logits_kernel<<<grid, 128, 0, s>>>(logits, ws.l_tok, ws.l_nbr, p, ws.status);
}

// ---------------------------------------------------------------------------------------------
// Acceptance (Sec. 2): draft i passes iff u_i < min(1, P_i / q_i(x_i)) with P_i = p(x_i) (strict)
// or the pooled mass of x_i and the longest distance-ordered neighbour prefix whose own mass
// stays <= delta (relaxed).  Verification stops at the first rejection.  One CTA per image.
__global__ void accept_kernel(Workspace ws, DecideParams p) {
  __shared__ double ratio_s[32];
  int b = blockIdx.x;
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  int K = p.n_draft_max, V = p.vocab;
  int nd = p.n_draft ? p.n_draft[b] : K;
  if (nd < 0 || nd > K) {
    if (threadIdx.x == 0) atomicOr(ws.status, VVS_DEV_BAD_ARG);
    nd = nd < 0 ? 0 : K;
  }
  for (int i = warp; i < K; i += nw) {
    double ratio = 0.0;
    if (i < nd) {
      int x = p.drafts[(size_t)b * p.drafts_ld + i] - p.vocab_offset;
      if (x < 0 || x >= V) {
        if (lane == 0) atomicOr(ws.status, VVS_DEV_BAD_TOKEN);
      } else {
        int drow = b * p.rows_per_seq + p.first_row + i;
        const bool direct = p.direct_probs != nullptr;
        float m = direct ? 0.f : ws.stat_m[drow], inv = direct ? 1.f : ws.stat_inv[drow];
        double mass = (double)(direct ? ws.l_tok[b * K + i] : prob_of(ws.l_tok[b * K + i], m, inv));
        if (p.mode == VVS_MODE_RELAXED && p.nbr_k > 1) {
          int beg = p.row_ptr[x], len = p.row_ptr[x + 1] - beg;
          if (len < 1 && lane == 0) atomicOr(ws.status, VVS_DEV_BAD_NEIGHBOUR);
          int kk = min(p.nbr_k, len);
          const float* ln = ws.l_nbr + ((size_t)b * K + i) * p.kmax;
          int j_end;
          const double cum = pooled_prefix(kk, (double)p.delta, lane, [&](int j) {
            return (double)(direct ? ln[j] : prob_of(ln[j], m, inv)); }, &j_end);
          mass += cum;
        }
        double qx = (double)p.draft_probs[((size_t)b * K + i) * V + x];
        ratio = qx > 0.0 ? fmin(1.0, mass / qx) : (mass > 0.0 ? 1.0 : 0.0);
      }
    }
    if (lane == 0) ratio_s[i] = ratio;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  int n = 0;
  bool open = true;
  for (int i = 0; i < K; ++i) {
    float margin = CUDART_INF_F;
    uint8_t bit = 0;
    if (open && i < nd) {
      double u = (double)p.uniforms[(size_t)b * (K + 1) + i];
      margin = (float)fabs(u - ratio_s[i]);
      if (u < ratio_s[i]) {
        bit = 1;
        ++n;
      } else {
        open = false;
      }
    }
    if (p.margins) p.margins[(size_t)b * (K + 1) + i] = margin;
    if (p.accept_mask) p.accept_mask[(size_t)b * K + i] = bit;
  }
  p.accept_len[b] = n;
  if (p.new_len && p.cache_len) {
    for (int c = 0; c < p.n_cfg; ++c) {
      int r = c * p.n_images + b;
      p.new_len[r] = p.cache_len[r] + p.n_forced + n;
    }
  }
  if (p.n_commit) {
    for (int c = 0; c < p.n_cfg; ++c) p.n_commit[c * p.n_images + b] = p.n_forced + n;
  }
  int t_sel = p.first_row + n;
  ws.sel_row[b] = (t_sel < p.rows_per_seq) ? b * p.rows_per_seq + t_sel : -1;
  ws.sel_kind[b] = (n < nd) ? 0 : 1;
}

void launch_accept(const Workspace& ws, const DecideParams& p, cudaStream_t s) {
  accept_kernel<<<p.n_images, 256, 0, s>>>(ws, p);
}

// ---------------------------------------------------------------------------------------------
__global__ void probs_kernel(const float* __restrict__ logits, const float* __restrict__ stat_m,
                             const float* __restrict__ stat_inv, float* __restrict__ probs, int v) {
  size_t row = blockIdx.y;
  grid_dep_launch();
  grid_dep_wait();
  float m = stat_m[row], inv = stat_inv[row];
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < v) probs[row * v + j] = prob_of(logits[row * v + j], m, inv);
}

// probs may alias logits (in-place normalisation)
void launch_probs_from_logits(const float* logits, const Workspace& ws, float* probs, int n_rows,
                              int v, bool pdl, cudaStream_t s) {
  launch_kernel(probs_kernel, dim3((v + 255) / 256, n_rows), dim3(256), 0, pdl, s, logits, ws.stat_m, ws.stat_inv, probs, v);
}

// target probabilities of the row each image samples from, out of stored guided logits
__global__ void select_p_row_kernel(const float* __restrict__ logits, Workspace ws, int v) {
  int b = blockIdx.y;
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= v) return;
  int row = ws.sel_row[b];
  float pr = 0.f;
  if (row >= 0) pr = prob_of(logits[(size_t)row * v + j], ws.stat_m[row], ws.stat_inv[row]);
  ws.p_row[(size_t)b * v + j] = pr;
}

void launch_select_p_row(const float* logits, const Workspace& ws, int n_images, int v, cudaStream_t s) {
  dim3 grid((v + 255) / 256, n_images);
  select_p_row_kernel<<<grid, 256, 0, s>>>(logits, ws, v);
}

// ---------------------------------------------------------------------------------------------
// Adjusted target of a relaxed rejection (flag adjusted_residual): in the row image b samples
// from, the pooled neighbours of the rejected draft x give their mass to x.  The row lives in
// ws.p_row (copied there first when the caller's probabilities are used directly); the pooled
// prefix is found again from the row's own float32 values, by the rule of accept_kernel.
// grid B, 256 threads.
__global__ void adjust_target_kernel(Workspace ws, DecideParams p) {
  const int b = blockIdx.x, V = p.vocab;
  const int sel = ws.sel_row[b];
  if (sel < 0) return;
  float* row = ws.p_row + (size_t)b * V;
  if (p.direct_probs) {
    const float* src = p.direct_probs + (size_t)sel * V;
    for (int j = threadIdx.x; j < V; j += blockDim.x) row[j] = src[j];
    __syncthreads();
  }
  if (ws.sel_kind[b] != 0 || threadIdx.x >= 32) return;    // bonus row: nothing was rejected
  const int lane = threadIdx.x;
  const int n = p.accept_len[b];
  const int x = p.drafts[(size_t)b * p.drafts_ld + n] - p.vocab_offset;
  if (x < 0 || x >= V) return;                             // reported by the acceptance kernel
  const int beg = p.row_ptr[x], len = p.row_ptr[x + 1] - beg;
  const int kk = min(p.nbr_k, len);
  auto mass_of = [&](int j) {
    const int c = p.col[beg + j];
    return (c >= 0 && c < V) ? (double)row[c] : 0.0;
  };
  int j_end;
  const double cum = pooled_prefix(kk, (double)p.delta, lane, mass_of, &j_end);
  const double mass = (double)row[x] + cum;
  __syncwarp();
  for (int j = 1 + lane; j < j_end; j += 32) {
    const int c = p.col[beg + j];
    if (c >= 0 && c < V) row[c] = 0.f;
  }
  __syncwarp();
  if (lane == 0) row[x] = (float)mass;
}

void launch_adjust_target(const Workspace& ws, const DecideParams& p, cudaStream_t s) {
  adjust_target_kernel<<<p.n_images, 256, 0, s>>>(ws, p);
}

// ---------------------------------------------------------------------------------------------
// Residual distribution (Sec. 2): r = max(0, p - q_n) at the first rejected draft n, or r = p for
// the bonus token; float32 difference, float64 accumulation.
__device__ __forceinline__ float residual_value(float pr, const float* q_row, int j, int kind) {
  if (kind != 0) return pr;
  return fmaxf(0.f, pr - q_row[j]);
}

// grid (n_chunks, B), block kSampleChunk/4 threads
__global__ void residual_mass_kernel(Workspace ws, DecideParams p, int n_chunks) {
  __shared__ double red_r[32], red_p[32];
  int c = blockIdx.x, b = blockIdx.y;
  int V = p.vocab, K = p.n_draft_max;
  int kind = ws.sel_kind[b];
  int n = p.accept_len[b];
  const float* q_row = p.draft_probs + ((size_t)b * K + (kind == 0 ? n : 0)) * V;
  const int sel = ws.sel_row[b];
  if (sel < 0) return;  // no row to sample from: sample_kernel reports -1
  const float* p_row = (p.direct_probs && !p.adjusted) ? p.direct_probs + (size_t)sel * V : ws.p_row + (size_t)b * V;
  double sr = 0.0, sp = 0.0;
  int end = min(V, (c + 1) * kSampleChunk);
  for (int j = c * kSampleChunk + threadIdx.x; j < end; j += blockDim.x) {
    float pr = p_row[j];
    sr += (double)residual_value(pr, q_row, j, kind);
    sp += (double)pr;
  }
  sr = warp_sum_d(sr);
  sp = warp_sum_d(sp);
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) {
    red_r[warp] = sr;
    red_p[warp] = sp;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double tr = 0.0, tp = 0.0;
    for (int w = 0; w < nw; ++w) {
      tr += red_r[w];
      tp += red_p[w];
    }
    ws.r_part[(size_t)b * n_chunks + c] = tr;
    ws.p_part[(size_t)b * n_chunks + c] = tp;
  }
}

// Inverse CDF in ascending token order: smallest j with cumulative mass > u * total.
// grid B, block kSampleChunk threads.
__global__ void sample_kernel(Workspace ws, DecideParams p, int n_chunks) {
  __shared__ double warp_tot[32];
  __shared__ double s_lo, s_t, s_total;
  __shared__ int s_chunk, s_use_p, s_first, s_last;
  int b = blockIdx.x;
  int V = p.vocab, K = p.n_draft_max;
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (ws.sel_row[b] < 0) {
    if (threadIdx.x == 0) {
      p.next_token[b] = -1;
      if (p.margins) p.margins[(size_t)b * (K + 1) + K] = CUDART_INF_F;
    }
    return;
  }
  int kind = ws.sel_kind[b];
  if (threadIdx.x == 0) {
    const double* rp = ws.r_part + (size_t)b * n_chunks;
    double total = 0.0;
    for (int c = 0; c < n_chunks; ++c) total += rp[c];
    int use_p = 0;
    if (!(total > 0.0)) {  // p == q numerically: fall back to the target row itself
      use_p = 1;
      rp = ws.p_part + (size_t)b * n_chunks;
      total = 0.0;
      for (int c = 0; c < n_chunks; ++c) total += rp[c];
    }
    double t = (double)p.uniforms[(size_t)b * (K + 1) + K] * total;
    double lo = 0.0;
    int chunk = -1, last_nz = 0;
    double last_lo = 0.0;
    for (int c = 0; c < n_chunks; ++c) {
      if (rp[c] > 0.0) {
        last_nz = c;
        last_lo = lo;
      }
      if (lo + rp[c] > t) {
        chunk = c;
        break;
      }
      lo += rp[c];
    }
    if (chunk < 0) {
      chunk = last_nz;
      lo = last_lo;
    }
    s_lo = lo;
    s_t = t;
    s_total = total;
    s_chunk = chunk;
    s_use_p = use_p;
    s_first = 0x7fffffff;
    s_last = -1;
  }
  __syncthreads();
  int n = p.accept_len[b];
  int eff_kind = s_use_p ? 1 : kind;
  const float* q_row = p.draft_probs + ((size_t)b * K + (eff_kind == 0 ? n : 0)) * V;
  const float* p_row = (p.direct_probs && !p.adjusted) ? p.direct_probs + (size_t)ws.sel_row[b] * V
                                                       : ws.p_row + (size_t)b * V;
  int j = s_chunk * kSampleChunk + threadIdx.x;
  double val = 0.0;
  if (j < V) val = (double)residual_value(p_row[j], q_row, j, eff_kind);
  double inc = warp_incl_scan_d(val, lane);
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    double w = warp_tot[lane];
    double ws_incl = warp_incl_scan_d(w, lane);
    warp_tot[lane] = ws_incl - w;  // exclusive prefix of each warp
  }
  __syncthreads();
  double cdf = s_lo + warp_tot[warp] + inc;
  if (j < V && cdf > s_t) atomicMin(&s_first, j);
  if (j < V && val > 0.0) atomicMax(&s_last, j);
  __syncthreads();
  int pick = (s_first != 0x7fffffff) ? s_first : s_last;
  if (j == pick) {
    p.next_token[b] = p.vocab_offset + j;
    if (p.margins) {
      double a = fabs(s_t - (cdf - val)), c2 = fabs(cdf - s_t);
      p.margins[(size_t)b * (K + 1) + K] = (float)(fmin(a, c2) / s_total);
    }
  }
  if (pick < 0 && threadIdx.x == 0) p.next_token[b] = -1;
}

void launch_residual_mass(const Workspace& ws, const DecideParams& p, cudaStream_t s) {
  int n_chunks = (p.vocab + kSampleChunk - 1) / kSampleChunk;
  dim3 grid(n_chunks, p.n_images);
  residual_mass_kernel<<<grid, kSampleChunk / 4, 0, s>>>(ws, p, n_chunks);
}

void launch_sample(const Workspace& ws, const DecideParams& p, cudaStream_t s) {
  int n_chunks = (p.vocab + kSampleChunk - 1) / kSampleChunk;
  sample_kernel<<<p.n_images, kSampleChunk, 0, s>>>(ws, p, n_chunks);
}

// ---------------------------------------------------------------------------------------------
// The whole decision of an image in one kernel: softmax statistics (when the rows are logits), acceptance,
// residual masses, inverse CDF.  A cluster of S CTAs per image: every CTA takes the acceptance decision for
// itself (a few dozen gathered values: cheaper than an exchange), then sums its contiguous part of the codebook, warp
// by warp in index order; the part sums are read through distributed shared memory and the one warp whose part
// holds the sample point walks it.  Replaces finalize / gather / accept / select / residual / sample, six launches
// of 3-7 us each on a few hundred kilobytes: the work is a chain of four dependent round trips to L2 (drafts; their values;
// the masses of a row; the range of the sample point), of six with neighbour lists (their places; their columns).  What does not depend
// on the statistics is requested before them, and the partials of a row come in one trip; sixteen warps take the rows
// and drafts of a usual block in one turn (16 images 8.4 -> 7.6 us, behind the LM head of one image 15.3 -> 14.1 us).
namespace {

constexpr int kDecideThreads = 512, kDecideWarps = kDecideThreads / 32;


// LOGITS: rows hold guided logits, statistics come from the [rows, n_tiles] softmax partials; else probabilities.
template <bool LOGITS>
__global__ void __launch_bounds__(kDecideThreads) decide_kernel(Workspace ws, DecideParams p, const float* __restrict__ rows,
                                                                int n_tiles) {
  __shared__ float s_m[32], s_inv[32];
  __shared__ double s_ratio[32];
  __shared__ double s_w[2][kDecideWarps];            // masses of this CTA's warps: residual, target
  __shared__ double s_seg[2];
  __shared__ double s_lo, s_t, s_total;
  __shared__ int s_n, s_kind, s_part, s_use_p;
  const int b = blockIdx.y, S = (int)gridDim.x, rank = (int)blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int K = p.n_draft_max, V = p.vocab;
  grid_dep_launch();
  grid_dep_wait();

  // ---- what the decision needs besides the statistics: requested first, so that it travels with them -----------------
  int nd = p.n_draft ? p.n_draft[b] : K;
  const float u_pick = p.uniforms[(size_t)b * (K + 1) + K], u_test = lane < K ? p.uniforms[(size_t)b * (K + 1) + lane] : 0.f;
  struct Draft {                                     // a drafted token: its draft probability, its value, its neighbour list
    float q, raw;
    int x, beg, len;
  };
  auto load_draft = [&](int i) {
    Draft d{0.f, 0.f, p.drafts[(size_t)b * p.drafts_ld + i] - p.vocab_offset, 0, 0};
    if (d.x >= 0 && d.x < V) {
      d.q = p.draft_probs[((size_t)b * K + i) * V + d.x];
      d.raw = rows[((size_t)b * p.rows_per_seq + p.first_row + i) * V + d.x];
      if (p.mode == VVS_MODE_RELAXED && p.nbr_k > 1) {
        d.beg = p.row_ptr[d.x];
        d.len = p.row_ptr[d.x + 1] - d.beg;
      }
    }
    return d;
  };
  Draft mine{};
  if (warp < K) mine = load_draft(warp);

  // ---- statistics of the image's rows: M = max_t m_t, S = sum_t s_t exp(m_t - M) ------------------------------------
  if (LOGITS) {
    for (int r = warp; r < p.rows_per_seq; r += kDecideWarps) {
      const int row = b * p.rows_per_seq + r;
      float mx = -CUDART_INF_F, sum = 0.f;
      const float* pm = ws.part_m + (size_t)row * n_tiles;
      const float* ps = ws.part_s + (size_t)row * n_tiles;
      for (int t0 = lane; t0 < n_tiles; t0 += 128) {
        float tm[4], ts[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const bool in = t0 + 32 * e < n_tiles;
          tm[e] = in ? pm[t0 + 32 * e] : -CUDART_INF_F;
          ts[e] = in ? ps[t0 + 32 * e] : 0.f;
        }
        const float top = fmaxf(mx, fmaxf(fmaxf(tm[0], tm[1]), fmaxf(tm[2], tm[3])));
        if (top > -CUDART_INF_F) {
          sum *= expf(mx - top);
#pragma unroll
          for (int e = 0; e < 4; ++e) sum += ts[e] * expf(tm[e] - top);
          mx = top;
        }
      }
      float all = mx;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) all = fmaxf(all, __shfl_xor_sync(0xffffffffu, all, o));
      sum = mx > -CUDART_INF_F ? sum * expf(mx - all) : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (lane == 0) {
        s_m[r] = all;
        s_inv[r] = 1.f / sum;
        if (rank == 0) {
          ws.stat_m[row] = all;
          ws.stat_inv[row] = 1.f / sum;
        }
      }
    }
    __syncthreads();
  }

  // ---- acceptance ratios, a warp per draft ---------------------------------------------------------------------------
  if (nd < 0 || nd > K) {
    if (tid == 0) atomicOr(ws.status, VVS_DEV_BAD_ARG);
    nd = nd < 0 ? 0 : K;
  }
  for (int i = warp; i < nd; i += kDecideWarps) {
    double ratio = 0.0;
    if (i != warp) mine = load_draft(i);
    const int x = mine.x;
    if (x < 0 || x >= V) {
      if (lane == 0) atomicOr(ws.status, VVS_DEV_BAD_TOKEN);
    } else {
      const int r = p.first_row + i;
      const float* row = rows + ((size_t)b * p.rows_per_seq + r) * V;
      const float m = LOGITS ? s_m[r] : 0.f, inv = LOGITS ? s_inv[r] : 1.f;
      const double qx = (double)mine.q;
      double mass = (double)(LOGITS ? prob_of(mine.raw, m, inv) : mine.raw);
      if (p.mode == VVS_MODE_RELAXED && p.nbr_k > 1) {
        const int beg = mine.beg, len = mine.len;
        if (len < 1 && lane == 0) atomicOr(ws.status, VVS_DEV_BAD_NEIGHBOUR);
        const int kk = min(p.nbr_k, len);
        // entries 1 .. kk-1, 128 at a time: their columns, then their values in flight together; with an unlimited
        // delta only the sum is wanted, else the longest prefix whose mass stays <= delta
        constexpr int kBatch = 4;
        const bool all = isinf(p.delta);
        double cum = 0.0;
        bool over = false;
        for (int j0 = 1; j0 < kk && !over; j0 += 32 * kBatch) {
          int c[kBatch];
          float pn[kBatch];
#pragma unroll
          for (int e = 0; e < kBatch; ++e) c[e] = j0 + e * 32 + lane < kk ? p.col[beg + j0 + e * 32 + lane] : -2;
#pragma unroll
          for (int e = 0; e < kBatch; ++e) {
            if (c[e] != -2 && (c[e] < 0 || c[e] >= V)) {
              atomicOr(ws.status, VVS_DEV_BAD_NEIGHBOUR);
              c[e] = -2;
            }
            pn[e] = c[e] >= 0 ? row[c[e]] : 0.f;
          }
#pragma unroll
          for (int e = 0; e < kBatch; ++e) {
            const double v = c[e] >= 0 ? (double)(LOGITS ? prob_of(pn[e], m, inv) : pn[e]) : 0.0;
            if (all) {
              cum += v;                               // this lane's share
            } else if (!over) {
              const double tot = cum + warp_incl_scan_d(v, lane);
              const unsigned stop = __ballot_sync(0xffffffffu, j0 + e * 32 + lane < kk && tot > (double)p.delta);
              const int last = stop ? __ffs(stop) - 2 : 31;        // last lane pooled
              const double upto = __shfl_sync(0xffffffffu, tot, last < 0 ? 0 : last);
              if (last >= 0) cum = upto;
              over = stop != 0;
            }
          }
        }
        mass += all ? warp_sum_d(cum) : cum;
      }
      ratio = qx > 0.0 ? fmin(1.0, mass / qx) : (mass > 0.0 ? 1.0 : 0.0);
    }
    if (lane == 0) s_ratio[i] = ratio;
  }
  __syncthreads();
  if (warp == 0) {                                    // accepted prefix: the first lane whose test fails
    const double u = lane < nd ? (double)u_test : 0.0;
    const bool pass = lane < nd && u < s_ratio[lane];
    const unsigned fails = ~__ballot_sync(0xffffffffu, pass);
    const int n = fails ? min(__ffs(fails) - 1, nd) : nd;
    if (lane == 0) {
      s_n = n;
      s_kind = n < nd ? 0 : 1;
    }
    if (rank == 0) {
      if (lane < K) {
        const bool judged = lane < nd && lane <= n;
        if (p.margins) p.margins[(size_t)b * (K + 1) + lane] = judged ? (float)fabs(u - s_ratio[lane]) : CUDART_INF_F;
        if (p.accept_mask) p.accept_mask[(size_t)b * K + lane] = lane < n ? 1 : 0;
      }
      if (lane == 0) p.accept_len[b] = n;
      if (lane < p.n_cfg) {
        const int r = lane * p.n_images + b;
        if (p.new_len && p.cache_len) p.new_len[r] = p.cache_len[r] + p.n_forced + n;
        if (p.n_commit) p.n_commit[r] = p.n_forced + n;
      }
    }
  }
  __syncthreads();

  // ---- masses of this CTA's part, a contiguous range per warp ------------------------------------------------------
  const int n = s_n, r_sel = p.first_row + n;
  const bool has_row = r_sel < p.rows_per_seq;
  const float* p_row = rows + ((size_t)b * p.rows_per_seq + (has_row ? r_sel : 0)) * V;
  const float* q_row = p.draft_probs + ((size_t)b * K + (s_kind == 0 ? n : 0)) * V;
  const float m = LOGITS ? s_m[has_row ? r_sel : 0] : 0.f, inv = LOGITS ? s_inv[has_row ? r_sel : 0] : 1.f;
  // a contiguous range per warp and, inside it, per lane (whole 16-byte pieces), so that the sample is found by one
  // scan of the lanes' sums and a walk of one lane's few codes
  const int per_lane = ((V + S * kDecideThreads - 1) / (S * kDecideThreads) + 3) & ~3;
  const int at = (rank * kDecideThreads + tid) * per_lane;
  const int v0 = min(V, at), v1 = min(V, at + per_lane), kind = s_kind;
  auto target = [&](float x) { return LOGITS ? prob_of(x, m, inv) : x; };
  auto value = [&](float pr, float q, int how) { return (double)(how != 0 ? pr : fmaxf(0.f, pr - q)); };
  const bool vec = (V & 3) == 0;                      // rows start on 16-byte boundaries
  double sr = 0.0, sp = 0.0;
  if (has_row) {
    if (vec) {
#pragma unroll 4
      for (int j = v0; j < v1; j += 4) {
        const float4 x = *reinterpret_cast<const float4*>(p_row + j);
        const float4 q = kind == 0 ? *reinterpret_cast<const float4*>(q_row + j) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float pr[4] = {target(x.x), target(x.y), target(x.z), target(x.w)}, qv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          sr += value(pr[e], qv[e], kind);
          sp += (double)pr[e];
        }
      }
    } else {
#pragma unroll 4
      for (int j = v0; j < v1; ++j) {
        const float pr = target(p_row[j]);
        sr += value(pr, kind == 0 ? q_row[j] : 0.f, kind);
        sp += (double)pr;
      }
    }
  }
  const double lane_mass[2] = {sr, sp};
  sr = warp_sum_d(sr);
  sp = warp_sum_d(sp);
  if (lane == 0) {
    s_w[0][warp] = sr;
    s_w[1][warp] = sp;
  }
  __syncthreads();
  if (tid < 2) {
    double s = 0.0;
    for (int w = 0; w < kDecideWarps; ++w) s += s_w[tid][w];
    s_seg[tid] = s;
  }
  if (S > 1) tc::cluster_sync();
  else __syncthreads();
  if (warp == 0) {
    double seg[2] = {0.0, 0.0};
    if (lane < S) {
      seg[0] = S > 1 ? tc::ld_cluster_f64(&s_seg[0], lane) : s_seg[0];
      seg[1] = S > 1 ? tc::ld_cluster_f64(&s_seg[1], lane) : s_seg[1];
    }
    const double total_r = warp_sum_d(seg[0]), total_p = warp_sum_d(seg[1]);
    const int use_p = total_r > 0.0 ? 0 : 1;          // p == q numerically: fall back to the target row itself
    const double val = seg[use_p], total = use_p ? total_p : total_r;
    const double t = (double)u_pick * total;
    const double incl = warp_incl_scan_d(val, lane);
    const unsigned hit = __ballot_sync(0xffffffffu, lane < S && incl > t), nz = __ballot_sync(0xffffffffu, val > 0.0);
    const int part = hit ? __ffs(hit) - 1 : nz ? 31 - __clz(nz) : 0;
    const double lo = __shfl_sync(0xffffffffu, incl - val, part);
    if (lane == 0) {
      s_lo = lo; s_t = t; s_total = total; s_use_p = use_p;
      s_part = has_row && total > 0.0 ? part : -1;
    }
  }
  if (S > 1) tc::cluster_arrive();   // (waited for at the end)
  __syncthreads();
  // ---- the sample point: smallest index whose cumulative mass exceeds t, in the part that holds it -----------------
  if (s_part < 0) {
    if (rank == 0 && tid == 0) {
      p.next_token[b] = -1;
      if (p.margins) p.margins[(size_t)b * (K + 1) + K] = CUDART_INF_F;
    }
  } else if (s_part == rank) {
    const int eff = s_use_p ? 1 : kind;
    const double* w_mass = s_w[s_use_p];
    int sel = -1, last_nz = 0;
    double lo = s_lo, sel_lo = lo, nz_lo = lo;
    for (int w = 0; w < kDecideWarps; ++w) {
      if (w_mass[w] > 0.0) { last_nz = w; nz_lo = lo; }
      if (lo + w_mass[w] > s_t) { sel = w; sel_lo = lo; break; }
      lo += w_mass[w];
    }
    if (sel < 0) { sel = last_nz; sel_lo = nz_lo; }
    if (warp == sel) {
      const double mine = lane_mass[s_use_p], incl = warp_incl_scan_d(mine, lane);
      const unsigned hit = __ballot_sync(0xffffffffu, sel_lo + incl > s_t), nz = __ballot_sync(0xffffffffu, mine > 0.0);
      const int src = hit ? __ffs(hit) - 1 : nz ? 31 - __clz(nz) : 0;
      if (lane == src) {
        double run = sel_lo + (incl - mine), pick_lo = run, pick_hi = run;
        int pick = -1;
        for (int j0 = v0; j0 < v1; j0 += 4) {
          float x[4], q[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int j = min(j0 + e, V - 1);
            x[e] = p_row[j];
            q[e] = eff == 0 ? q_row[j] : 0.f;
          }
          bool found = false;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const double val = j0 + e < v1 ? value(target(x[e]), q[e], eff) : 0.0;
            if (!found && val > 0.0) {
              pick = j0 + e;
              pick_lo = run;
              pick_hi = run + val;
              found = pick_hi > s_t;
            }
            run += val;
          }
          if (found) break;
        }
        p.next_token[b] = pick < 0 ? -1 : p.vocab_offset + pick;
        if (p.margins && pick >= 0)
          p.margins[(size_t)b * (K + 1) + K] = (float)(fmin(fabs(s_t - pick_lo), fabs(pick_hi - s_t)) / s_total);
      }
    }
  }
  if (S > 1) tc::cluster_wait();      // nobody leaves while its sums may be read
}

}  // namespace

// Parts of a codebook: 2048 codes or more each, eight CTAs (the portable cluster) at most, whatever the number of images.
// One / two / four / eight CTAs, strict, 16 images: 4096 codes 4.8 / 5.4 / 5.4 / 5.7 us, 8192 codes 6.0 / 5.7 / 5.5 / 5.7,
// 16384 codes 9.8 / 7.0 / 5.9 / 5.7, 32768 codes 15.3 / 10.9 / 7.7 / 6.2 (one image: 4.4 / 5.0, 5.3 / 5.4 / 5.2, 8.7 / 6.7 /
// 5.6 / 5.2, 12.4 / 9.2 / 6.2 / 5.3).  At 4096 codes the line is half a microsecond early.
int launch_decide(const float* rows, bool logits, int n_tiles, const Workspace& ws, const DecideParams& p, bool pdl,
                  cudaStream_t s) {
  int S = 1;
  while (S < 8 && p.vocab >= 2048 * 2 * S) S *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(S, p.n_images, 1);
  cfg.blockDim = dim3(kDecideThreads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (S > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = S;
    attr[na].val.clusterDim.y = 1;
    attr[na++].val.clusterDim.z = 1;
  }
  if (pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na++].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  const cudaError_t e = logits ? cudaLaunchKernelEx(&cfg, decide_kernel<true>, ws, p, rows, n_tiles)
                               : cudaLaunchKernelEx(&cfg, decide_kernel<false>, ws, p, rows, n_tiles);
  return e == cudaSuccess ? VVS_OK : VVS_ERR_CUDA;
}

}  // namespace vvs
