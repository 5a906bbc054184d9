// Storage-type-generic kernels of the verify step: embedding gather, RMSNorm, a warp-per-output
// projection kernel, RoPE + KV append, block-vs-cache attention, SwiGLU gating, guidance and
// softmax statistics.  They serve float32 contexts (which have no tensor-core path) and are the
// in-library cross-check of the bf16 tensor-core kernels.
#include <math_constants.h>

#include "tc_common.cuh"
#include "vvs_internal.cuh"

namespace vvs {

template <typename T> struct VecOf;
template <> struct VecOf<float> { static constexpr int n = 4; };
template <> struct VecOf<__nv_bfloat16> { static constexpr int n = 8; };

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}

// 16-byte vector load widened to float
__device__ __forceinline__ void load_vec(const float* p, float* o) {
  float4 v = *reinterpret_cast<const float4*>(p);
  o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void load_vec(const __nv_bfloat16* p, float* o) {
  uint4 u = *reinterpret_cast<const uint4*>(p);
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float2 f = __bfloat1622float2(h[j]);
    o[2 * j] = f.x;
    o[2 * j + 1] = f.y;
  }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// block-wide reductions for blockDim.x <= 1024 (multiple of 32); `red` holds 32 floats
__device__ float block_sum(float v, float* red) {
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  float t = (lane < nw) ? red[lane] : 0.f;
  return warp_sum(t);
}
__device__ float block_max(float v, float* red) {
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_max(v);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  float t = (lane < nw) ? red[lane] : -CUDART_INF_F;
  return warp_max(t);
}

// ---------------------------------------------------------------------------------------------
// x0[r, t, :] = tok_emb[block[b, t]]  (cond and uncond sequences of an image share the block)
template <typename T>
__global__ void embed_kernel(const T* __restrict__ tok_emb, const int32_t* __restrict__ block,
                             float* __restrict__ x, int n_images, int t_len, int d, int tok_rows,
                             int32_t* status) {
  int m = blockIdx.x;
  int r = m / t_len, t = m % t_len;
  int b = r % n_images;
  grid_dep_launch();
  grid_dep_wait();
  int tok = block[b * t_len + t];
  bool ok = tok >= 0 && tok < tok_rows;
  if (!ok && threadIdx.x == 0) atomicOr(status, VVS_DEV_BAD_TOKEN);
  const T* src = tok_emb + (size_t)(ok ? tok : 0) * d;
  float* dst = x + (size_t)m * d;
  for (int i = threadIdx.x; i < d; i += blockDim.x) dst[i] = ok ? to_f(src[i]) : 0.f;
}

template <typename T>
void launch_embed(const T* tok_emb, const int32_t* block, float* x, int n_images, int n_cfg,
                  int t_len, int d, int tok_rows, int32_t* status, cudaStream_t s) {
  embed_kernel<T><<<n_images * n_cfg * t_len, 256, 0, s>>>(tok_emb, block, x, n_images, t_len, d,
                                                           tok_rows, status);
}

// ---------------------------------------------------------------------------------------------
// out[m, :] = x[m, :] * rsqrt(mean(x^2) + eps) * scale
template <typename T>
__global__ void rmsnorm_kernel(const float* __restrict__ x, const T* __restrict__ scale,
                               T* __restrict__ out, int d, float eps) {
  __shared__ float red[32];
  grid_dep_launch();
  grid_dep_wait();
  const float* row = x + (size_t)blockIdx.x * d;
  float ss = 0.f;
  for (int i = threadIdx.x; i < d; i += blockDim.x) ss += row[i] * row[i];
  ss = block_sum(ss, red);
  float rs = rsqrtf(ss / (float)d + eps);
  T* o = out + (size_t)blockIdx.x * d;
  for (int i = threadIdx.x; i < d; i += blockDim.x) o[i] = from_f<T>(row[i] * rs * to_f(scale[i]));
}

// The same for many rows of a bf16 context: one warp per row, 16-byte loads, no shared memory; as a
// programmatic dependent of the projection before it (the row is read after griddepcontrol.wait).
__global__ void __launch_bounds__(128) rmsnorm_rows_kernel(const float* __restrict__ x,
                                                           const __nv_bfloat16* __restrict__ scale,
                                                           __nv_bfloat16* __restrict__ out, int m, int d, float eps) {
  constexpr int kKeep = 12;            // 16-byte pieces of the row a lane keeps in registers (d <= 1536)
  const int lane = threadIdx.x & 31, row_i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (row_i >= m) return;
  const float* row = x + (size_t)row_i * d;
  float4 keep[kKeep];
#pragma unroll
  for (int u = 0; u < kKeep; ++u) {
    const int i = lane * 4 + u * 128;
    keep[u] = i < d ? *reinterpret_cast<const float4*>(row + i) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float ss = 0.f;
#pragma unroll
  for (int u = 0; u < kKeep; ++u)
    ss += keep[u].x * keep[u].x + keep[u].y * keep[u].y + keep[u].z * keep[u].z + keep[u].w * keep[u].w;
  for (int i = lane * 4 + kKeep * 128; i < d; i += 128) {
    const float4 v = *reinterpret_cast<const float4*>(row + i);
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  const float rs = rsqrtf(ss / (float)d + eps);
  __nv_bfloat16* o = out + (size_t)row_i * d;
  auto emit = [&](int i, const float4& v) {
    const uint2 g = *reinterpret_cast<const uint2*>(scale + i);
    const __nv_bfloat162 g0 = *reinterpret_cast<const __nv_bfloat162*>(&g.x);
    const __nv_bfloat162 g1 = *reinterpret_cast<const __nv_bfloat162*>(&g.y);
    __nv_bfloat162 r0 = __floats2bfloat162_rn(v.x * rs * __bfloat162float(g0.x), v.y * rs * __bfloat162float(g0.y));
    __nv_bfloat162 r1 = __floats2bfloat162_rn(v.z * rs * __bfloat162float(g1.x), v.w * rs * __bfloat162float(g1.y));
    uint2 pk;
    pk.x = *reinterpret_cast<uint32_t*>(&r0);
    pk.y = *reinterpret_cast<uint32_t*>(&r1);
    *reinterpret_cast<uint2*>(o + i) = pk;
  };
#pragma unroll
  for (int u = 0; u < kKeep; ++u) {
    const int i = lane * 4 + u * 128;
    if (i < d) emit(i, keep[u]);
  }
  for (int i = lane * 4 + kKeep * 128; i < d; i += 128) emit(i, *reinterpret_cast<const float4*>(row + i));
}

// Few rows: one CTA of 128 threads per row (every thread holds at most kKeepB 16-byte pieces), so the
// row's loads are all in flight at once and the kernel is two dependent memory round trips long.
__global__ void __launch_bounds__(128) rmsnorm_row_block_kernel(const float* __restrict__ x,
                                                                const __nv_bfloat16* __restrict__ scale,
                                                                __nv_bfloat16* __restrict__ out, int d, float eps) {
  constexpr int kKeepB = 8;            // d <= 4096
  __shared__ float red[4];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  uint2 g[kKeepB];
#pragma unroll
  for (int u = 0; u < kKeepB; ++u) {                  // the scale is an input of the whole step: before the wait
    const int i = tid * 4 + u * 512;
    g[u] = i < d ? *reinterpret_cast<const uint2*>(scale + i) : make_uint2(0u, 0u);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const float* row = x + (size_t)blockIdx.x * d;
  float4 keep[kKeepB];
  float ss = 0.f;
#pragma unroll
  for (int u = 0; u < kKeepB; ++u) {
    const int i = tid * 4 + u * 512;
    keep[u] = i < d ? *reinterpret_cast<const float4*>(row + i) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int u = 0; u < kKeepB; ++u)
    ss += keep[u].x * keep[u].x + keep[u].y * keep[u].y + keep[u].z * keep[u].z + keep[u].w * keep[u].w;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if (lane == 0) red[warp] = ss;
  __syncthreads();
  const float rs = rsqrtf((red[0] + red[1] + red[2] + red[3]) / (float)d + eps);
  __nv_bfloat16* o = out + (size_t)blockIdx.x * d;
#pragma unroll
  for (int u = 0; u < kKeepB; ++u) {
    const int i = tid * 4 + u * 512;
    if (i < d) {
      const __nv_bfloat162 g0 = *reinterpret_cast<const __nv_bfloat162*>(&g[u].x);
      const __nv_bfloat162 g1 = *reinterpret_cast<const __nv_bfloat162*>(&g[u].y);
      __nv_bfloat162 r0 = __floats2bfloat162_rn(keep[u].x * rs * __bfloat162float(g0.x), keep[u].y * rs * __bfloat162float(g0.y));
      __nv_bfloat162 r1 = __floats2bfloat162_rn(keep[u].z * rs * __bfloat162float(g1.x), keep[u].w * rs * __bfloat162float(g1.y));
      uint2 pk;
      pk.x = *reinterpret_cast<uint32_t*>(&r0);
      pk.y = *reinterpret_cast<uint32_t*>(&r1);
      *reinterpret_cast<uint2*>(o + i) = pk;
    }
  }
}

template <typename T>
void launch_rmsnorm(const float* x, const T* scale, T* out, int m, int d, float eps, cudaStream_t s, bool pdl) {
  launch_kernel(rmsnorm_kernel<T>, dim3(m), dim3(256), 0, pdl, s, x, scale, out, d, eps);
}

static cudaError_t launch_dependent(const void* fn, dim3 grid, dim3 block, void** args, bool pdl, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

void launch_rmsnorm_rows(const float* x, const __nv_bfloat16* scale, __nv_bfloat16* out, int m, int d, float eps,
                         bool pdl, cudaStream_t s) {
  if (m <= 64 && d <= 4096) {          // few rows: a CTA per row
    void* args1[] = {&x, &scale, &out, &d, &eps};
    launch_dependent(reinterpret_cast<const void*>(rmsnorm_row_block_kernel), dim3(m), dim3(128), args1, pdl, s);
    return;
  }
  void* args[] = {&x, &scale, &out, &m, &d, &eps};
  launch_dependent(reinterpret_cast<const void*>(rmsnorm_rows_kernel), dim3((m + 3) / 4), dim3(128), args, pdl, s);
}

// ---------------------------------------------------------------------------------------------
// Projections on the CUDA cores: acc[m, n] = sum_k a[m, k] * w[n, k], one warp per weight row (or pair of rows), MT
// activation rows per pass, with what surrounds a projection folded in:
//   QKV     a = norm(x) * scale; rotation of q and k pairs, q to its buffer, k and v to cache slots L_r + t
//   GATEUP  a = norm(x) * scale; silu(gate) * up
//   ADD     residual x += acc
//   STORE   plain product
//   NORM_STORE  a = norm(x) * scale, which is also written out; plain product (the LM head after the last layer)
// A small model's step is a chain of dependent kernels of a few microseconds each, so what counts is their number
// (five per layer instead of ten) and the loads in a row inside one: weights are requested before
// griddepcontrol.wait, the activations of all rows of a piece together and a piece ahead (one row after the other they
// were as many round trips to L2: 8-10 us a kernel).  In float32 1/rms multiplies the finished sums, so no pass over the
// rows comes first, and the final norm is part of the LM head.  (Tiny float32 step of 5 rows: 128 -> 66 -> 49 us.)
template <typename T>
struct RowGemm {
  int m, n, k;                 // n: warps' worth of columns (pairs for QKV)
  const T* a;                  // ADD, STORE: activations [m, k]
  const float* x_in;           // QKV, GATEUP, NORM_STORE: residual rows [m, k]
  const T* scale; float eps;
  const T* w; const T* w2;     // GATEUP: gate, up
  float* c; int ldc;           // ADD, STORE
  T* act;                      // GATEUP [m, n]; NORM_STORE: the normalised rows [m, k]
  T* q; T* kv_k; T* kv_v;      // QKV
  const float* inv_freq; const int32_t* cache_len; int32_t* status;
  int d, n_heads, hd, s_max, rope_mode, grid_w, n_prefix, layer, kv_rows, t_len;
};

template <typename T, int EPI>
__global__ void __launch_bounds__(128) row_gemm_kernel(const RowGemm<T> p) {
  constexpr int VEC = VecOf<T>::n, MT = 8;
  constexpr bool NORM = EPI == ROW_QKV || EPI == ROW_GATEUP || EPI == ROW_NORM_STORE;
  constexpr int NW = EPI == ROW_QKV || EPI == ROW_GATEUP ? 2 : 1, PF = NORM ? 4 : 8;           // weight rows per warp, pieces of them in flight
  constexpr bool FOLD = NORM && sizeof(T) == 4;                 // 1/rms multiplies the sums; nothing is rounded before them
  __shared__ float s_rs[MT];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int col = blockIdx.x * 4 + warp, m0 = blockIdx.y * MT, k = p.k;
  const bool live = col < p.n;
  const T* w[NW];
  w[0] = p.w + (size_t)(EPI == ROW_QKV ? 2 * col : col) * k;
  if (NW == 2) w[NW - 1] = EPI == ROW_QKV ? w[0] + k : p.w2 + (size_t)col * k;
  uint4 wv[NW][PF];
  auto fetch = [&](int base) {
#pragma unroll
    for (int j = 0; j < PF; ++j) {
      const int k0 = base + (j * 32 + lane) * VEC;
#pragma unroll
      for (int r = 0; r < NW; ++r)
        wv[r][j] = live && k0 < k ? __ldg(reinterpret_cast<const uint4*>(w[r] + k0)) : make_uint4(0, 0, 0, 0);
    }
  };
  fetch(0);
  grid_dep_launch();
  grid_dep_wait();
  if (NORM && !FOLD) {
    for (int i = warp; i < MT; i += 4) {
      float ss = 0.f;
      if (m0 + i < p.m) {
        const float* row = p.x_in + (size_t)(m0 + i) * k;
#pragma unroll 4
        for (int j = lane * 4; j < k; j += 128) {
          const float4 v = *reinterpret_cast<const float4*>(row + j);
          ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
        }
      }
      ss = warp_sum(ss);
      if (lane == 0) s_rs[i] = rsqrtf(ss / (float)k + p.eps);
    }
    __syncthreads();
  }
  if (!live && EPI != ROW_NORM_STORE) return;
  float acc[NW][MT], ss[MT];
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    ss[i] = 0.f;
#pragma unroll
    for (int r = 0; r < NW; ++r) acc[r][i] = 0.f;
  }
  // A piece's activations of all rows are requested before the first is used, the next piece's with them (rows and columns
  // past the end repeat the last ones; their weights are zero, their sums are not stored).
  const int last_m = p.m - 1 - m0, last_k = k - VEC;
  const T* a0 = NORM ? nullptr : p.a + (size_t)m0 * k;
  const float* x0 = NORM ? p.x_in + (size_t)m0 * k : nullptr;
  constexpr int AV = NORM ? VEC / 4 : 1;                        // 16-byte pieces of a row's activations
  uint4 av4[2][MT][AV];
  auto request = [&](int slot, int k0) {
    const int kc = min(k0, last_k);
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int q = 0; q < AV; ++q)
        av4[slot][i][q] = NORM ? *reinterpret_cast<const uint4*>(x0 + (size_t)min(i, last_m) * k + kc + 4 * q)
                               : *reinterpret_cast<const uint4*>(a0 + (size_t)min(i, last_m) * k + kc);
  };
  request(0, lane * VEC);
  for (int base = 0; base < k; base += PF * 32 * VEC) {
    if (base > 0) fetch(base);
#pragma unroll
    for (int j = 0; j < PF; ++j) {
      const int k0 = base + (j * 32 + lane) * VEC;
      if (base + j * 32 * VEC >= k) break;
      request((j + 1) & 1, k0 + 32 * VEC);
      float wf[NW][VEC], sc[VEC];
#pragma unroll
      for (int r = 0; r < NW; ++r) load_vec(reinterpret_cast<const T*>(&wv[r][j]), wf[r]);
      if (NORM) load_vec(p.scale + min(k0, last_k), sc);
#pragma unroll
      for (int i = 0; i < MT; ++i) {
        float av[VEC];
        if (NORM) {
          const float rs = FOLD ? 1.f : s_rs[i];
#pragma unroll
          for (int q = 0; q < AV; ++q) load_vec(reinterpret_cast<const float*>(&av4[j & 1][i][q]), av + 4 * q);
#pragma unroll
          for (int e = 0; e < VEC; ++e) {
            if (FOLD) ss[i] = k0 < k ? fmaf(av[e], av[e], ss[i]) : ss[i];
            av[e] = FOLD ? av[e] * sc[e] : to_f(from_f<T>(av[e] * rs * sc[e]));
          }
        } else {
          load_vec(reinterpret_cast<const T*>(&av4[j & 1][i][0]), av);
        }
#pragma unroll
        for (int r = 0; r < NW; ++r)
#pragma unroll
          for (int e = 0; e < VEC; ++e) acc[r][i] = fmaf(av[e], wf[r][e], acc[r][i]);
      }
    }
  }
  float v[NW];                                   // lanes 4 i .. 4 i + 3 keep row m0 + i
#pragma unroll
  for (int r = 0; r < NW; ++r) v[r] = tc::warp_sums(acc[r], lane);
  const int row = m0 + (lane >> 2);
  if (FOLD) {
    const float rs = rsqrtf(tc::warp_sums(ss, lane) / (float)k + p.eps);
#pragma unroll
    for (int r = 0; r < NW; ++r) v[r] *= rs;
    if (EPI == ROW_NORM_STORE && blockIdx.x == 0) {               // the normalised rows themselves, two per warp
      for (int i = warp; i < MT && m0 + i < p.m; i += 4) {
        const float rs_i = __shfl_sync(0xffffffffu, rs, 4 * i);
        for (int j = lane; j < k; j += 32) p.act[(size_t)(m0 + i) * k + j] = from_f<T>(p.x_in[(size_t)(m0 + i) * k + j] * rs_i * to_f(p.scale[j]));
      }
    }
  }
  if ((lane & 3) || row >= p.m || !live) return;
  if constexpr (EPI == ROW_ADD) {
    p.c[(size_t)row * p.ldc + col] += v[0];
  } else if constexpr (EPI == ROW_STORE || EPI == ROW_NORM_STORE) {
    p.c[(size_t)row * p.ldc + col] = v[0];
  } else if constexpr (EPI == ROW_GATEUP) {
    p.act[(size_t)row * p.n + col] = from_f<T>(v[0] / (1.f + expf(-v[0])) * v[NW - 1]);
  } else {
    const int r = row / p.t_len, t = row - r * p.t_len, fill = p.cache_len[r], pos = fill + t;
    const bool ok = fill >= 0 && fill + p.t_len <= p.s_max;
    if (!ok && col == 0) atomicOr(p.status, VVS_DEV_CACHE_OVERFLOW);
    const int n = 2 * col, sec = n / p.d, e = n - sec * p.d, h = e / p.hd, i2 = e - h * p.hd;
    float y0 = v[0], y1 = v[NW - 1];
    if (sec < 2) {
      float coord = 0.f;                         // coordinate driving this pair: first / second head half
      if (p.rope_mode == VVS_ROPE_1D) {
        coord = (float)pos;
      } else if (p.rope_mode == VVS_ROPE_2D_GRID && pos >= p.n_prefix) {
        const int g = pos - p.n_prefix;
        coord = (float)(i2 < p.hd / 2 ? g / p.grid_w : g % p.grid_w);
      }
      float sn, cs;
      sincosf(coord * p.inv_freq[i2 >> 1], &sn, &cs);
      const float a0 = y0;
      y0 = a0 * cs - y1 * sn;
      y1 = a0 * sn + y1 * cs;
    }
    T* dst = nullptr;
    if (sec == 0) dst = p.q + (size_t)row * p.d + e;
    else if (ok) dst = (sec == 1 ? p.kv_k : p.kv_v) + ((((size_t)p.layer * p.kv_rows + r) * p.n_heads + h) * p.s_max + pos) * p.hd + i2;
    if (dst) {
      dst[0] = from_f<T>(y0);
      dst[1] = from_f<T>(y1);
    }
  }
}

template <typename T>
static void launch_row_gemm(int epi, const RowGemm<T>& p, bool pdl, cudaStream_t s) {
  const dim3 grid((p.n + 3) / 4, (p.m + 7) / 8);
  if (epi == ROW_QKV) launch_kernel(row_gemm_kernel<T, ROW_QKV>, grid, dim3(128), 0, pdl, s, p);
  else if (epi == ROW_GATEUP) launch_kernel(row_gemm_kernel<T, ROW_GATEUP>, grid, dim3(128), 0, pdl, s, p);
  else if (epi == ROW_ADD) launch_kernel(row_gemm_kernel<T, ROW_ADD>, grid, dim3(128), 0, pdl, s, p);
  else launch_kernel(row_gemm_kernel<T, ROW_STORE>, grid, dim3(128), 0, pdl, s, p);
}

template <typename T>
void launch_row_qkv(const float* x, const T* scale, float eps, const T* w, const float* inv_freq, T* q, T* kv_k, T* kv_v,
                    const int32_t* cache_len, const vvs_model_desc& md, int layer, int kv_rows, int m, int t_len, int32_t* status,
                    bool pdl, cudaStream_t s) {
  RowGemm<T> p{};
  p.m = m; p.n = 3 * md.d_model / 2; p.k = md.d_model; p.x_in = x; p.scale = scale; p.eps = eps; p.w = w; p.q = q; p.kv_k = kv_k;
  p.kv_v = kv_v; p.inv_freq = inv_freq; p.cache_len = cache_len; p.status = status; p.d = md.d_model; p.n_heads = md.n_heads;
  p.hd = md.head_dim; p.s_max = md.s_max; p.rope_mode = md.rope_mode; p.grid_w = md.rope_grid_w; p.n_prefix = md.n_prefix;
  p.layer = layer; p.kv_rows = kv_rows; p.t_len = t_len;
  launch_row_gemm<T>(ROW_QKV, p, pdl, s);
}
// hid = norm(x) * scale, c[m, n] = hid . w[n] (float32: bf16 contexts round hid before the product, see rmsnorm_kernel)
void launch_row_norm_product(const float* x, const float* scale, float eps, const float* w, float* hid, float* c, int m, int n, int k,
                             bool pdl, cudaStream_t s) {
  RowGemm<float> p{};
  p.m = m; p.n = n; p.k = k; p.x_in = x; p.scale = scale; p.eps = eps; p.w = w; p.act = hid; p.c = c; p.ldc = n;
  launch_kernel(row_gemm_kernel<float, ROW_NORM_STORE>, dim3((n + 3) / 4, (m + 7) / 8), dim3(128), 0, pdl, s, p);
}
template <typename T>
void launch_row_gateup(const float* x, const T* scale, float eps, const T* gate, const T* up, T* act, int m, int ff, int d, bool pdl,
                       cudaStream_t s) {
  RowGemm<T> p{};
  p.m = m; p.n = ff; p.k = d; p.x_in = x; p.scale = scale; p.eps = eps; p.w = gate; p.w2 = up; p.act = act;
  launch_row_gemm<T>(ROW_GATEUP, p, pdl, s);
}
// c[m, n] (+)= sum_k a[m, k] * w[n, k]
template <typename T>
void launch_row_product(const T* a, const T* w, float* c, int m, int n, int k, int ldc, bool accumulate, bool pdl, cudaStream_t s) {
  RowGemm<T> p{};
  p.m = m; p.n = n; p.k = k; p.a = a; p.w = w; p.c = c; p.ldc = ldc;
  launch_row_gemm<T>(accumulate ? ROW_ADD : ROW_STORE, p, pdl, s);
}

// ---------------------------------------------------------------------------------------------
// Block-vs-cache attention: query row t of sequence r sees cache slots [0, L_r + t].  One CTA per (head, sequence,
// query row): scores by groups of lanes that read a key row with 16-byte loads side by side, then softmax, then the
// output by (column group, key phase) with a reduction over the phases.  A row's keys stay in L2 / L1 between the
// CTAs of a head; with a few dozen (head, row) pairs the kernel is a chain of three round trips (40 -> 7.3 us with four
// heads, 5 rows and 69 keys, where a lane walked a whole key and a warp all keys of a column in turn).
template <typename T, int HD>
__global__ void __launch_bounds__(128) attention_kernel(const T* __restrict__ q, const T* __restrict__ kv_k,
                                                        const T* __restrict__ kv_v, const int32_t* __restrict__ cache_len,
                                                        T* __restrict__ out, int d, int n_heads, int s_max, int layer,
                                                        int kv_rows, int t_len) {
  extern __shared__ float sc[];                   // scores [s_max], then the phases' sums [kPh][HD]
  constexpr int VEC = VecOf<T>::n, kLanes = HD / (2 * VEC), kGroups = 128 / kLanes;
  constexpr int kCols = HD / VEC, kPh = 128 / kCols;
  __shared__ float red[32];
  const int h = blockIdx.x, r = blockIdx.y, t = blockIdx.z, tid = threadIdx.x;
  grid_dep_launch();
  const int fill = cache_len[r];
  const size_t o = ((size_t)r * t_len + t) * d + (size_t)h * HD;
  const size_t base = (((size_t)layer * kv_rows + r) * n_heads + h) * (size_t)s_max * HD;
  const bool ok = fill >= 0 && fill + t_len <= s_max;
  if (ok && ((reinterpret_cast<uintptr_t>(kv_k) | reinterpret_cast<uintptr_t>(kv_v)) & 127) == 0) {
    // the cached rows into L1 while the projection before this kernel is still running (it writes slots fill .. only, and
    // a row is whole lines)
    constexpr int kLines = HD * (int)sizeof(T) / 128;
    for (int i = tid; i < fill * kLines && i < 512; i += 128) {
      const size_t at = base + (size_t)i * (128 / sizeof(T));
      asm volatile("prefetch.global.L1 [%0];" ::"l"(kv_k + at));
      asm volatile("prefetch.global.L1 [%0];" ::"l"(kv_v + at));
    }
  }
  grid_dep_wait();
  if (!ok) {
    for (int i = tid; i < HD; i += 128) out[o + i] = from_f<T>(0.f);
    return;
  }
  const int nk = fill + t + 1;
  const float scale = rsqrtf((float)HD);
  // ---- scores: group g takes keys g, g + kGroups, ..; lane c of it columns [c VEC, ..) and the same in the second half
  const int g = tid / kLanes, c = tid & (kLanes - 1);
  float q0[VEC], q1[VEC];
  load_vec(q + o + c * VEC, q0);
  load_vec(q + o + HD / 2 + c * VEC, q1);
  float mx = -CUDART_INF_F;
#pragma unroll 4
  for (int j0 = 0; j0 < nk; j0 += kGroups) {
    const int j = j0 + g;
    float k0[VEC], k1[VEC], s = 0.f;
    const T* kr = kv_k + base + (size_t)(j < nk ? j : 0) * HD + c * VEC;
    load_vec(kr, k0);
    load_vec(kr + HD / 2, k1);
#pragma unroll
    for (int e = 0; e < VEC; ++e) s = fmaf(q0[e], k0[e], fmaf(q1[e], k1[e], s));
#pragma unroll
    for (int w = kLanes / 2; w > 0; w >>= 1) s += __shfl_xor_sync(0xffffffffu, s, w);
    s *= scale;
    if (j < nk) {
      mx = fmaxf(mx, s);
      if (c == 0) sc[j] = s;
    }
  }
  mx = block_max(mx, red);                        // (its barriers also publish the scores)
  float sum = 0.f;
  for (int j = tid; j < nk; j += 128) {
    const float e = expf(sc[j] - mx);
    sc[j] = e;
    sum += e;
  }
  sum = block_sum(sum, red);
  // ---- output ----
  const int cg = tid % kCols, ph = tid / kCols;
  float acc[VEC];
#pragma unroll
  for (int e = 0; e < VEC; ++e) acc[e] = 0.f;
  const T* vb = kv_v + base + cg * VEC;
#pragma unroll 8
  for (int j = ph; j < nk; j += kPh) {
    float v[VEC];
    load_vec(vb + (size_t)j * HD, v);
    const float pj = sc[j];
#pragma unroll
    for (int e = 0; e < VEC; ++e) acc[e] = fmaf(pj, v[e], acc[e]);
  }
  float* part = sc + s_max;
#pragma unroll
  for (int e = 0; e < VEC; ++e) part[ph * HD + cg * VEC + e] = acc[e];
  __syncthreads();
  const float inv = 1.f / sum;
  for (int i = tid; i < HD; i += 128) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kPh; ++w) s += part[w * HD + i];
    out[o + i] = from_f<T>(s * inv);
  }
}

template <typename T>
void launch_attention(const T* q, const T* kv_k, const T* kv_v, const int32_t* cache_len, T* out,
                      const vvs_model_desc& md, int layer, int kv_rows, int n_rows, int t_len, bool pdl, cudaStream_t s) {
  // phases x head_dim = 128 x VEC whatever the head_dim
  const size_t smem = ((size_t)md.s_max + 128 * VecOf<T>::n) * sizeof(float);
  auto* kernel = md.head_dim == 64 ? attention_kernel<T, 64> : attention_kernel<T, 128>;
  if (smem > 48 * 1024) ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), (int)smem);
  launch_kernel(kernel, dim3(md.n_heads, n_rows, t_len), dim3(128), smem, pdl, s, q, kv_k, kv_v, cache_len, out, (int)md.d_model,
                (int)md.n_heads, (int)md.s_max, layer, kv_rows, t_len);
}

// ---------------------------------------------------------------------------------------------
// act[m, j] = silu(gate[m, j]) * up[m, j]; grid (column chunks of 1024, rows), 4 columns per thread
template <typename T>
__global__ void silu_mul_kernel(float* __restrict__ gu, T* __restrict__ act, int ff, int clear_src) {
  float* row = gu + (size_t)blockIdx.y * 2 * ff;
  T* o = act + (size_t)blockIdx.y * ff;
  const int j = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");   // returns at once unless launched as a programmatic dependent
  if (j >= ff) return;                       // ff is a multiple of 8
  const float4 g = *reinterpret_cast<const float4*>(row + j);
  const float4 u = *reinterpret_cast<const float4*>(row + ff + j);
  o[j] = from_f<T>(g.x / (1.f + expf(-g.x)) * u.x);
  o[j + 1] = from_f<T>(g.y / (1.f + expf(-g.y)) * u.y);
  o[j + 2] = from_f<T>(g.z / (1.f + expf(-g.z)) * u.z);
  o[j + 3] = from_f<T>(g.w / (1.f + expf(-g.w)) * u.w);
  if (clear_src) {                             // split-K sums are added into this buffer: leave it zero
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4*>(row + j) = z;
    *reinterpret_cast<float4*>(row + ff + j) = z;
  }
}

template <typename T>
void launch_silu_mul(float* gu, T* act, int m, int ff, cudaStream_t s, bool clear_src, bool pdl) {
  int clear = clear_src ? 1 : 0;
  void* args[] = {&gu, &act, &ff, &clear};
  launch_dependent(reinterpret_cast<const void*>(silu_mul_kernel<T>), dim3((ff + 1023) / 1024, m), dim3(256), args,
                   pdl, s);
}

// ---------------------------------------------------------------------------------------------
// guided logits / temperature:  l = l_u + s (l_c - l_u)  (or l_c without guidance), and the row's max and sum of
// exp(l - max) as a single "tile" of softmax partials
__global__ void __launch_bounds__(256) guide_stats_kernel(const float* __restrict__ raw, float* __restrict__ logits,
                                                          float* __restrict__ part_m, float* __restrict__ part_s, int n_images,
                                                          int n_cfg, int rows_per_seq, int v, float cfg_scale, float inv_temp) {
  __shared__ float red[32];
  const int row = blockIdx.x;  // b * rows_per_seq + t
  grid_dep_launch();
  grid_dep_wait();
  const float* lc = raw + (size_t)row * v;
  const float* lu = raw + ((size_t)n_images * rows_per_seq + row) * v;
  float* o = logits + (size_t)row * v;
  float mx = -CUDART_INF_F;
#pragma unroll 4
  for (int j = threadIdx.x; j < v; j += 256) {
    float l = lc[j];
    if (n_cfg == 2) {
      const float u = lu[j];
      l = u + cfg_scale * (l - u);
    }
    l *= inv_temp;
    o[j] = l;
    mx = fmaxf(mx, l);
  }
  mx = block_max(mx, red);
  float sum = 0.f;
  for (int j = threadIdx.x; j < v; j += 256) sum += expf(o[j] - mx);      // this thread's own values
  sum = block_sum(sum, red);
  if (threadIdx.x == 0) {
    part_m[row] = mx;
    part_s[row] = sum;
  }
}

void launch_guide_stats(const float* raw, float* logits, float* part_m, float* part_s, int n_images, int n_cfg, int rows_per_seq,
                        int v, float cfg_scale, float inv_temp, bool pdl, cudaStream_t s) {
  launch_kernel(guide_stats_kernel, dim3(n_images * rows_per_seq), dim3(256), 0, pdl, s, raw, logits, part_m, part_s, n_images,
                n_cfg, rows_per_seq, v, cfg_scale, inv_temp);
}

// explicit instantiations
#define VVS_INSTANTIATE(T)                                                                             \
  template void launch_embed<T>(const T*, const int32_t*, float*, int, int, int, int, int, int32_t*,    \
                                cudaStream_t);                                                          \
  template void launch_rmsnorm<T>(const float*, const T*, T*, int, int, float, cudaStream_t, bool);     \
  template void launch_row_qkv<T>(const float*, const T*, float, const T*, const float*, T*, T*, T*,    \
                                  const int32_t*, const vvs_model_desc&, int, int, int, int, int32_t*,  \
                                  bool, cudaStream_t);                                                  \
  template void launch_row_gateup<T>(const float*, const T*, float, const T*, const T*, T*, int, int,   \
                                     int, bool, cudaStream_t);                                          \
  template void launch_row_product<T>(const T*, const T*, float*, int, int, int, int, bool, bool,       \
                                      cudaStream_t);                                                    \
  template void launch_attention<T>(const T*, const T*, const T*, const int32_t*, T*,                   \
                                    const vvs_model_desc&, int, int, int, int, bool, cudaStream_t);     \
  template void launch_silu_mul<T>(float*, T*, int, int, cudaStream_t, bool, bool);
VVS_INSTANTIATE(float)
VVS_INSTANTIATE(__nv_bfloat16)

}  // namespace vvs
