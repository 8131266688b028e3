// Segment-mean pooling, router softmax, causal shift, and their backward
// (Eq. 3 and Algorithm 1 of the Lory paper).  All arithmetic in fp32.
#include "routing.cuh"

#include <cooperative_groups.h>

namespace lory {

// ---------------------------------------------------------------------------------------
// h_bar[s, :] = (1/T) sum_t x[s*T + t, :]
// HBM-bound (x once).  A block of 8 warps sums a run of a segment's tokens for 32 * VEC columns, warp w rows w, w+8, ...
// of it, a lane VEC consecutive columns (one 16-byte load per row).  Where there are too few segments to fill the GPU,
// the blocks of a cluster (up to 8) share a segment's tokens and the first adds their sums through distributed shared
// memory, in a fixed order (2 segments of 1000 tokens, d = 1024: 30 -> 4 us; with enough segments clusters only cost).
// Another block's shared memory may be written only once that block is known to run: every block arrives at the cluster's
// barrier first thing and waits on it right before its write, when all have long arrived.
// ---------------------------------------------------------------------------------------
template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
  static constexpr int N = 4;
  __device__ static void load(const float* p, float (&v)[4]) {
    float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  }
};
template <>
struct Vec16<bf16> {
  static constexpr int N = 8;
  __device__ static void load(const bf16* p, float (&v)[8]) {
    uint4 q = *reinterpret_cast<const uint4*>(p);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&q);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float2 f = __bfloat1622float2(h[i]);
      v[2 * i] = f.x; v[2 * i + 1] = f.y;
    }
  }
};

template <typename T>
__global__ void __launch_bounds__(256) pool_kernel(const T* __restrict__ x, float* __restrict__ h_bar,
                                                    int Tseg, int d, int parts, uint32_t* status) {
  constexpr int VEC = Vec16<T>::N;
  const int s = blockIdx.x / parts, part = blockIdx.x - s * parts;   // part = rank in the cluster
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int col = (blockIdx.y * 32 + lane) * VEC;
  __shared__ float red[8][32 * VEC];
  __shared__ float xch[8][32 * VEC];   // the first block's: one row per block of the cluster
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  if (parts > 1) cluster.barrier_arrive();
  pdl_launch();
  pdl_wait();
  if (status && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 64) status[threadIdx.x] = 0;
  const int run = (Tseg + parts - 1) / parts, t_end = min(Tseg, (part + 1) * run);
  float acc[VEC];
#pragma unroll
  for (int i = 0; i < VEC; ++i) acc[i] = 0.f;
  const bool vec_ok = (col + VEC <= d) && (d % VEC == 0);
  const T* base = x + (size_t)s * Tseg * d;
  int t = part * run + warp;
  if (vec_ok) {
    // four independent 16-byte loads in flight per lane
    for (; t + 24 < t_end; t += 32) {
      float v0[VEC], v1[VEC], v2[VEC], v3[VEC];
      Vec16<T>::load(base + (size_t)t * d + col, v0);
      Vec16<T>::load(base + (size_t)(t + 8) * d + col, v1);
      Vec16<T>::load(base + (size_t)(t + 16) * d + col, v2);
      Vec16<T>::load(base + (size_t)(t + 24) * d + col, v3);
#pragma unroll
      for (int i = 0; i < VEC; ++i) acc[i] += (v0[i] + v1[i]) + (v2[i] + v3[i]);
    }
#pragma unroll 4
    for (; t < t_end; t += 8) {
      float v[VEC];
      Vec16<T>::load(base + (size_t)t * d + col, v);
#pragma unroll
      for (int i = 0; i < VEC; ++i) acc[i] += v[i];
    }
  } else {
    for (; t < t_end; t += 8) {
      const T* row = base + (size_t)t * d;
#pragma unroll
      for (int i = 0; i < VEC; ++i)
        if (col + i < d) acc[i] += to_f32(row[col + i]);
    }
  }
#pragma unroll
  for (int i = 0; i < VEC; ++i) red[warp][lane * VEC + i] = acc[i];
  __syncthreads();
  const int c = threadIdx.x, gc = blockIdx.y * 32 * VEC + c;
  float sum = 0.f;
  if (c < 32 * VEC) {
#pragma unroll
    for (int w = 0; w < 8; ++w) sum += red[w][c];
  }
  if (parts > 1) {
    cluster.barrier_wait();   // the first block has started
    if (c < 32 * VEC) *cluster.map_shared_rank(&xch[part][c], 0) = sum;
    cluster.sync();
    if (part > 0) return;
    sum = 0.f;
    if (c < 32 * VEC)
      for (int q = 0; q < parts; ++q) sum += xch[q][c];
  }
  if (c < 32 * VEC && gc < d) h_bar[(size_t)s * d + gc] = sum / (float)Tseg;
}

// ---------------------------------------------------------------------------------------
// p_s = softmax(W_r h_bar_s); w_{b,0} = p_{b,0}; w_{b,n} = p_{b,n-1}.
// One block per segment; its warps (one per expert when E <= 32) take the experts in turn.
// ---------------------------------------------------------------------------------------
// One routing-weight row: fp32 (workspace and, if asked, the caller's copy) and the bf16 hi + lo tables.
__device__ __forceinline__ void write_weight_row(const float* p_sm, size_t row, int E, int lane, float* w_out,
                                                 const RouteExtra& ex) {
  for (int e = lane; e < E; e += 32) {
    w_out[row * E + e] = p_sm[e];
    if (ex.w_copy) ex.w_copy[row * E + e] = p_sm[e];
  }
  if (ex.hi) {
    for (int e = lane; e < ex.Epad; e += 32) {
      const float v = e < E ? p_sm[e] : 0.f;
      const bf16 h = __float2bfloat16_rn(v);
      ex.hi[row * ex.Epad + e] = h;
      ex.lo[row * ex.Epad + e] = __float2bfloat16_rn(v - __bfloat162float(h));
    }
  }
  if (ex.frag) {
    const int kt = (E + 15) >> 4;
    for (int e = lane; e < kt * 16; e += 32) {
      const float v = e < E ? p_sm[e] : 0.f;
      const bf16 h = __float2bfloat16_rn(v);
      bf16* dst = ex.frag + w_frag_offset(row, e, kt);
      dst[0] = h;
      dst[256] = __float2bfloat16_rn(v - __bfloat162float(h));
    }
  }
  if (ex.comb) {
    // [hi | lo | hi | hi | lo | lo], 32 columns each
    for (int c = lane; c < 192; c += 32) {
      const int e = c & 31, part = c >> 5;
      const float v = e < E ? p_sm[e] : 0.f;
      const bf16 h = __float2bfloat16_rn(v);
      const bool is_hi = part == 0 || part == 2 || part == 3;
      ex.comb[row * 192 + c] = is_hi ? h : __float2bfloat16_rn(v - __bfloat162float(h));
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(1024) router_kernel(const float* __restrict__ h_bar,
                                                     const T* __restrict__ w_r, float* __restrict__ p_ws,
                                                     float* __restrict__ route_p, float* __restrict__ w_out,
                                                     int N, int d, int E, int prefix, const RouteExtra ex) {
  extern __shared__ float sm[];  // z[E]
  const int s = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* h = h_bar + (size_t)s * d;
  const int nwarps = blockDim.x >> 5;
  pdl_launch();
  pdl_wait();
  for (int e = warp; e < E; e += nwarps) {
    const T* wr = w_r + (size_t)e * d;
    float acc = 0.f;
    constexpr int VEC = Vec16<T>::N;
    if (d % VEC == 0) {
#pragma unroll 4
      for (int j = lane * VEC; j < d; j += 32 * VEC) {
        float wv[VEC];
        Vec16<T>::load(wr + j, wv);
#pragma unroll
        for (int i = 0; i < VEC; i += 4) {
          float4 hv = *reinterpret_cast<const float4*>(h + j + i);
          acc += wv[i] * hv.x + wv[i + 1] * hv.y + wv[i + 2] * hv.z + wv[i + 3] * hv.w;
        }
      }
    } else {
      for (int j = lane; j < d; j += 32) acc += to_f32(wr[j]) * h[j];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) sm[e] = acc;
  }
  __syncthreads();
  if (warp == 0) {
    float m = -INFINITY;
    for (int e = lane; e < E; e += 32) m = fmaxf(m, sm[e]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float sum = 0.f;
    for (int e = lane; e < E; e += 32) {
      float ez = expf(sm[e] - m);
      sm[e] = ez;
      sum += ez;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const float inv = 1.0f / sum;
    const int n = s % N;
    for (int e = lane; e < E; e += 32) {
      float p = sm[e] * inv;
      sm[e] = p;
      p_ws[(size_t)s * E + e] = p;
      if (route_p) route_p[(size_t)s * E + e] = p;
    }
    __syncwarp();
    if (prefix) {
      // prefix routing: the first segment's probabilities route every segment of its sequence
      if (n == 0)
        for (int m2 = 0; m2 < N; ++m2) write_weight_row(sm, (size_t)(s + m2), E, lane, w_out, ex);
    } else {
      if (n == 0) write_weight_row(sm, (size_t)s, E, lane, w_out, ex);          // first segment routes itself
      if (n < N - 1) write_weight_row(sm, (size_t)(s + 1), E, lane, w_out, ex);  // and every segment routes the next
    }
  }
}

// ---------------------------------------------------------------------------------------
// Backward of the router path.
// ---------------------------------------------------------------------------------------
// dw[s,:] = sum of the partial slabs; dz_s = p_s * (dp_s - <dp_s, p_s>) with dp_{b,n} = dw_{b,n+1} (0 for the
// last segment); dh_bar_s = W_r^T dz_s.  One block per segment.  Latency-bound: the block's threads are spread over the
// 2 E values it needs (its own row for the dw output and, next to it in a slab, the next segment's for dp) and over the
// slabs, with eight loads in flight each; a chain of one load per slab and warp took most of the 16 us this kernel had
// (8 segments, 8 experts, 444 slabs: now 6).
static const int kRouterBwdThreads = 512;
template <typename T>
__global__ void __launch_bounds__(kRouterBwdThreads)
router_bwd_kernel(const float* __restrict__ partial, int n_slabs, const float* __restrict__ p, const T* __restrict__ w_r,
                  float* __restrict__ dw, float* __restrict__ d_route_w, float* __restrict__ dz,
                  float* __restrict__ dh_bar, int S, int N, int d, int E, int prefix) {
  constexpr int NT = kRouterBwdThreads, VEC = Vec16<T>::N;
  __shared__ __align__(16) float red[3 * 128 * VEC > NT ? 3 * 128 * VEC : NT];
  extern __shared__ float sm[];  // rows[2 E], dz[E]
  float* dw_sm = sm;
  float* dp_sm = sm + E;
  float* dz_sm = sm + 2 * E;
  const int s = blockIdx.x, n = s % N, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const size_t SE = (size_t)S * E;
  pdl_launch();
  pdl_wait();
  // out[c] (+)= sum over the slabs and over `rows` consecutive segments of the values of segment `row` on, c < width
  auto reduce = [&](float* out, size_t row, int width, int rows, bool add) {
    int span = 32;
    while (span < width && span < NT) span <<= 1;
    const int groups = NT / span, g = tid / span, total = n_slabs * rows;
    for (int c0 = 0; c0 < width; c0 += span) {
      const int c = c0 + (tid & (span - 1));
      float acc = 0.f;
      if (c < width) {
        const float* src = partial + row * E + c;
        int q = g;
        for (; q + 7 * groups < total; q += 8 * groups) {
          float v[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int k = q + i * groups, m = rows == 1 ? 0 : k / n_slabs;
            v[i] = src[(size_t)(k - m * n_slabs) * SE + (size_t)m * E];
          }
          acc += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
        }
#pragma unroll 4
        for (; q < total; q += groups) {
          const int m = rows == 1 ? 0 : q / n_slabs;
          acc += src[(size_t)(q - m * n_slabs) * SE + (size_t)m * E];
        }
      }
      red[tid] = acc;
      __syncthreads();
      if (tid < span && c < width) {
        float v = 0.f;
        for (int k = 0; k < groups; ++k) v += red[k * span + tid];
        out[c] = add ? out[c] + v : v;
      }
      __syncthreads();
    }
  };
  const bool prefix_mode = (prefix & 1) != 0, first_grad = (prefix & 2) != 0;
  // gradient reaching p_s: from the next segment's weights, or (prefix routing) from segments 1..N-1 if s is the
  // first segment of its sequence; the first segment's own use of p_s carries no gradient (stop-gradient)
  const bool next = !prefix_mode && n < N - 1;
  reduce(dw_sm, (size_t)s, next ? 2 * E : E, 1, false);
  if (!next) {
    for (int e = tid; e < E; e += NT) dp_sm[e] = 0.f;
    __syncthreads();
    if (prefix_mode && n == 0 && N > 1) reduce(dp_sm, (size_t)s + 1, E, N - 1, true);
  }
  for (int e = tid; e < E; e += NT) {
    const float v = dw_sm[e];
    dw[(size_t)s * E + e] = v;
    if (d_route_w) d_route_w[(size_t)s * E + e] = v;
    if (first_grad && n == 0) dp_sm[e] += v;   // no stop-gradient: the first segment's own weights also feed p_s
  }
  __syncthreads();
  if (warp == 0) {
    float dot = 0.f;
    for (int e = lane; e < E; e += 32) dot += dp_sm[e] * p[(size_t)s * E + e];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    for (int e = lane; e < E; e += 32) {
      float v = p[(size_t)s * E + e] * (dp_sm[e] - dot);
      dz_sm[e] = v;
      dz[(size_t)s * E + e] = v;
    }
  }
  __syncthreads();
  // dh_bar_s = W_r^T dz_s.  A thread takes VEC consecutive columns (one 16-byte load per expert row) and a quarter of the
  // experts; the quarters meet in shared memory.  All loads of a thread are independent.
  if (d % VEC == 0) {
    const int nvec = d / VEC, quarter = tid >> 7, vt = tid & 127;
    const int eq = (E + 3) / 4, e_begin = quarter * eq, e_end = min(E, e_begin + eq);
    for (int v0 = 0; v0 < nvec; v0 += 128) {
      const int v = v0 + vt;
      float acc[VEC];
#pragma unroll
      for (int i = 0; i < VEC; ++i) acc[i] = 0.f;
      if (v < nvec) {
#pragma unroll 8
        for (int e = e_begin; e < e_end; ++e) {
          float wv[VEC];
          Vec16<T>::load(w_r + (size_t)e * d + (size_t)v * VEC, wv);
          const float z = dz_sm[e];
#pragma unroll
          for (int i = 0; i < VEC; ++i) acc[i] += z * wv[i];
        }
      }
      if (quarter > 0) {
#pragma unroll
        for (int i = 0; i < VEC; ++i) red[((quarter - 1) * VEC + i) * 128 + vt] = acc[i];
      }
      __syncthreads();
      if (quarter == 0 && v < nvec) {
#pragma unroll
        for (int i = 0; i < VEC; ++i) acc[i] += red[i * 128 + vt] + red[(VEC + i) * 128 + vt] + red[(2 * VEC + i) * 128 + vt];
#pragma unroll
        for (int i = 0; i < VEC; i += 4)
          *reinterpret_cast<float4*>(dh_bar + (size_t)s * d + (size_t)v * VEC + i) = make_float4(acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
      }
      __syncthreads();
    }
  } else {
    for (int j = tid; j < d; j += NT) {
      float a0 = 0.f;
      for (int e = 0; e < E; ++e) a0 += dz_sm[e] * to_f32(w_r[(size_t)e * d + j]);
      dh_bar[(size_t)s * d + j] = a0;
    }
  }
}

// dW_r[e, j] = sum_s dz[s,e] h_bar[s,j].  grid (ceil(d/64), ceil(E/4)), block 512 = 64 columns x 8 runs of
// segments: a thread sums its run for one column and four experts (each h_bar element it loads serves the four),
// then the eight runs are added in a fixed order through shared memory.
template <typename T>
__global__ void __launch_bounds__(512) dwr_kernel(const float* __restrict__ dz, const float* __restrict__ h_bar,
                                                  T* __restrict__ dw_r, int S, int d, int E, int accumulate) {
  __shared__ float red[8][4][64];
  const int jj = threadIdx.x & 63, part = threadIdx.x >> 6;
  const int j = blockIdx.x * 64 + jj, e0 = blockIdx.y * 4;
  const int run = (S + 7) / 8;
  const int s_begin = part * run, s_end = min(S, s_begin + run);
  pdl_launch();
  pdl_wait();
  float a[4] = {0.f, 0.f, 0.f, 0.f};
  if (j < d) {
#pragma unroll 4
    for (int s = s_begin; s < s_end; ++s) {
      const float h = h_bar[(size_t)s * d + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (e0 + i < E) a[i] += dz[(size_t)s * E + e0 + i] * h;
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) red[part][i][jj] = a[i];
  __syncthreads();
  if (threadIdx.x < 256) {
    const int i = threadIdx.x >> 6, e = e0 + i;
    if (j < d && e < E) {
      float out = 0.f;
#pragma unroll
      for (int q = 0; q < 8; ++q) out += red[q][i][jj];
      if (accumulate) out += to_f32(dw_r[(size_t)e * d + j]);
      dw_r[(size_t)e * d + j] = from_f32<T>(out);
    }
  }
}

// ---------------------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------------------
template <typename T>
int launch_pool_router(const T* x, const T* w_r, float* h_bar, float* p_ws, float* route_p, float* w_out,
                       int B, int N, int Tseg, int d, int E, int prefix, cudaStream_t st, RouteExtra extra) {
  const int S = B * N;
  constexpr int VEC = Vec16<T>::N;
  const long blocks = S * ceil_div(d, 32 * VEC);
  // a cluster per segment until there are two blocks per SM, as long as each block has 32 rows
  int parts = 1;
  while (parts < 8 && blocks * parts < 296 && Tseg >= 64 * parts) parts *= 2;
  LORY_TRY(launch_overlapped(pool_kernel<T>, dim3((unsigned)(S * parts), (unsigned)ceil_div(d, 32 * VEC)), 256, 0, st, parts, x,
                             h_bar, Tseg, d, parts, extra.status));
  const int router_threads = E >= 32 ? 1024 : (E > 8 ? 32 * E : 256);  // one warp per expert, 8 to 32 warps
  return launch_overlapped(router_kernel<T>, dim3((unsigned)S), router_threads, E * sizeof(float), st, 1, h_bar, w_r, p_ws,
                           route_p, w_out, N, d, E, prefix, extra);
}

template <typename T>
int launch_router_backward(const float* dw_partial, int n_slabs, const float* p_ws, const float* h_bar,
                           const T* w_r, float* dw, float* d_route_w, float* dz, float* dh_bar, T* dw_r,
                           int B, int N, int d, int E, int prefix, cudaStream_t st) {
  const int S = B * N;
  const size_t smem = 3 * (size_t)E * sizeof(float);   // up to 48 KB beside the static 12 KB
  if (smem > 32 * 1024) LORY_CUDA_OK(cudaFuncSetAttribute(router_bwd_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 48 * 1024));
  LORY_TRY(launch_overlapped(router_bwd_kernel<T>, dim3((unsigned)S), kRouterBwdThreads, smem, st, 1, dw_partial, n_slabs, p_ws,
                             w_r, dw, d_route_w, dz, dh_bar, S, N, d, E, prefix));
  return launch_overlapped(dwr_kernel<T>, dim3((unsigned)ceil_div(d, 64), (unsigned)ceil_div(E, 4)), 512, 0, st, 1, dz, h_bar,
                           dw_r, S, d, E, (prefix & 4) ? 1 : 0);
}

// one thread per expert; the S weights of an expert are E floats apart
__global__ void expert_utilization_kernel(const float* __restrict__ route_w, int S, int E, int* __restrict__ counts) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  const float thr = 2.0f / (float)E;
  int n = 0;
  for (int s = 0; s < S; ++s) n += route_w[(size_t)s * E + e] > thr ? 1 : 0;
  counts[e] = n;
}

int launch_expert_utilization(const float* route_w, int S, int E, int* counts, cudaStream_t st) {
  expert_utilization_kernel<<<(unsigned)ceil_div(E, 128), 128, 0, st>>>(route_w, S, E, counts);
  LORY_AFTER_LAUNCH();
  return LORY_OK;
}

#define INST(T)                                                                                              \
  template int launch_pool_router<T>(const T*, const T*, float*, float*, float*, float*, int, int, int, int, \
                                     int, int, cudaStream_t, RouteExtra);                                    \
  template int launch_router_backward<T>(const float*, int, const float*, const float*, const T*, float*,    \
                                         float*, float*, float*, T*, int, int, int, int, int, cudaStream_t);
INST(float)
INST(bf16)
#undef INST

}  // namespace lory
