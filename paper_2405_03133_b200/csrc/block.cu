// The layer inside a pre-norm residual block (the LLaMA block of Section 4.1):  y = x + Lory(RMSNorm(x)).
// RMSNorm(x) = x / sqrt(mean_j x_j^2 + eps) * gamma per token; all arithmetic in fp32.
// The forward residual is added in the epilogue of the last GEMM of the layer; the backward residual rides in the RMSNorm backward kernel.
#include "block.cuh"

namespace lory {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 16-byte vectors of the storage type as floats
template <typename T>
struct V16;
template <>
struct V16<float> {
  static constexpr int N = 4;
  __device__ static void load(const float* p, float (&v)[4]) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  }
  __device__ static void store(float* p, const float (&v)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};
template <>
struct V16<bf16> {
  static constexpr int N = 8;
  __device__ static void load(const bf16* p, float (&v)[8]) {
    const uint4 q = *reinterpret_cast<const uint4*>(p);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&q);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = __bfloat1622float2(h[i]);
      v[2 * i] = f.x; v[2 * i + 1] = f.y;
    }
  }
  __device__ static void store(bf16* p, const float (&v)[8]) {
    uint4 q;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&q);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    *reinterpret_cast<uint4*>(p) = q;
  }
};

// One warp per token row, grid-stride over rows; HBM-bound (x in, x_hat out).  x_hat = x * inv * gamma (storage type),
// inv [tokens] float.  KV > 0: the row (at most 32 * KV 16-byte vectors, a whole number of them) stays in registers
// between the two uses, and its loads are in flight together; KV = 0: any row, read twice.
template <typename T, int KV>
__global__ void __launch_bounds__(256) rmsnorm_kernel(const T* __restrict__ x, const T* __restrict__ gamma,
                                                      T* __restrict__ x_hat, float* __restrict__ inv_rms, long tokens,
                                                      int d, float eps) {
  constexpr int VEC = V16<T>::N;
  const int lane = threadIdx.x & 31;
  const long warp0 = (long)blockIdx.x * 8 + (threadIdx.x >> 5), nwarps = (long)gridDim.x * 8;
  pdl_launch();
  pdl_wait();
  for (long t = warp0; t < tokens; t += nwarps) {
    const T* row = x + t * d;
    T* out = x_hat + t * d;
    float ss = 0.f;
    if (KV > 0) {
      float v[KV > 0 ? KV : 1][VEC];
#pragma unroll
      for (int k = 0; k < KV; ++k) {
        const int j = (k * 32 + lane) * VEC;
#pragma unroll
        for (int i = 0; i < VEC; ++i) v[k][i] = 0.f;
        if (j < d) V16<T>::load(row + j, v[k]);
      }
#pragma unroll
      for (int k = 0; k < KV; ++k)
#pragma unroll
        for (int i = 0; i < VEC; ++i) ss += v[k][i] * v[k][i];
      const float inv = rsqrtf(warp_sum(ss) / (float)d + eps);
      if (lane == 0) inv_rms[t] = inv;
#pragma unroll
      for (int k = 0; k < KV; ++k) {
        const int j = (k * 32 + lane) * VEC;
        if (j < d) {
          float g[VEC];
          V16<T>::load(gamma + j, g);
#pragma unroll
          for (int i = 0; i < VEC; ++i) v[k][i] = v[k][i] * inv * g[i];
          V16<T>::store(out + j, v[k]);
        }
      }
    } else {
      const bool vec = d % VEC == 0;
      if (vec) {
#pragma unroll 4
        for (int j = lane * VEC; j < d; j += 32 * VEC) {
          float v[VEC];
          V16<T>::load(row + j, v);
#pragma unroll
          for (int i = 0; i < VEC; ++i) ss += v[i] * v[i];
        }
      } else {
        for (int j = lane; j < d; j += 32) {
          const float v = to_f32(row[j]);
          ss += v * v;
        }
      }
      const float inv = rsqrtf(warp_sum(ss) / (float)d + eps);
      if (lane == 0) inv_rms[t] = inv;
      if (vec) {
        for (int j = lane * VEC; j < d; j += 32 * VEC) {
          float v[VEC], g[VEC];
          V16<T>::load(row + j, v);
          V16<T>::load(gamma + j, g);
#pragma unroll
          for (int i = 0; i < VEC; ++i) v[i] = v[i] * inv * g[i];
          V16<T>::store(out + j, v);
        }
      } else {
        for (int j = lane; j < d; j += 32) out[j] = from_f32<T>(to_f32(row[j]) * inv * to_f32(gamma[j]));
      }
    }
  }
}

// With n = x * inv, dn = dxh * gamma:  dx = inv * (dn - n * mean_j(dn_j n_j)) + dy  (the residual path),
// and this block's partial of dgamma_j = sum over tokens of dxh_j n_j  ->  slab[blockIdx.x, d].
// One warp per token row, grid-stride over rows; HBM-bound (x, dxh, dy in, dx out).  KV > 0 as above: a row is read once,
// and a lane keeps the dgamma sums of its own columns; the warps' sums are added in shared memory, in a fixed order.
// KV = 0: any row, in passes over spans of columns.
template <typename T, int KV>
__global__ void __launch_bounds__(256) rmsnorm_bwd_kernel(const T* __restrict__ x, const T* __restrict__ gamma,
                                                          const float* __restrict__ inv_rms,
                                                          const T* __restrict__ dxh, const T* __restrict__ dy,
                                                          T* __restrict__ dx, float* __restrict__ slab, long tokens,
                                                          int d) {
  constexpr int VEC = V16<T>::N, K1 = KV > 0 ? KV : 1;
  constexpr int SPAN = 32 * VEC;
  __shared__ float part[8][SPAN];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long warp0 = (long)blockIdx.x * 8 + warp, nwarps = (long)gridDim.x * 8;
  pdl_launch();
  pdl_wait();
  if (KV > 0) {
    float acc[K1][VEC];
#pragma unroll
    for (int k = 0; k < KV; ++k)
#pragma unroll
      for (int i = 0; i < VEC; ++i) acc[k][i] = 0.f;
    for (long t = warp0; t < tokens; t += nwarps) {
      const float inv = inv_rms[t];
      float xv[K1][VEC], gv[K1][VEC];
#pragma unroll
      for (int k = 0; k < KV; ++k) {
        const int j = (k * 32 + lane) * VEC;
#pragma unroll
        for (int i = 0; i < VEC; ++i) xv[k][i] = gv[k][i] = 0.f;
        if (j < d) {
          V16<T>::load(x + t * d + j, xv[k]);
          V16<T>::load(dxh + t * d + j, gv[k]);
        }
      }
      float dot = 0.f;
#pragma unroll
      for (int k = 0; k < KV; ++k) {
        const int j = (k * 32 + lane) * VEC;
        if (j < d) {
          float gm[VEC];
          V16<T>::load(gamma + j, gm);
#pragma unroll
          for (int i = 0; i < VEC; ++i) {
            xv[k][i] *= inv;                    // n
            acc[k][i] += gv[k][i] * xv[k][i];
            gv[k][i] *= gm[i];                  // dn
            dot += gv[k][i] * xv[k][i];
          }
        }
      }
      const float m = warp_sum(dot) / (float)d;
#pragma unroll
      for (int k = 0; k < KV; ++k) {
        const int j = (k * 32 + lane) * VEC;
        if (j < d) {
          float o[VEC];
          V16<T>::load(dy + t * d + j, o);
#pragma unroll
          for (int i = 0; i < VEC; ++i) o[i] += inv * (gv[k][i] - xv[k][i] * m);
          V16<T>::store(dx + t * d + j, o);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < KV; ++k) {   // columns [k * 32 * VEC, (k + 1) * 32 * VEC)
      __syncthreads();
#pragma unroll
      for (int i = 0; i < VEC; ++i) part[warp][lane * VEC + i] = acc[k][i];
      __syncthreads();
      const int c = threadIdx.x, j = k * 32 * VEC + c;
      if (c < 32 * VEC && j < d) {
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) sum += part[w][c];
        slab[(size_t)blockIdx.x * d + j] = sum;
      }
    }
    return;
  }
  const bool vec = d % VEC == 0;
  for (int j0 = 0; j0 < d; j0 += SPAN) {
    const int width = min(SPAN, d - j0);
    float acc[VEC];   // column j0 + lane * VEC + i, or (rows that are no whole vectors) j0 + i * 32 + lane
#pragma unroll
    for (int i = 0; i < VEC; ++i) acc[i] = 0.f;
    for (long t = warp0; t < tokens; t += nwarps) {
      const float inv = inv_rms[t];
      const T* xr = x + t * d;
      const T* gr = dxh + t * d;
      if (j0 == 0) {   // dx of the whole row
        float dot = 0.f;
        if (vec) {
#pragma unroll 2
          for (int j = lane * VEC; j < d; j += 32 * VEC) {
            float xv[VEC], gv[VEC], gm[VEC];
            V16<T>::load(xr + j, xv);
            V16<T>::load(gr + j, gv);
            V16<T>::load(gamma + j, gm);
#pragma unroll
            for (int i = 0; i < VEC; ++i) dot += gv[i] * gm[i] * xv[i];
          }
        } else {
          for (int j = lane; j < d; j += 32) dot += to_f32(gr[j]) * to_f32(gamma[j]) * to_f32(xr[j]);
        }
        const float m = warp_sum(dot) * inv / (float)d;
        if (vec) {
          for (int j = lane * VEC; j < d; j += 32 * VEC) {
            float xv[VEC], gv[VEC], gm[VEC], o[VEC];
            V16<T>::load(xr + j, xv);
            V16<T>::load(gr + j, gv);
            V16<T>::load(gamma + j, gm);
            V16<T>::load(dy + t * d + j, o);
#pragma unroll
            for (int i = 0; i < VEC; ++i) o[i] += inv * (gv[i] * gm[i] - xv[i] * inv * m);
            V16<T>::store(dx + t * d + j, o);
          }
        } else {
          for (int j = lane; j < d; j += 32)
            dx[t * d + j] = from_f32<T>(inv * (to_f32(gr[j]) * to_f32(gamma[j]) - to_f32(xr[j]) * inv * m) + to_f32(dy[t * d + j]));
        }
      }
      if (vec) {
        if (lane * VEC < width) {
          float xv[VEC], gv[VEC];
          V16<T>::load(xr + j0 + lane * VEC, xv);
          V16<T>::load(gr + j0 + lane * VEC, gv);
#pragma unroll
          for (int i = 0; i < VEC; ++i) acc[i] += gv[i] * xv[i] * inv;
        }
      } else {
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
          const int j = i * 32 + lane;
          if (j < width) acc[i] += to_f32(gr[j0 + j]) * to_f32(xr[j0 + j]) * inv;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < VEC; ++i) part[warp][vec ? lane * VEC + i : i * 32 + lane] = acc[i];
    __syncthreads();
    for (int j = threadIdx.x; j < width; j += 256) {
      float sum = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) sum += part[w][j];
      slab[(size_t)blockIdx.x * d + j0 + j] = sum;
    }
    __syncthreads();
  }
}

// dgamma[j] = sum over slabs (+ the old value when accumulating).  A block takes 32 columns and spreads the slabs over
// its 8 warps (one thread per column walked all 296 slabs: 20 of the 36 us of the norm's backward at d = 1000).
template <typename T>
__global__ void __launch_bounds__(256) dgamma_reduce_kernel(const float* __restrict__ slab, int n_slabs, int d,
                                                            T* __restrict__ dgamma, int accumulate) {
  __shared__ float part[8][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = blockIdx.x * 32 + lane;
  pdl_launch();
  pdl_wait();
  float a = 0.f;
  if (j < d) {
#pragma unroll 8
    for (int c = warp; c < n_slabs; c += 8) a += slab[(size_t)c * d + j];
  }
  part[warp][lane] = a;
  __syncthreads();
  if (warp == 0 && j < d) {
    float out = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) out += part[w][lane];
    if (accumulate) out += to_f32(dgamma[j]);
    dgamma[j] = from_f32<T>(out);
  }
}

int block_norm_slabs(long tokens) {
  const long want = (tokens + 7) / 8;
  return (int)(want < 296 ? want : 296);
}

template <typename T>
constexpr int kMaxVectors = 64 / V16<T>::N;   // the most vectors per lane: 64 values
// Vectors per lane of a row that fits registers, 0 for the element-wise form.
template <typename T>
static int row_vectors(int d) {
  constexpr int VEC = V16<T>::N;
  const int k = (d / VEC + 31) / 32;
  return d % VEC == 0 && k * VEC <= 64 ? (k <= 2 ? 2 : (k <= 4 ? 4 : (k <= 8 ? 8 : 16))) : 0;
}

template <typename T>
int launch_rmsnorm(const T* x, const T* gamma, T* x_hat, float* inv_rms, long tokens, int d, float eps,
                   cudaStream_t st) {
  const long want = (tokens + 7) / 8;
  const dim3 grid((unsigned)(want < 1184 ? want : 1184));
  auto go = [&](auto kern) { return launch_overlapped(kern, grid, 256, 0, st, 1, x, gamma, x_hat, inv_rms, tokens, d, eps); };
  switch (row_vectors<T>(d)) {
    case 2: return go(rmsnorm_kernel<T, 2>);
    case 4: return go(rmsnorm_kernel<T, 4>);
    case 8: return go(rmsnorm_kernel<T, 8>);
    case 16: return go(rmsnorm_kernel<T, kMaxVectors<T>>);
    default: return go(rmsnorm_kernel<T, 0>);
  }
}

template <typename T>
int launch_rmsnorm_backward(const T* x, const T* gamma, const float* inv_rms, const T* dxh, const T* dy, T* dx,
                            T* dgamma, float* slab, long tokens, int d, int accumulate, cudaStream_t st) {
  const int n_slabs = block_norm_slabs(tokens);
  auto go = [&](auto kern) {
    return launch_overlapped(kern, dim3((unsigned)n_slabs), 256, 0, st, 1, x, gamma, inv_rms, dxh, dy, dx, slab, tokens, d);
  };
  int r;
  switch (row_vectors<T>(d)) {
    case 2: r = go(rmsnorm_bwd_kernel<T, 2>); break;
    case 4: r = go(rmsnorm_bwd_kernel<T, 4>); break;
    case 8: r = go(rmsnorm_bwd_kernel<T, 8>); break;
    case 16: r = go(rmsnorm_bwd_kernel<T, kMaxVectors<T>>); break;
    default: r = go(rmsnorm_bwd_kernel<T, 0>);
  }
  LORY_TRY(r);
  return launch_overlapped(dgamma_reduce_kernel<T>, dim3((unsigned)ceil_div(d, 32)), 256, 0, st, 1, slab, n_slabs, d, dgamma,
                           accumulate);
}

#define INST(T)                                                                                                  \
  template int launch_rmsnorm<T>(const T*, const T*, T*, float*, long, int, float, cudaStream_t);                \
  template int launch_rmsnorm_backward<T>(const T*, const T*, const float*, const T*, const T*, T*, T*, float*,  \
                                          long, int, int, cudaStream_t);
INST(float)
INST(bf16)
#undef INST

}  // namespace lory
