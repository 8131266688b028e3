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

// One warp per token row, grid-stride over rows.  x_hat = x * inv * gamma (storage type), inv [tokens] float.
// Rows whose length is a multiple of the 16-byte vector go through vector loads and stores.
template <typename T>
__global__ void __launch_bounds__(256) rmsnorm_kernel(const T* __restrict__ x, const T* __restrict__ gamma,
                                                      T* __restrict__ x_hat, float* __restrict__ inv_rms, long tokens,
                                                      int d, float eps) {
  constexpr int VEC = V16<T>::N;
  const int lane = threadIdx.x & 31;
  const long warp0 = (long)blockIdx.x * 8 + (threadIdx.x >> 5), nwarps = (long)gridDim.x * 8;
  const bool vec = (d % VEC) == 0;
  for (long t = warp0; t < tokens; t += nwarps) {
    const T* row = x + t * d;
    T* out = x_hat + t * d;
    float ss = 0.f;
    if (vec) {
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
    ss = warp_sum(ss);
    const float inv = rsqrtf(ss / (float)d + eps);
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

// With n = x * inv, dn = dxh * gamma:  dx = inv * (dn - n * mean_j(dn_j n_j)) + dy  (the residual path),
// and this block's partial of dgamma_j = sum over tokens of dxh_j n_j  ->  slab[blockIdx.x, d].
// One warp per token row, grid-stride over rows; each lane keeps the dgamma partial sums of its own columns
// (up to KMAX 16-byte vectors per lane; wider rows take more passes over this warp's rows), and the eight warps'
// partials are summed through shared memory.
template <typename T>
__global__ void __launch_bounds__(256) rmsnorm_bwd_kernel(const T* __restrict__ x, const T* __restrict__ gamma,
                                                          const float* __restrict__ inv_rms,
                                                          const T* __restrict__ dxh, const T* __restrict__ dy,
                                                          T* __restrict__ dx, float* __restrict__ slab, long tokens,
                                                          int d) {
  constexpr int VEC = V16<T>::N, KMAX = 4;
  constexpr int SPAN = 32 * VEC * KMAX;  // columns one pass covers
  __shared__ float part[8][SPAN];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long warp0 = (long)blockIdx.x * 8 + warp, nwarps = (long)gridDim.x * 8;
  const bool vec = (d % VEC) == 0;
  for (int j0 = 0; j0 < d; j0 += SPAN) {
    const int width = min(SPAN, d - j0);
    float acc[KMAX][VEC];
#pragma unroll
    for (int k = 0; k < KMAX; ++k)
#pragma unroll
      for (int i = 0; i < VEC; ++i) acc[k][i] = 0.f;
    for (long t = warp0; t < tokens; t += nwarps) {
      const float inv = inv_rms[t];
      const T* xr = x + t * d;
      const T* gr = dxh + t * d;
      // the row's mean of dn * n is needed only while dx is produced (first pass over the columns)
      float m = 0.f;
      if (j0 == 0) {
        float dot = 0.f;
        if (vec) {
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
        m = warp_sum(dot) * inv / (float)d;
      }
      if (vec) {
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
          const int j = (k * 32 + lane) * VEC;
          if (j < width) {
            float xv[VEC], gv[VEC];
            V16<T>::load(xr + j0 + j, xv);
            V16<T>::load(gr + j0 + j, gv);
#pragma unroll
            for (int i = 0; i < VEC; ++i) acc[k][i] += gv[i] * xv[i] * inv;
          }
        }
        if (j0 == 0) {
          for (int j = lane * VEC; j < d; j += 32 * VEC) {
            float xv[VEC], gv[VEC], gm[VEC], yv[VEC], o[VEC];
            V16<T>::load(xr + j, xv);
            V16<T>::load(gr + j, gv);
            V16<T>::load(gamma + j, gm);
            V16<T>::load(dy + t * d + j, yv);
#pragma unroll
            for (int i = 0; i < VEC; ++i) o[i] = inv * (gv[i] * gm[i] - xv[i] * inv * m) + yv[i];
            V16<T>::store(dx + t * d + j, o);
          }
        }
      } else {
#pragma unroll
        for (int k = 0; k < KMAX * VEC; ++k) {
          const int j = k * 32 + lane;
          if (j < width) acc[k / VEC][k % VEC] += to_f32(gr[j0 + j]) * to_f32(xr[j0 + j]) * inv;
        }
        if (j0 == 0) {
          for (int j = lane; j < d; j += 32) {
            const float n = to_f32(xr[j]) * inv;
            const float dn = to_f32(gr[j]) * to_f32(gamma[j]);
            dx[t * d + j] = from_f32<T>(inv * (dn - n * m) + to_f32(dy[t * d + j]));
          }
        }
      }
    }
    // column j of this pass lives in acc[k][i]: vector layout j = (k*32 + lane)*VEC + i, scalar layout j = (k*VEC+i)*32 + lane
#pragma unroll
    for (int k = 0; k < KMAX; ++k)
#pragma unroll
      for (int i = 0; i < VEC; ++i) {
        const int j = vec ? (k * 32 + lane) * VEC + i : (k * VEC + i) * 32 + lane;
        if (j < width) part[warp][j] = acc[k][i];
      }
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

// dgamma[j] = sum over slabs (+ the old value when accumulating)
template <typename T>
__global__ void dgamma_reduce_kernel(const float* __restrict__ slab, int n_slabs, int d, T* __restrict__ dgamma,
                                     int accumulate) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= d) return;
  float a0 = 0.f, a1 = 0.f;
  int c = 0;
  for (; c + 1 < n_slabs; c += 2) {
    a0 += slab[(size_t)c * d + j];
    a1 += slab[(size_t)(c + 1) * d + j];
  }
  if (c < n_slabs) a0 += slab[(size_t)c * d + j];
  float out = a0 + a1;
  if (accumulate) out += to_f32(dgamma[j]);
  dgamma[j] = from_f32<T>(out);
}

int block_norm_slabs(long tokens) {
  const long want = (tokens + 7) / 8;
  return (int)(want < 296 ? want : 296);
}

template <typename T>
int launch_rmsnorm(const T* x, const T* gamma, T* x_hat, float* inv_rms, long tokens, int d, float eps,
                   cudaStream_t st) {
  const long want = (tokens + 7) / 8;
  const unsigned grid = (unsigned)(want < 1184 ? want : 1184);
  rmsnorm_kernel<T><<<grid, 256, 0, st>>>(x, gamma, x_hat, inv_rms, tokens, d, eps);
  LORY_AFTER_LAUNCH();
  return LORY_OK;
}

template <typename T>
int launch_rmsnorm_backward(const T* x, const T* gamma, const float* inv_rms, const T* dxh, const T* dy, T* dx,
                            T* dgamma, float* slab, long tokens, int d, int accumulate, cudaStream_t st) {
  const int n_slabs = block_norm_slabs(tokens);
  rmsnorm_bwd_kernel<T><<<n_slabs, 256, 0, st>>>(x, gamma, inv_rms, dxh, dy, dx, slab, tokens, d);
  LORY_AFTER_LAUNCH();
  dgamma_reduce_kernel<T><<<(unsigned)ceil_div(d, 256), 256, 0, st>>>(slab, n_slabs, d, dgamma, accumulate);
  LORY_AFTER_LAUNCH();
  return LORY_OK;
}

#define INST(T)                                                                                                  \
  template int launch_rmsnorm<T>(const T*, const T*, T*, float*, long, int, float, cudaStream_t);                \
  template int launch_rmsnorm_backward<T>(const T*, const T*, const float*, const T*, const T*, T*, T*, float*,  \
                                          long, int, int, cudaStream_t);
INST(float)
INST(bf16)
#undef INST

}  // namespace lory
