#include "simt.cuh"

#include <type_traits>

namespace lory {

template <typename TA, typename TB, typename TC>
__global__ void __launch_bounds__(256) simt_gemm_kernel(SimtGemm p) {
  constexpr int BM = 64, BN = 64, BK = 16;
  __shared__ float As[BK][BM + 4];
  __shared__ float Bs[BK][BN + 4];
  const int g = blockIdx.z;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const TA* A = reinterpret_cast<const TA*>(p.A);
  const TB* B = reinterpret_cast<const TB*>(p.B);
  TC* C = reinterpret_cast<TC*>(p.C) + (size_t)g * p.c_g;
  int k_begin = 0, k_end = p.K;
  if (p.k_chunk > 0) {
    k_begin = g * p.k_chunk;
    k_end = min(p.K, k_begin + p.k_chunk);
  } else {
    A += (size_t)g * p.a_g;
    B += (size_t)g * p.b_g;
  }
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  const bool a_kfast = (p.a_k == 1);
  const bool b_nfast = (p.b_n == 1);
  for (int k0 = k_begin; k0 < k_end; k0 += BK) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int idx = tid + i * 256;
      int kk, mm;
      if (a_kfast) { kk = idx & 15; mm = idx >> 4; } else { mm = idx & 63; kk = idx >> 6; }
      int gm = m0 + mm, gk = k0 + kk;
      As[kk][mm] = (gm < p.M && gk < k_end) ? to_f32(A[(size_t)gm * p.a_m + (size_t)gk * p.a_k]) : 0.f;
      int nn;
      if (b_nfast) { nn = idx & 63; kk = idx >> 6; } else { kk = idx & 15; nn = idx >> 4; }
      int gn = n0 + nn;
      gk = k0 + kk;
      Bs[kk][nn] = (gn < p.N && gk < k_end) ? to_f32(B[(size_t)gk * p.b_k + (size_t)gn * p.b_n]) : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int gm = m0 + ty * 4 + i;
    if (gm >= p.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int gn = n0 + tx * 4 + j;
      if (gn >= p.N) continue;
      TC* c = C + (size_t)gm * p.c_m + (size_t)gn * p.c_n;
      float v = acc[i][j];
      if (p.accumulate) v += to_f32(*c);
      *c = from_f32<TC>(v);
    }
  }
}

template <typename TA, typename TB, typename TC>
int launch_simt_gemm(const SimtGemm& g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.groups <= 0) return LORY_OK;
  dim3 grid((unsigned)ceil_div(g.N, 64), (unsigned)ceil_div(g.M, 64), (unsigned)g.groups);
  if (grid.y > 65535u || grid.z > 65535u) return LORY_ERR_SHAPE;
  simt_gemm_kernel<TA, TB, TC><<<grid, 256, 0, st>>>(g);
  LORY_AFTER_LAUNCH();
  return LORY_OK;
}

// ---------------------------------------------------------------------------------------
// FFN contractions
// ---------------------------------------------------------------------------------------
static int sm_count_simt() {
  static int n[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!n[dev] && (cudaDeviceGetAttribute(&n[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n[dev] <= 0)) n[dev] = 148;
  return n[dev];
}

// Fills in the tile counts of every job for tiles of bm x (columns of the outputs) tn; the number of tiles, or < 0.
static long fma_tiles(FmaArgs& a, int groups, int bm, int tn) {
  long acc = 0;
  for (int i = 0; i < a.jobs; ++i) {
    FmaJob& j = a.job[i];
    j.m_tiles = (int)ceil_div(j.M, bm);
    j.n_tiles = (int)ceil_div(j.N, tn);
    acc += (long)j.m_tiles * j.n_tiles * groups;
    if (acc > 0x7fffffffL) return -1;
    j.tile_end = (int)acc;
  }
  return acc;
}
// Whether inputs (returned) and outputs (FmaJob::vec) allow 4-element vectors.
template <typename T, bool A_K, bool B_K>
static bool fma_vectors(FmaArgs& a) {
  bool vec = true;
  for (int i = 0; i < a.jobs; ++i) {
    FmaJob& j = a.job[i];
    const uintptr_t out = (uintptr_t)j.C0 | (uintptr_t)j.C1 | (uintptr_t)j.C2 | (uintptr_t)j.E0 | (uintptr_t)j.E1;
    j.vec = j.ldc % 4 == 0 && j.c_g % 4 == 0 && out % (4 * sizeof(T)) == 0;
    const uintptr_t in = (uintptr_t)j.A0 | (uintptr_t)j.A1 | (uintptr_t)j.B0 | (uintptr_t)j.B1;
    vec = vec && j.lda % 4 == 0 && j.ldb % 4 == 0 && j.a_g % 4 == 0 && j.b_g % 4 == 0 && in % (4 * sizeof(T)) == 0 &&
          (A_K ? j.K : j.M) % 4 == 0 && (B_K ? j.K : j.N) % 4 == 0;
  }
  return vec;
}
template <bool A_K, bool B_K, int MODE, int EPI, bool VEC>
static int launch_fma32(const FmaArgs& a, long tiles, cudaStream_t st) {
  auto kern = fma32_kernel<A_K, B_K, MODE, EPI, VEC>;
  static bool done[64];   // the attribute belongs to the (kernel, device) pair
  int dev = 0;
  LORY_CUDA_OK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !done[dev]) {
    LORY_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Fma32::SMEM));
    if (dev >= 0 && dev < 64) done[dev] = true;
  }
  return launch_kernel(false, kern, dim3((unsigned)tiles), 32 * Fma32::KG, Fma32::SMEM, st, 1, a);
}

// Tile choice.  128-row tiles have the best ratio of FMAs to shared-memory reads and need enough of them; below two per
// SM 64-row tiles, below one per SM 32-row tiles (d = 256, f = 688, 8 segments of 128: dx 91, 62 and 54 us).  Two k-groups
// per CTA where an SM gets fewer than three CTAs, and always with 32 rows, where a thread has too few FMAs between its
// shared-memory reads to hide them (16-token segments, d = 301: 168 -> 136 us).  fp32 with less than half a 64-row tile per
// SM: the kernel that shares a 32-row tile's contraction between eight warps.
template <typename T, bool A_K, bool B_K, int MODE, int EPI>
static int fma_launch(FmaArgs a, int groups, cudaStream_t st) {
  constexpr int TILE_N = MODE == FMA_DUALB ? 32 : 64;
  const int sms = sm_count_simt();
  int mmax = 0;
  const bool vec = fma_vectors<T, A_K, B_K>(a);
  bool wide = false;   // rows too long for 32-bit offsets inside a tile: one general shape
  for (int i = 0; i < a.jobs; ++i) {
    mmax = a.job[i].M > mmax ? a.job[i].M : mmax;
    wide = wide || (!vec && (fma_wide(a.job[i].lda) || fma_wide(a.job[i].ldb)));
  }
  const long c128 = fma_tiles(a, groups, 128, TILE_N), c64 = fma_tiles(a, groups, 64, TILE_N);
  const int bm = wide ? 32 : (mmax > 64 && c128 >= 2L * sms) ? 128 : ((mmax > 32 && c64 >= sms) ? 64 : 32);
  const long tiles = fma_tiles(a, groups, bm, TILE_N);
  if (tiles < 0) return LORY_ERR_SHAPE;
  if (tiles == 0) return LORY_OK;
  const dim3 grid((unsigned)tiles);
  auto pick = [&](auto v) -> int {
    constexpr bool V = decltype(v)::value;
    if constexpr (sizeof(T) == 4) {
      if (bm == 32 && c64 * 2 < sms) return launch_fma32<A_K, B_K, MODE, EPI, V>(a, tiles, st);
    }
    if constexpr (!V) {
      if (wide) return launch_kernel(false, fma_gemm_kernel<T, A_K, B_K, MODE, EPI, 32, 2, V, true>, grid, 256, 0, st, 1, a);
    }
    const bool two = bm == 32 || tiles < 3L * sms;
    if (bm == 128) return launch_kernel(false, fma_gemm_kernel<T, A_K, B_K, MODE, EPI, 128, 1, V>, grid, 128, 0, st, 1, a);
    if (bm == 64 && two) return launch_kernel(false, fma_gemm_kernel<T, A_K, B_K, MODE, EPI, 64, 2, V>, grid, 256, 0, st, 1, a);
    if (bm == 64) return launch_kernel(false, fma_gemm_kernel<T, A_K, B_K, MODE, EPI, 64, 1, V>, grid, 128, 0, st, 1, a);
    return launch_kernel(false, fma_gemm_kernel<T, A_K, B_K, MODE, EPI, 32, 2, V>, grid, 256, 0, st, 1, a);
  };
  return vec ? pick(std::true_type()) : pick(std::false_type());
}
static FmaArgs one_job(const FmaJob& j) {
  FmaArgs a = {};
  a.job[0] = j;
  a.jobs = 1;
  return a;
}
template <typename T>
int fma_gemm_swiglu(FmaJob j, int groups, cudaStream_t st) { return fma_launch<T, true, true, FMA_DUALB, FMA_SWIGLU>(one_job(j), groups, st); }
template <typename T>
int fma_gemm_nt(FmaJob j, int groups, cudaStream_t st) { return fma_launch<T, true, true, FMA_PLAIN, FMA_STORE>(one_job(j), groups, st); }
template <typename T>
int fma_gemm_dswiglu(FmaJob j, int groups, cudaStream_t st) { return fma_launch<T, true, false, FMA_PLAIN, FMA_DSWIGLU>(one_job(j), groups, st); }
template <typename T>
int fma_gemm_tn(const FmaJob (&j)[3], int groups, cudaStream_t st) {
  FmaArgs a = {};
  for (int i = 0; i < 3; ++i) a.job[i] = j[i];
  a.jobs = 3;
  return fma_launch<T, false, false, FMA_PLAIN, FMA_STORE>(a, groups, st);
}
template <typename T>
int fma_gemm_dx(FmaJob j, int groups, const float* rowvec, float scale, cudaStream_t st) {
  FmaArgs a = one_job(j);
  a.rowvec = rowvec;
  a.row_scale = scale;
  return fma_launch<T, true, false, FMA_DUALK, FMA_ROWADD>(a, groups, st);
}

// ---------------------------------------------------------------------------------------
// Merge: Wbar_k[s, p] = sum_e w[s, e] W_k[e, p].  HBM-bound: 4 (E + S) bytes per parameter.  A thread owns four consecutive
// parameters and walks the segments 16 at a time; the experts' values come from L1 after the first walk.  grid.y = matrix.
// ---------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(128) fma_merge_kernel(const __grid_constant__ FmaMerge<T> p) {
  constexpr int SC = 16;
  __shared__ __align__(16) float s_w[32][SC];  // [expert][segment of the chunk]
  const int k = blockIdx.y;
  pdl_launch();
  pdl_wait();
  const long i0 = ((long)blockIdx.x * 128 + threadIdx.x) * 4;
  const int left = i0 < p.n ? (int)min(4L, p.n - i0) : 0;
  const bool vec = (p.n & 3) == 0 && (((uintptr_t)p.w[k] | (uintptr_t)p.wbar[k]) & (4 * sizeof(T) - 1)) == 0;
  for (int s0 = 0; s0 < p.S; s0 += SC) {
    if (s0 > 0) __syncthreads();
    for (int i = threadIdx.x; i < p.E * SC; i += 128) {
      const int e = i / SC, s = s0 + i % SC;
      s_w[e][i % SC] = s < p.S ? p.route[(size_t)s * p.E + e] : 0.f;
    }
    __syncthreads();
    float acc[SC][4];
#pragma unroll
    for (int s = 0; s < SC; ++s) acc[s][0] = acc[s][1] = acc[s][2] = acc[s][3] = 0.f;
    for (int e = 0; e < p.E; ++e) {
      float v[4];
      load4(p.w[k] + (size_t)e * p.n + i0, left, vec, v);
#pragma unroll
      for (int s4 = 0; s4 < SC; s4 += 4) {
        const float4 w = *reinterpret_cast<const float4*>(&s_w[e][s4]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[s4][i] = fmaf(w.x, v[i], acc[s4][i]);
          acc[s4 + 1][i] = fmaf(w.y, v[i], acc[s4 + 1][i]);
          acc[s4 + 2][i] = fmaf(w.z, v[i], acc[s4 + 2][i]);
          acc[s4 + 3][i] = fmaf(w.w, v[i], acc[s4 + 3][i]);
        }
      }
    }
#pragma unroll
    for (int s = 0; s < SC; ++s)
      if (s0 + s < p.S) store4(p.wbar[k] + (size_t)(s0 + s) * p.n + i0, left, vec, acc[s]);
  }
}

// ---------------------------------------------------------------------------------------
// Adjoint of the merge, one pass over dWbar: dW_k[e, p] = sum_s w[s, e] dWbar_k[s, p] and dw[s, e] += sum_p dWbar_k[s, p]
// W_k[e, p].  HBM-bound: 4 (S + 2 E) bytes per parameter.  A CTA takes tiles of 256 parameters in turn, 32 segments at a
// time: a thread owns one parameter for the first product (its dWbar value is in a register); the second runs on the tiles
// in shared memory, 4 segments x EMAX / 8 experts per thread with the parameters split over four neighbouring lanes.  Rows
// of 260 floats keep the 16-byte reads of four-apart rows on different banks.  The CTA's dw sums stay in shared memory.
// ---------------------------------------------------------------------------------------
static const int kFmaTile = 256, kFmaRow = 260, kFmaSegs = 32;
static size_t fma_adjoint_smem(int S, int E, int emax) {
  return ((size_t)(kFmaSegs + emax) * kFmaRow + (size_t)kFmaSegs * emax + (size_t)S * E) * sizeof(float);
}

template <typename T, int EMAX>
__global__ void __launch_bounds__(256) fma_adjoint_kernel(const __grid_constant__ FmaMerge<T> p) {
  constexpr int EB = EMAX / 8;
  extern __shared__ __align__(16) float s_dyn[];
  float* s_d = s_dyn;                          // [32 segments][260]
  float* s_e = s_d + kFmaSegs * kFmaRow;       // [EMAX][260]
  float* s_w = s_e + EMAX * kFmaRow;           // [32][EMAX] routing weights of the chunk
  float* s_dw = s_w + kFmaSegs * EMAX;         // [S][E]
  const int tid = threadIdx.x, ks = tid & 3, sg = (tid >> 2) & 7, eg = tid >> 5;
  for (int i = tid; i < p.S * p.E; i += 256) s_dw[i] = 0.f;
  pdl_launch();
  pdl_wait();
  const int per = (int)((p.n + kFmaTile - 1) / kFmaTile), chunks = (p.S + kFmaSegs - 1) / kFmaSegs;
  // One step = one chunk of segments of one tile.  The next step's values are on their way in registers (ve, vd) while
  // this one is worked on: 198 -> 128 us at S = 18, E = 6, n = 670 000.
  float ve[EMAX], vd[kFmaSegs];
  auto fetch = [&](int tile, int chunk) {
    const int k = tile / per;
    const long i0 = (long)(tile - k * per) * kFmaTile + tid;
    const bool in = i0 < p.n;
    if (chunk == 0) {
#pragma unroll
      for (int e = 0; e < EMAX; ++e) ve[e] = (in && e < p.E) ? to_f32(p.w[k][(size_t)e * p.n + i0]) : 0.f;
    }
    const T* d = p.wbar[k] + (size_t)chunk * kFmaSegs * p.n + i0;
    const int ns = in ? p.S - chunk * kFmaSegs : 0;
#pragma unroll
    for (int s = 0; s < kFmaSegs; ++s) vd[s] = s < ns ? to_f32(d[(size_t)s * p.n]) : 0.f;
  };
  float acc[EMAX];
  int tile = blockIdx.x, chunk = 0;
  if (tile < 3 * per) fetch(tile, 0);
  while (tile < 3 * per) {
    const int s0 = chunk * kFmaSegs, ns = min(kFmaSegs, p.S - s0), k = tile / per;
    const long i0 = (long)(tile - k * per) * kFmaTile + tid;
    const bool last = chunk + 1 == chunks;
    __syncthreads();   // the tiles in shared memory have been read
    if (chunk == 0) {
#pragma unroll
      for (int e = 0; e < EMAX; ++e) {
        s_e[e * kFmaRow + tid] = ve[e];
        acc[e] = 0.f;
      }
    }
#pragma unroll
    for (int s = 0; s < kFmaSegs; ++s) s_d[s * kFmaRow + tid] = vd[s];
    for (int i = tid; i < kFmaSegs * EMAX; i += 256) {
      const int s = i / EMAX, e = i % EMAX;
      s_w[i] = (s < ns && e < p.E) ? p.route[(size_t)(s0 + s) * p.E + e] : 0.f;
    }
    __syncthreads();
    const int next_chunk = last ? 0 : chunk + 1, next_tile = last ? tile + (int)gridDim.x : tile;
    if (next_tile < 3 * per) fetch(next_tile, next_chunk);
    for (int s = 0; s < ns; ++s) {
      const float d = s_d[s * kFmaRow + tid];
#pragma unroll
      for (int e = 0; e < EMAX; e += 4) {
        const float4 w = *reinterpret_cast<const float4*>(&s_w[s * EMAX + e]);
        acc[e] = fmaf(w.x, d, acc[e]);
        acc[e + 1] = fmaf(w.y, d, acc[e + 1]);
        acc[e + 2] = fmaf(w.z, d, acc[e + 2]);
        acc[e + 3] = fmaf(w.w, d, acc[e + 3]);
      }
    }
    if (last && i0 < p.n) {
#pragma unroll
      for (int e = 0; e < EMAX; ++e)
        if (e < p.E) {
          T* q = p.dw[k] + (size_t)e * p.n + i0;
          *q = from_f32<T>(p.accumulate ? acc[e] + to_f32(*q) : acc[e]);
        }
    }
    const unsigned mask = __ballot_sync(0xffffffffu, sg * 4 < ns);   // the lanes that go in (eg is the warp's)
    if (sg * 4 < ns && eg * EB < p.E) {
      float dot[4][EB];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int e = 0; e < EB; ++e) dot[i][e] = 0.f;
#pragma unroll 2
      for (int j = 0; j < kFmaTile / 16; ++j) {
        float4 d4[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) d4[i] = *reinterpret_cast<const float4*>(&s_d[(sg * 4 + i) * kFmaRow + (j * 4 + ks) * 4]);
#pragma unroll
        for (int e = 0; e < EB; ++e) {
          const float4 w4 = *reinterpret_cast<const float4*>(&s_e[(eg * EB + e) * kFmaRow + (j * 4 + ks) * 4]);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            dot[i][e] = fmaf(d4[i].x, w4.x, fmaf(d4[i].y, w4.y, fmaf(d4[i].z, w4.z, fmaf(d4[i].w, w4.w, dot[i][e]))));
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int e = 0; e < EB; ++e) {
          float x = dot[i][e];
          x += __shfl_xor_sync(mask, x, 1);
          x += __shfl_xor_sync(mask, x, 2);
          const int s = s0 + sg * 4 + i, ee = eg * EB + e;
          if (ks == 0 && s < p.S && ee < p.E) s_dw[s * p.E + ee] += x;
        }
    }
    tile = next_tile;
    chunk = next_chunk;
  }
  __syncthreads();
  float* slab = p.slabs + (size_t)blockIdx.x * p.S * p.E;
  for (int i = tid; i < p.S * p.E; i += 256) slab[i] = s_dw[i];
}

bool fma_merge_supported(int S, int E) {
  return E <= 32 && fma_adjoint_smem(S, E, E <= 8 ? 8 : (E <= 16 ? 16 : 32)) <= 160 * 1024;
}
int fma_adjoint_slabs(long n) {
  const long tiles = 3 * ceil_div(n, kFmaTile), cap = 2L * sm_count_simt();
  return (int)(tiles < cap ? tiles : cap);
}
template <typename T>
int launch_fma_merge(const FmaMerge<T>& p, cudaStream_t st) {
  return launch_kernel(false, fma_merge_kernel<T>, dim3((unsigned)ceil_div(p.n, 512), 3), 128, 0, st, 1, p);
}
template <typename T, int EMAX>
static int launch_fma_adjoint_t(const FmaMerge<T>& p, cudaStream_t st) {
  const size_t smem = fma_adjoint_smem(p.S, p.E, EMAX);
  LORY_CUDA_OK(cudaFuncSetAttribute(fma_adjoint_kernel<T, EMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024));
  return launch_kernel(false, fma_adjoint_kernel<T, EMAX>, dim3((unsigned)fma_adjoint_slabs(p.n)), 256, smem, st, 1, p);
}
template <typename T>
int launch_fma_adjoint(const FmaMerge<T>& p, cudaStream_t st) {
  if (p.E <= 8) return launch_fma_adjoint_t<T, 8>(p, st);
  if (p.E <= 16) return launch_fma_adjoint_t<T, 16>(p, st);
  return launch_fma_adjoint_t<T, 32>(p, st);
}

template int launch_simt_gemm<float, float, float>(const SimtGemm&, cudaStream_t);
template int launch_simt_gemm<float, bf16, bf16>(const SimtGemm&, cudaStream_t);
template int launch_simt_gemm<bf16, bf16, float>(const SimtGemm&, cudaStream_t);
#define INST(T)                                                                              \
  template int fma_gemm_swiglu<T>(FmaJob, int, cudaStream_t);                                \
  template int fma_gemm_nt<T>(FmaJob, int, cudaStream_t);                                    \
  template int fma_gemm_dswiglu<T>(FmaJob, int, cudaStream_t);                               \
  template int fma_gemm_tn<T>(const FmaJob (&)[3], int, cudaStream_t);                       \
  template int fma_gemm_dx<T>(FmaJob, int, const float*, float, cudaStream_t);               \
  template int launch_fma_merge<T>(const FmaMerge<T>&, cudaStream_t);                        \
  template int launch_fma_adjoint<T>(const FmaMerge<T>&, cudaStream_t);
INST(float)
INST(bf16)
#undef INST

}  // namespace lory
