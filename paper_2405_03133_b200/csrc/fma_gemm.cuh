// Grouped fp32-FMA GEMM of the plain-FMA pipeline (fp32 mode, whose 1e-4 rules tensor-core products out, and bf16 with
// more than 64 experts or LORY_FLAG_SIMT).
//
//   C_g[m, n] = sum_k A_g[m, k] B_g[k, n]        fp32 accumulation, operands of type T with one contiguous dimension each
//
// FMA-bound (2 M N K flops per group at 128 FMA per SM and clock, 74 TFLOP/s).  A group of 128 threads computes BM x 64
// outputs, BM / 16 rows x 8 columns per thread, as packed pairs (fma.rn.f32x2: the same rate as two FMAs in half the issue
// slots); k-blocks of 16 pass through registers into a double-buffered shared tile, so one barrier per block is enough.
// A CTA has KG such groups that take the k-blocks in turn and add their sums at the end.  What keeps a small layer from
// the bound is not the inner loop but too few tiles: BM and KG are chosen by the host so that every SM gets work
// (fma_launch in simt.cu).
// Dual forms: MODE_DUALB multiplies the same A by 32 columns of B0 and the same 32 columns of B1 (gate and up projections,
// so that the SwiGLU is applied where both values are in one thread), MODE_DUALK runs over (A0, B0) and then (A1, B1).
#pragma once
#include "common.cuh"

namespace lory {

enum FmaMode { FMA_PLAIN = 0, FMA_DUALB = 1, FMA_DUALK = 2 };
enum FmaEpi {
  FMA_STORE = 0,    // C0 = acc (+ residual)
  FMA_SWIGLU = 1,   // DUALB: C0 = G, C1 = U, C2 = silu(G) U
  FMA_DSWIGLU = 2,  // acc = dH; C0 = dG, C1 = dU from E0 = G, E1 = U
  FMA_ROWADD = 3    // C0 = acc + rowvec[g, n] * row_scale
};

// One problem of a launch: all groups of one product.
struct FmaJob {
  const void *A0, *A1, *B0, *B1;
  void *C0, *C1, *C2;
  const void *E0, *E1;  // DSWIGLU: G, U; STORE: E0 = residual (may be NULL); all laid out like C0
  int M, N, K;
  int lda, ldb, ldc;    // elements between consecutive rows of the stored matrices
  long a_g, b_g, c_g;   // elements between groups
  int m_tiles, n_tiles;
  int tile_end;         // exclusive prefix sum of m_tiles * n_tiles * groups over the jobs
  int vec;              // C0..C2, E0, E1 allow 4-element vectors
};
struct FmaArgs {
  FmaJob job[3];
  int jobs;
  const float* rowvec;
  float row_scale;
};

template <typename T>
struct Vec4;
template <>
struct Vec4<float> {
  __device__ static void load(const float* p, float (&v)[4]) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  }
  __device__ static void store(float* p, const float (&v)[4]) { *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]); }
};
template <>
struct Vec4<bf16> {
  __device__ static void load(const bf16* p, float (&v)[4]) {
    const uint2 q = *reinterpret_cast<const uint2*>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.y));
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
  }
  __device__ static void store(bf16* p, const float (&v)[4]) {
    uint2 q;
    *reinterpret_cast<__nv_bfloat162*>(&q.x) = __floats2bfloat162_rn(v[0], v[1]);
    *reinterpret_cast<__nv_bfloat162*>(&q.y) = __floats2bfloat162_rn(v[2], v[3]);
    *reinterpret_cast<uint2*>(p) = q;
  }
};
// n <= 4 consecutive elements, as one vector where that is allowed
template <typename T>
__device__ __forceinline__ void load4(const T* p, int n, bool vec, float (&v)[4]) {
  if (vec && n >= 4) {
    Vec4<T>::load(p, v);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = i < n ? to_f32(p[i]) : 0.f;
  }
}
template <typename T>
__device__ __forceinline__ void store4(T* p, int n, bool vec, const float (&v)[4]) {
  if (vec && n >= 4) {
    Vec4<T>::store(p, v);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < n) p[i] = from_f32<T>(v[i]);
  }
}
// Addresses.  A group's activations [T, f] may have more than 2^31 elements, so element (row, col) lies at a 64-bit offset.
// fma_row: with the pitch of a row in bytes, two instructions (row times elements, scaled afterwards, takes three).
// fma_offset: from the start of a tile (at most 128 rows), whose own offset is 64-bit; 32 bits do there as long as a row
// has fewer than 2^24 elements (WIDE otherwise).  Which one a kernel uses was measured: one load per element has no
// registers left for the 64-bit rows (d = 1021, f = 2749: 6.45 ms a step against 5.90), the vector loads and the cp.async
// rings would rather not form the tile's offset for every block (8 segments of 128 tokens, d = 256: 199 us against 183).
template <typename T>
__host__ __device__ __forceinline__ const T* fma_row(const T* p, int row, size_t pitch) {
  return reinterpret_cast<const T*>(reinterpret_cast<const char*>(p) + (size_t)(unsigned)row * pitch);
}
template <bool WIDE>
__host__ __device__ __forceinline__ long fma_offset(int row, int ld, int col) {
  return WIDE ? (long)row * ld + col : (long)(row * ld + col);
}
__host__ __device__ __forceinline__ bool fma_wide(int ld) { return ld >= 1 << 24; }

__device__ __forceinline__ void fma2(float2& c, float a, const float2& b) {
  unsigned long long ap, &cp = reinterpret_cast<unsigned long long&>(c);
  asm("mov.b64 %0, {%1, %1};" : "=l"(ap) : "f"(a));
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(cp) : "l"(ap), "l"(reinterpret_cast<const unsigned long long&>(b)));
}

// Finishes one row of a thread's outputs: v[j] are the four columns c0 + j * STEP of the CTA's tile (two products: the first
// half of the j the gate, the second half the up values of the same columns).
template <typename T, int MODE, int EPI, int JN, int STEP>
__device__ __forceinline__ void fma_store_row(const FmaArgs& p, const FmaJob& J, float (&v)[JN][4], int g, int m, int n0, int c0,
                                              bool vec) {
  const size_t row = (size_t)g * J.c_g + (size_t)m * J.ldc;
  if constexpr (EPI == FMA_SWIGLU) {
#pragma unroll
    for (int j = 0; j < JN / 2; ++j) {
      const int n = n0 + c0 + j * STEP, left = J.N - n;
      if (left <= 0) continue;
      float h[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) h[i] = v[j][i] * sigmoidf_(v[j][i]) * v[j + JN / 2][i];
      store4(static_cast<T*>(J.C0) + row + n, left, vec, v[j]);
      store4(static_cast<T*>(J.C1) + row + n, left, vec, v[j + JN / 2]);
      store4(static_cast<T*>(J.C2) + row + n, left, vec, h);
    }
  } else {
#pragma unroll
    for (int j = 0; j < JN; ++j) {
      const int n = n0 + c0 + j * STEP, left = J.N - n;
      if (left <= 0) continue;
      if (EPI == FMA_DSWIGLU) {
        float gg[4], uu[4], du[4];
        load4(static_cast<const T*>(J.E0) + row + n, left, vec, gg);
        load4(static_cast<const T*>(J.E1) + row + n, left, vec, uu);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float s = sigmoidf_(gg[i]), dh = v[j][i];
          v[j][i] = dh * uu[i] * s * (1.0f + gg[i] * (1.0f - s));
          du[i] = dh * gg[i] * s;
        }
        store4(static_cast<T*>(J.C1) + row + n, left, vec, du);
      } else if (EPI == FMA_ROWADD) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i < left) v[j][i] += p.rowvec[(size_t)g * J.N + n + i] * p.row_scale;
      } else if (J.E0) {
        float o[4];
        load4(static_cast<const T*>(J.E0) + row + n, left, vec, o);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[j][i] += o[i];
      }
      store4(static_cast<T*>(J.C0) + row + n, left, vec, v[j]);
    }
  }
}

// A_K: A is stored [m][k] (else [k][m]); B_K: B is stored [n][k] (else [k][n]).  VEC: every row of A and B starts on a
// 4-element boundary and has a multiple of 4 elements (one load and one predicate per four elements: 35 -> 48 TFLOP/s at
// d = 768, f = 2064).  WIDE: see fma_offset (without VEC only).
template <typename T, bool A_K, bool B_K, int MODE, int EPI, int BM, int KG, bool VEC, bool WIDE = false>
__global__ void __launch_bounds__(128 * KG, 3) fma_gemm_kernel(const __grid_constant__ FmaArgs p) {
  constexpr int BN = 64, BK = 16, MR = BM / 16, W = VEC ? 4 : 1;   // W: elements per load
  constexpr int NA = BM * BK / 128 / W, NB = BN * BK / 128 / W;    // loads per thread and block
  constexpr int TILE_N = MODE == FMA_DUALB ? 32 : 64;
  __shared__ __align__(16) float sA[KG][2][BK][BM + 4];
  __shared__ __align__(16) float sB[KG][2][BK][BN + 4];
  const int kg = KG == 1 ? 0 : threadIdx.x >> 7, tid = threadIdx.x & 127, ty = tid >> 3, tx = tid & 7;
  int tile = blockIdx.x, ji = 0;
  while (ji + 1 < p.jobs && tile >= p.job[ji].tile_end) ++ji;
  const FmaJob& J = p.job[ji];
  tile -= ji ? p.job[ji - 1].tile_end : 0;
  pdl_launch();
  pdl_wait();
  const int m0 = tile % J.m_tiles * BM, rest = tile / J.m_tiles, n0 = rest % J.n_tiles * TILE_N, g = rest / J.n_tiles;
  const int nkb = (J.K + BK - 1) / BK, total = MODE == FMA_DUALK ? 2 * nkb : nkb;

  // Load j of a block is element (k, x) of the tile, x along m or n; W elements along the contiguous dimension.  In shared
  // memory a k-row is stored with x ^ 8 (k / 4) where the contiguous dimension is k: the four k-quads of one x, written by
  // neighbouring lanes, then lie on different banks.
  auto at = [&](bool kc, int width, int j, int& k, int& x) {
    const int idx = tid + j * 128;
    if (kc) {
      k = (idx & (BK / W - 1)) * W;
      x = idx / (BK / W);
    } else {
      x = idx % (width / W) * W;
      k = idx / (width / W);
    }
  };
  float ra[NA][W], rb[NB][W];
  const T* const A0 = static_cast<const T*>(J.A0) + (size_t)g * J.a_g;
  const T* const A1 = MODE == FMA_DUALK ? static_cast<const T*>(J.A1) + (size_t)g * J.a_g : A0;
  const T* const B0 = static_cast<const T*>(J.B0) + (size_t)g * J.b_g;
  const T* const B1 = MODE != FMA_PLAIN ? static_cast<const T*>(J.B1) + (size_t)g * J.b_g : B0;
  const size_t pa = (size_t)J.lda * sizeof(T), pb = (size_t)J.ldb * sizeof(T);
  auto load_w = [&](const T* q, bool ok, float (&v)[W]) {
    if (VEC) {
      float t[4] = {0.f, 0.f, 0.f, 0.f};
      if (ok) Vec4<T>::load(q, t);
#pragma unroll
      for (int i = 0; i < W; ++i) v[i] = t[i];
    } else {
      v[0] = ok ? to_f32(*q) : 0.f;
    }
  };
  auto fetch = [&](int i) {
    const bool second = MODE == FMA_DUALK && i >= nkb;
    const int k0 = (second ? i - nkb : i) * BK;
    // VEC: rows and columns of the matrix; else of the tile, which starts at these offsets
    const T* const A = (second ? A1 : A0) + (VEC ? 0 : fma_offset<true>(A_K ? m0 : k0, J.lda, A_K ? k0 : m0));
    const long b0 = VEC ? 0 : fma_offset<true>(B_K ? n0 : k0, J.ldb, B_K ? k0 : n0);
    auto elem = [&](const T* p, int r, int c, int ld, size_t pitch) { return VEC ? fma_row(p + c, r, pitch) : p + fma_offset<WIDE>(r, ld, c); };
#pragma unroll
    for (int j = 0; j < NA; ++j) {
      int k, x;
      at(A_K, BM, j, k, x);
      const int m = VEC ? m0 + x : x, kk = VEC ? k0 + k : k;
      load_w(elem(A, A_K ? m : kk, A_K ? kk : m, J.lda, pa), m0 + x < J.M && k0 + k < J.K, ra[j]);
    }
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      int k, x;
      at(B_K, BN, j, k, x);
      const bool up = MODE == FMA_DUALB && x >= 32;
      const int xn = up ? x - 32 : x;
      const int n = VEC ? n0 + xn : xn, kk = VEC ? k0 + k : k;
      load_w(elem((up || second ? B1 : B0) + b0, B_K ? n : kk, B_K ? kk : n, J.ldb, pb), n0 + xn < J.N && k0 + k < J.K, rb[j]);
    }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int j = 0; j < NA; ++j) {
      int k, x;
      at(A_K, BM, j, k, x);
#pragma unroll
      for (int i = 0; i < W; ++i) {
        if (A_K) sA[kg][buf][k + i][x ^ ((k + i) >> 2) * 8] = ra[j][i];
        else sA[kg][buf][k][x + i] = ra[j][i];
      }
    }
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      int k, x;
      at(B_K, BN, j, k, x);
#pragma unroll
      for (int i = 0; i < W; ++i) {
        if (B_K) sB[kg][buf][k + i][x ^ ((k + i) >> 2) * 8] = rb[j][i];
        else sB[kg][buf][k][x + i] = rb[j][i];
      }
    }
  };
  auto sync_group = [&] {
    if (KG == 1) __syncthreads();
    else asm volatile("bar.sync %0, 128;" ::"r"(kg + 1) : "memory");
  };

  // thread (ty, tx): rows ty * 4 .. + 3 and 64 + ty * 4 .. + 3 (BM = 128), one of the two (64) or ty * 2, + 1 (32);
  // columns tx * 4 .. + 3 and 32 + tx * 4 .. + 3
  float2 acc[MR][4];
#pragma unroll
  for (int i = 0; i < MR; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  int buf = 0;
  if (kg < total) {
    fetch(kg);
    put(0);
  }
  for (int i = kg; i < total; i += KG) {
    sync_group();
    const bool more = i + KG < total;
    if (more) fetch(i + KG);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[MR];
      if (MR >= 4) {
#pragma unroll
        for (int h = 0; h < MR / 4; ++h) {
          const float4 v = *reinterpret_cast<const float4*>(&sA[kg][buf][kk][h * 64 + (ty * 4 ^ (A_K ? (kk >> 2) * 8 : 0))]);
          a[(4 * h) % MR] = v.x; a[(4 * h + 1) % MR] = v.y; a[(4 * h + 2) % MR] = v.z; a[(4 * h + 3) % MR] = v.w;
        }
      } else {
        const float2 v = *reinterpret_cast<const float2*>(&sA[kg][buf][kk][ty * 2 ^ (A_K ? (kk >> 2) * 8 : 0)]);
        a[0] = v.x; a[1] = v.y;
      }
      const float4 b0 = *reinterpret_cast<const float4*>(&sB[kg][buf][kk][tx * 4 ^ (B_K ? (kk >> 2) * 8 : 0)]);
      const float4 b1 = *reinterpret_cast<const float4*>(&sB[kg][buf][kk][32 + (tx * 4 ^ (B_K ? (kk >> 2) * 8 : 0))]);
      const float2 b[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
      for (int r = 0; r < MR; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) fma2(acc[r][j], a[r], b[j]);
    }
    buf ^= 1;
    if (more) put(buf);
  }
  if (KG > 1) {
    // the groups' sums meet in shared memory (16 columns of accumulators at a time fit the A tiles)
    float* x = &sA[0][0][0][0];
    static_assert(KG <= 2, "two groups at most");
#pragma unroll
    for (int r = 0; r < MR; ++r) {
      __syncthreads();
      if (kg == 1) {
#pragma unroll
        for (int j = 0; j < 4; ++j) *reinterpret_cast<float2*>(&x[(j * 128 + tid) * 2]) = acc[r][j];
      }
      __syncthreads();
      if (kg == 0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 o = *reinterpret_cast<const float2*>(&x[(j * 128 + tid) * 2]);
          acc[r][j].x += o.x;
          acc[r][j].y += o.y;
        }
      }
    }
    if (kg == 1) return;
  }

  const bool vec = J.vec != 0;
#pragma unroll
  for (int r = 0; r < MR; ++r) {
    const int m = m0 + (MR >= 4 ? (r >> 2) * 64 + ty * 4 + (r & 3) : ty * 2 + r);
    if (m >= J.M) continue;
    float v[2][4] = {{acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y}, {acc[r][2].x, acc[r][2].y, acc[r][3].x, acc[r][3].y}};
    fma_store_row<T, MODE, EPI, 2, 32>(p, J, v, g, m, n0, tx * 4, vec);
  }
}

// -----------------------------------------------------------------------------------------------------------------
// The same for fp32 operands and too few tiles to fill the GPU: 32 x 64 tiles whose contraction is shared by the eight warps
// of a CTA, each with a cp.async ring of its own (transposing on the way where the contraction runs along the stored rows)
// and no barrier until the end, where the warps' sums meet in shared memory and every warp finishes one row in eight.  A lane
// computes 8 x 8 outputs, which needs a quarter of the shared-memory reads per FMA of the 2 x 8 above.  us, the kernel above ->
// this one, 8 segments of 128 tokens, d = 256, f = 688: gemm2 31 -> 23, dx 53 -> 27.
// -----------------------------------------------------------------------------------------------------------------
struct Fma32 {
  static constexpr int KG = 8, BM = 32, BN = 64, BK = 16, STG = 3;
  static constexpr int A_ROW = BM + 4, B_ROW = BN + 4, BLOCK = BK * (A_ROW + B_ROW);  // floats
  static constexpr int SMEM = KG * STG * BLOCK * 4;
};

// A_K, B_K, VEC as above.
template <bool A_K, bool B_K, int MODE, int EPI, bool VEC>
__global__ void __launch_bounds__(32 * Fma32::KG, 1) fma32_kernel(const __grid_constant__ FmaArgs p) {
  using F = Fma32;
  constexpr int KG = F::KG, BK = F::BK, STG = F::STG, JN = 2;
  constexpr int WA = VEC && !A_K ? 4 : 1, WB = VEC && !B_K ? 4 : 1;                // elements per copy
  constexpr int NA = F::BM * BK / 32 / WA, NB = F::BN * BK / 32 / WB;              // copies per lane and block
  constexpr int TILE_N = MODE == FMA_DUALB ? F::BN / 2 : F::BN;
  extern __shared__ __align__(16) float s_tile[];   // [warp][stage][A: BK rows of A_ROW | B: BK rows of B_ROW]
  const int kg = threadIdx.x >> 5, lane = threadIdx.x & 31, ty = lane >> 3, tx = lane & 7;
  int tile = blockIdx.x, ji = 0;
  while (ji + 1 < p.jobs && tile >= p.job[ji].tile_end) ++ji;
  const FmaJob& J = p.job[ji];
  tile -= ji ? p.job[ji - 1].tile_end : 0;
  const int m0 = tile % J.m_tiles * F::BM, rest = tile / J.m_tiles, n0 = rest % J.n_tiles * TILE_N, g = rest / J.n_tiles;
  const int nkb = (J.K + BK - 1) / BK, total = MODE == FMA_DUALK ? 2 * nkb : nkb;
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(s_tile + kg * STG * F::BLOCK);

  // Copy j of a block is element (k, x) of the tile, x along m or n; 1 or 4 elements along the contiguous dimension.  Where
  // that is k, a warp takes eight k of four neighbouring x: 32-byte pieces of memory, 32 different banks.
  auto at = [&](bool kc, int width, int w, int j, int& k, int& x) {
    const int idx = lane + j * 32;
    if (kc) {
      x = (idx >> 3) % width;
      k = (idx & 7) + 8 * ((idx >> 3) / width);
    } else {
      x = idx % (width / w) * w;
      k = idx / (width / w);
    }
  };
  // Columns of the B tile: for two products, 32 of the first and the same 32 of the second.
  auto b_col = [&](int x, bool& up) {
    up = MODE == FMA_DUALB && x >= 32;
    return n0 + (up ? x - 32 : x);
  };
  const float* const A0 = static_cast<const float*>(J.A0) + (size_t)g * J.a_g;
  const float* const A1 = MODE == FMA_DUALK ? static_cast<const float*>(J.A1) + (size_t)g * J.a_g : A0;
  const float* const B0 = static_cast<const float*>(J.B0) + (size_t)g * J.b_g;
  const float* const B1 = MODE != FMA_PLAIN ? static_cast<const float*>(J.B1) + (size_t)g * J.b_g : B0;
  const size_t pa = (size_t)J.lda * sizeof(float), pb = (size_t)J.ldb * sizeof(float);
  auto copy = [&](uint32_t dst, const float* src, bool ok, int w) {   // outside the matrix: zeros
    if (w == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16u : 0u) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(ok ? 4u : 0u) : "memory");
  };
  auto issue = [&](int i, int st) {
    if (i < total) {
      const bool second = MODE == FMA_DUALK && i >= nkb;
      const int k0 = (second ? i - nkb : i) * BK;
      const float* const A = second ? A1 : A0;
      const uint32_t sa = ring + st * F::BLOCK * 4, sb = sa + BK * F::A_ROW * 4;
#pragma unroll
      for (int j = 0; j < NA; ++j) {
        int k, x;
        at(A_K, F::BM, WA, j, k, x);
        const int m = m0 + x, kk = k0 + k;
        const bool ok = m < J.M && kk < J.K;
        copy(sa + (k * F::A_ROW + x) * 4, ok ? fma_row(A + (A_K ? kk : m), A_K ? m : kk, pa) : A0, ok, WA);
      }
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        int k, x;
        bool up;
        at(B_K, F::BN, WB, j, k, x);
        const int n = b_col(x, up), kk = k0 + k;
        const bool ok = n < J.N && kk < J.K;
        const float* const B = up || second ? B1 : B0;
        copy(sb + (k * F::B_ROW + x) * 4, ok ? fma_row(B + (B_K ? kk : n), B_K ? n : kk, pb) : B0, ok, WB);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  float2 acc[8][2 * JN];   // rows ty * 4 + (r & 3) + (r >> 2) * 16, columns tx * 4 + j * 32
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int j = 0; j < 2 * JN; ++j) acc[r][j] = make_float2(0.f, 0.f);
#pragma unroll
  for (int st = 0; st < STG - 1; ++st) issue(kg + st * KG, st);
  int st = 0;
  for (int i = kg; i < total; i += KG) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STG - 2) : "memory");
    __syncwarp();   // the block is complete, and every lane is done with the stage that is filled next
    issue(i + (STG - 1) * KG, st == 0 ? STG - 1 : st - 1);
    const float* const sa = s_tile + (kg * STG + st) * F::BLOCK + ty * 4;
    const float* const sb = s_tile + (kg * STG + st) * F::BLOCK + BK * F::A_ROW + tx * 4;
    st = st + 1 == STG ? 0 : st + 1;
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[8];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 v = *reinterpret_cast<const float4*>(sa + kk * F::A_ROW + h * 16);
        a[4 * h] = v.x; a[4 * h + 1] = v.y; a[4 * h + 2] = v.z; a[4 * h + 3] = v.w;
      }
      float2 b[2 * JN];
#pragma unroll
      for (int j = 0; j < JN; ++j) {
        const float4 v = *reinterpret_cast<const float4*>(sb + kk * F::B_ROW + j * 32);
        b[2 * j] = make_float2(v.x, v.y);
        b[2 * j + 1] = make_float2(v.z, v.w);
      }
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int j = 0; j < 2 * JN; ++j) fma2(acc[r][j], a[r], b[j]);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();   // the rings have been read
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int j = 0; j < 2 * JN; ++j) {
      s_tile[(kg * 64 + r * 8 + 2 * j) * 32 + lane] = acc[r][j].x;
      s_tile[(kg * 64 + r * 8 + 2 * j + 1) * 32 + lane] = acc[r][j].y;
    }
  __syncthreads();
  const int r = kg, m = m0 + ty * 4 + (r & 3) + (r >> 2) * 16;   // this warp's row of every lane's eight
  if (m >= J.M) return;
  float v[JN][4];
#pragma unroll
  for (int j = 0; j < JN; ++j)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float sum = 0.f;
#pragma unroll
      for (int q = 0; q < KG; ++q) sum += s_tile[(q * 64 + r * 8 + 4 * j + c) * 32 + lane];
      v[j][c] = sum;
    }
  fma_store_row<float, MODE, EPI, JN, 32>(p, J, v, g, m, n0, tx * 4, J.vec != 0);
}

}  // namespace lory
