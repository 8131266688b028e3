// Plain FMA (CUDA-core) contractions.  These carry the fp32 mode (tensor cores cannot meet its 1e-4 tolerance) and the
// diagnostic LORY_FLAG_SIMT mode of the bf16 path.
#pragma once
#include "common.cuh"
#include "fma_gemm.cuh"

namespace lory {

// C_g[m,n] (+)= sum_k A_g[m,k] * B_g[k,n], fp32 accumulation, arbitrary element strides (the merge and its adjoint with
// more experts or segments than the kernels below hold).
// With k_chunk > 0 the K range is split: group g covers k in [g*k_chunk, min(K,(g+1)*k_chunk))
// (a_g / b_g are ignored), and C_g is the g-th partial slab.
struct SimtGemm {
  const void* A; const void* B; void* C;
  int M, N, K, groups;
  long a_m, a_k, a_g;
  long b_k, b_n, b_g;
  long c_m, c_n, c_g;
  int k_chunk;
  int accumulate;
};

template <typename TA, typename TB, typename TC>
int launch_simt_gemm(const SimtGemm& g, cudaStream_t st);

// The contractions of the merged FFNs (fma_gemm.cuh).  Unused jobs' fields: M = 0.  m_tiles .. vec are filled in here.
template <typename T> int fma_gemm_swiglu(FmaJob j, int groups, cudaStream_t st);             // A [m][k], B0, B1 [n][k]
template <typename T> int fma_gemm_nt(FmaJob j, int groups, cudaStream_t st);                 // A [m][k], B [n][k]
template <typename T> int fma_gemm_dswiglu(FmaJob j, int groups, cudaStream_t st);            // A [m][k], B [k][n]
template <typename T> int fma_gemm_tn(const FmaJob (&j)[3], int groups, cudaStream_t st);     // A [k][m], B [k][n], three problems
template <typename T> int fma_gemm_dx(FmaJob j, int groups, const float* rowvec, float scale, cudaStream_t st);

// Merge and adjoint over the three expert matrices of n parameters each (all [., n] row-major), up to 32 experts.
template <typename T>
struct FmaMerge {
  const T* w[3];     // experts [E, n]
  T* wbar[3];        // merged weights [S, n] (the adjoint: their gradients, read)
  T* dw[3];          // adjoint: expert gradients [E, n]
  const float* route;  // [S, E]
  float* slabs;      // adjoint: [fma_adjoint_slabs, S, E]
  long n;
  int S, E, accumulate;
};
bool fma_merge_supported(int S, int E);
int fma_adjoint_slabs(long n);
template <typename T> int launch_fma_merge(const FmaMerge<T>& p, cudaStream_t st);
template <typename T> int launch_fma_adjoint(const FmaMerge<T>& p, cudaStream_t st);

}  // namespace lory
