// Decode: the cached merged FFN of each sequence on a few new tokens per sequence.
//
//   H = silu(X Wbar1^T) * (X Wbar3^T)      Y = H Wbar2^T       per segment (= sequence), n <= 64 tokens
//
// Bound by reading the merged weights once (6 d f bytes per sequence) whatever n is, so what counts is that every SM has
// enough of them on the way from the first moment to the last.  The grouped GEMM (tokens as the 128-row operand, 256- or
// 64-column tiles) has too few tiles for that with few sequences (22 for one sequence at f = 2752) and an uneven last wave
// with more.  Here the WEIGHT ROWS are the M dimension of warp-level matrix instructions (m16n8k16) and the tokens the N
// dimension.  A CTA takes tiles of MT x 16 weight rows (8 of Wbar1 and the same 8 of Wbar3, so that a lane ends up with gate
// and up value of one hidden unit; 16 or 8 rows of Wbar2) and its eight warps each an eighth of the contraction; their
// sums meet in shared memory.  A warp's weights come through a cp.async ring of its own that runs ahead across tile
// boundaries, so neither a tile's reduction nor its end leaves the memory idle (loading each tile's weights into
// registers: 118 instead of 92 us for eight sequences at d = 2048, f = 5504).  Any assignment of a block's 64 columns to k
// positions will do as long as both operands use the same, so a lane reads whole 16-byte vectors (groups t and t + 4 of a
// row).  The second kernel is launched while the first runs (programmatic dependent launch) and has its first weights on
// the way before it waits for H.
// us per call, grouped GEMM -> here, d = 1024, f = 2752, one token: 1 sequence 32.8 -> 9.0, 8: 45.5 -> 26.3, 32: 122 -> 85
// (6.4 TB/s); 40 tokens, 4 sequences: 36.3 -> 30.5.
#pragma once
#include "common.cuh"
#include "stream_tc.cuh"

namespace lory {

struct DecodeParams {
  const bf16 *wa, *wb;  // blocked weights [R, K] of every segment: Wbar1, Wbar3 (gate) or Wbar2
  const bf16* x;        // [S, n, K] tokens: x or H
  bf16* out;            // [S, n, R]: H or Y
  int S, n, R, K, Cb;   // Cb = 64-column blocks of a weight row
  uint32_t* status;     // cleared by the gate kernel (nothing here could time out)
};

enum DecodeMode { DECODE_GATE = 0, DECODE_16 = 1, DECODE_8 = 2 };

// NT: token tiles of 8.  MT: weight tiles of 16 rows worked on together, so that a token value fetched serves them all.
template <int MODE, int NT, int MT>
struct Decode {
  static constexpr int TR = MT * (MODE == DECODE_16 ? 16 : 8);         // output rows per tile
  static constexpr int STAGE = MT * (MODE == DECODE_8 ? 8 : 16) * 128; // one 64-column block of a tile's rows
  static constexpr int RED = 8 * MT * NT * 512;                        // the warps' sums
  static constexpr int CTAS = RED <= 16384 ? 2 : 1;
  static constexpr int FIT = (226 * 1024 / CTAS - 1024 - RED) / (8 * STAGE);
  static constexpr int STG = FIT > 5 ? 5 : FIT;
  static constexpr int SMEM = 8 * STG * STAGE + RED;
  static_assert(STG >= 3, "two blocks per warp on the way");
};

template <int MODE, int NT, int MT>
__global__ void __launch_bounds__(256, Decode<MODE, NT, MT>::CTAS) decode_kernel(const __grid_constant__ DecodeParams p) {
  using D = Decode<MODE, NT, MT>;
  constexpr int TR = D::TR, STG = D::STG;
  constexpr bool TWO = MODE != DECODE_8;   // rows 8..15 of the instruction are used
  extern __shared__ uint4 s_w[];           // [warp][stage][rows][128 B], then the warps' sums
  float4* red = reinterpret_cast<float4*>(s_w) + 8 * STG * D::STAGE / 16;  // [warp][MT][NT][lane]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int tps = (p.R + TR - 1) / TR, tiles = tps * p.S;
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(s_w) + warp * (STG * D::STAGE);
  if (MODE == DECODE_GATE) {
    pdl_wait();  // whatever ran before may have written x or the weights
    if (blockIdx.x == 0 && threadIdx.x == 0) *p.status = 0;
  }
  pdl_launch();  // after the wait: a dependent kernel that starts now finds the weights complete
  // the issuing cursor: the block to load next, STG - 1 blocks ahead of the one being used
  int it = blockIdx.x, icb = warp;
  const int row0 = lane >> 3, c = lane & 7;
  auto issue = [&](uint32_t stage) {
    while (it < tiles && icb >= p.Cb) {
      it += gridDim.x;
      icb = warp;
    }
    if (it < tiles) {
      const int s = it / tps, r0 = (it - s * tps) * TR;
      const uint32_t d0 = stage + row0 * 128 + ((c ^ stage_swizzle(row0)) << 4);
      const uint32_t d1 = stage + row0 * 128 + 512 + ((c ^ stage_swizzle(row0 + 4)) << 4);
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const int r = r0 + m * (TR / MT);   // the merge pads rows to a multiple of 64, a tile never leaves them
        const size_t o = (((size_t)(r >> 6) * p.Cb + icb) * p.S + s) * 4096 + (size_t)((r & 63) + row0) * 64 + c * 8;
        cp_async_16b(d0 + m * 2048, p.wa + o, 16u);
        cp_async_16b(d1 + m * 2048, p.wa + o + 4 * 64, 16u);
        if (TWO) {
          const bf16* b = MODE == DECODE_GATE ? p.wb + o : p.wa + o + 8 * 64;
          cp_async_16b(d0 + m * 2048 + 1024, b, 16u);
          cp_async_16b(d1 + m * 2048 + 1024, b + 4 * 64, 16u);
        }
      }
      icb += 8;
    }
    cp_async_commit();
  };
#pragma unroll
  for (int i = 0; i < STG - 1; ++i) issue(ring + i * D::STAGE);
  if (MODE != DECODE_GATE) pdl_wait();  // H is complete from here on
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  int cur = 0;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int s = tile / tps, r0 = (tile - s * tps) * TR;
    const bf16* xs = p.x + (size_t)s * p.n * p.K;
    float acc[MT][NT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int j = 0; j < NT; ++j) acc[m][j][0] = acc[m][j][1] = acc[m][j][2] = acc[m][j][3] = 0.f;
    for (int cb = warp; cb < p.Cb; cb += 8) {
      const int c0 = cb * 64 + t * 8;
      uint4 x[NT][2];
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const int tok = j * 8 + g;
        const bf16* q = xs + (size_t)tok * p.K + c0;
        x[j][0] = (tok < p.n && c0 < p.K) ? *reinterpret_cast<const uint4*>(q) : zero;
        x[j][1] = (tok < p.n && c0 + 32 < p.K) ? *reinterpret_cast<const uint4*>(q + 32) : zero;
      }
      cp_async_wait<STG - 2>();
      __syncwarp();
      issue(ring + (cur == 0 ? STG - 1 : cur - 1) * D::STAGE);
      const uint32_t a = ring + cur * D::STAGE + g * 128, k0 = (uint32_t)(t ^ stage_swizzle(g)) << 4, k1 = k0 ^ 64u;
      cur = cur + 1 == STG ? 0 : cur + 1;
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        const uint32_t am = a + m * 2048;
        const uint4 w0 = lds_16b(am + k0), w2 = lds_16b(am + k1);
        const uint4 w1 = TWO ? lds_16b(am + 1024 + k0) : zero, w3 = TWO ? lds_16b(am + 1024 + k1) : zero;
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i)
            mma_bf16_16x8x16(acc[m][j], make_uint4(word_of(w0, i), word_of(w1, i), word_of(w2, i), word_of(w3, i)),
                             word_of(x[j][0], i), word_of(x[j][1], i));
      }
    }
    if (tile != (int)blockIdx.x) __syncthreads();  // the previous tile's sums have been read
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int j = 0; j < NT; ++j)
        red[((warp * MT + m) * NT + j) * 32 + lane] = make_float4(acc[m][j][0], acc[m][j][1], acc[m][j][2], acc[m][j][3]);
    __syncthreads();
    for (int i = threadIdx.x; i < MT * NT * 32; i += 256) {
      const int ln = i & 31, j = (i >> 5) % NT, m = (i >> 5) / NT;
      float4 v = red[i];
#pragma unroll
      for (int q = 1; q < 8; ++q) {
        const float4 o = red[q * MT * NT * 32 + i];
        v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
      }
      const int r = r0 + m * (TR / MT) + (ln >> 2), tok = j * 8 + 2 * (ln & 3);
      bf16* o = p.out + ((size_t)s * p.n + tok) * p.R + r;
      if (MODE == DECODE_GATE) {
        v.x = v.x * sigmoid_fast(v.x) * v.z;
        v.y = v.y * sigmoid_fast(v.y) * v.w;
      }
      if (r < p.R && tok < p.n) o[0] = __float2bfloat16_rn(v.x);
      if (r < p.R && tok + 1 < p.n) o[p.R] = __float2bfloat16_rn(v.y);
      if (MODE == DECODE_16) {
        if (r + 8 < p.R && tok < p.n) o[8] = __float2bfloat16_rn(v.z);
        if (r + 8 < p.R && tok + 1 < p.n) o[p.R + 8] = __float2bfloat16_rn(v.w);
      }
    }
  }
  cp_async_wait<0>();
}

}  // namespace lory
