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
// (6.4 TB/s).
#pragma once
#include <cuda.h>

#include "common.cuh"
#include "stream_tc.cuh"
#include "umma.cuh"

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

// -----------------------------------------------------------------------------------------------------------
// The same for 17 to 64 tokens, on tcgen05: weights as the 128-row operand, tokens as the 16- to 64-column one, both by TMA
// into one ring, accumulators in TMEM (two of them, so that a tile's way out overlaps the next one's contraction).  A gate
// tile is 64 rows of Wbar1 and the same 64 of Wbar3; a down-projection tile of 64 rows (tr = 64) lets the instruction's other
// rows read whatever follows in shared memory and end in accumulator lanes that nobody looks at.
// Bound by HBM once there is enough to do (32 sequences, 64 tokens, d = 2048, f = 5504: 685 -> 340 us, 6.4 TB/s), before that by
// the chain of one thread per stage (barrier, copies or MMAs, barrier: 0.2 us, whatever the bytes): hence two or three column
// blocks per stage, weights and tokens copied by a thread each, and no arithmetic in those loops that need not be there.
// Warps: 0 and 6 TMA, 1 MMA, 2..5 epilogue.
// -----------------------------------------------------------------------------------------------------------
struct DecodeMma {
  int S, n, R, K;
  int tr, kb;        // weight rows of a tile (gate: 128, both matrices together), 64-column blocks of a stage
  int nb;            // n rounded up to 16: columns of the instruction
  int stages, tail;  // ring; bytes behind it: the up values, and what the last stage's 128-row operand reads may touch
  bf16* out;         // [S, n, R]: H or Y
  uint32_t* status;
};

template <bool GATE>
__global__ void __launch_bounds__(224) decode_mma_kernel(const __grid_constant__ CUtensorMap tmW0,
                                                         const __grid_constant__ CUtensorMap tmW1,
                                                         const __grid_constant__ CUtensorMap tmX,
                                                         const __grid_constant__ DecodeMma p) {
  constexpr int MAX_STAGES = 8;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full_bar[MAX_STAGES], empty_bar[MAX_STAGES], tmem_full_bar[2], tmem_empty_bar[2];
  __shared__ uint32_t tmem_base_smem;
  __shared__ volatile uint32_t abort_flag;
  const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
  const int a_bytes = p.tr * 128, kb_bytes = a_bytes + p.nb * 128, stage_bytes = p.kb * kb_bytes;
  const int tile_rows = GATE ? p.tr / 2 : p.tr;
  const int tps = (p.R + tile_rows - 1) / tile_rows, tiles = tps * p.S;
  const int steps = ((p.K + 63) / 64 + p.kb - 1) / p.kb;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      ptx::mbar_init(&full_bar[s], 2);
      ptx::mbar_init(&empty_bar[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&tmem_full_bar[a], 1);
      ptx::mbar_init(&tmem_empty_bar[a], 128);
    }
    abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(&tmW0);
    if (GATE) ptx::prefetch_tmap(&tmW1);
    ptx::prefetch_tmap(&tmX);
  }
  if (warp == 1) {
    ptx::tmem_alloc(&tmem_base_smem, 128);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = tmem_base_smem;
  if (GATE) {
    pdl_wait();  // whatever ran before may have written x or the weights
    if (!dbg::kOn && blockIdx.x == 0 && threadIdx.x == 0) *p.status = 0;
  }
  pdl_launch();  // after the wait: a dependent kernel that starts now finds the weights complete

  if (warp == 0 || warp == 6) {
    // the weights and the tokens of a stage, from one thread each: half the chain of copies per stage
    if (ptx::elect_one() && dbg::check(dbg::smem_ok(smem, p.stages * stage_bytes + p.tail), p.status)) {
      const bool weights = warp == 0;
      if (!GATE && !weights) pdl_wait();  // H is complete from here on; the weights were before
      const uint32_t tx = (uint32_t)(p.kb * (weights ? a_bytes : kb_bytes - a_bytes));
      uint32_t ph = 0, issued = 0, last_parity = 0;
      int s = 0;
      for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int g = tile / tps, r0 = (tile - g * tps) * tile_rows;
        for (int cb = 0; cb < steps * p.kb;) {
          if (!ptx::mbar_wait(&empty_bar[s], ph ^ 1, &abort_flag)) {
            atomicOr(p.status, STATUS_TIMEOUT_TMA);
            abort_flag = 1;
          }
          ptx::mbar_expect_tx(&full_bar[s], tx);
          uint8_t* d = smem + s * stage_bytes;
          if (weights) {
            for (int j = 0; j < p.kb; ++j, ++cb, d += kb_bytes) {   // past the last block: zeros
              ptx::tma_load_5d(d, &tmW0, &full_bar[s], 0, r0 & 63, g, cb, r0 >> 6);
              if (GATE) ptx::tma_load_5d(d + a_bytes / 2, &tmW1, &full_bar[s], 0, r0 & 63, g, cb, r0 >> 6);
            }
          } else {
            for (int j = 0; j < p.kb; ++j, ++cb, d += kb_bytes)
              ptx::tma_load_3d(d + a_bytes, &tmX, &full_bar[s], cb * 64, 0, g);
          }
          issued |= 1u << s;
          last_parity = (last_parity & ~(1u << s)) | (ph << s);
          if (++s == p.stages) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (abort_flag) {
        // let this thread's copies in flight land before the CTA's shared memory goes away
        for (int q = 0; q < p.stages; ++q)
          if (issued & (1u << q)) ptx::mbar_wait(&full_bar[q], (last_parity >> q) & 1, &abort_flag, 1u << 20);
      }
    }
  } else if (warp == 1) {
    if (ptx::elect_one()) {
      const uint32_t idesc = ptx::make_idesc_bf16(128, p.nb, false, false);
      const uint64_t desc0 = ptx::make_smem_desc(0, 16, 1024);
      const uint32_t smem16 = ptx::smem_u32(smem) >> 4;
      int s = 0;
      uint32_t ph = 0, it = 0;
      for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++it) {
        const uint32_t acc = it & 1;
        if (!ptx::mbar_wait(&tmem_empty_bar[acc], ((it >> 1) & 1) ^ 1, &abort_flag)) {
          atomicOr(p.status, STATUS_TIMEOUT_MMA);
          abort_flag = 1;
        }
        ptx::tc_fence_after_sync();
        const uint32_t d = tmem_base + acc * 64;
        const bool acc_ok = dbg::check(dbg::tmem_ok(d, tmem_base, 128, 64), p.status);
        for (int i = 0; i < steps; ++i) {
          if (!ptx::mbar_wait(&full_bar[s], ph, &abort_flag)) {
            atomicOr(p.status, STATUS_TIMEOUT_MMA);
            abort_flag = 1;
          }
          ptx::tc_fence_after_sync();
          uint32_t a16 = smem16 + ((uint32_t)(s * stage_bytes) >> 4);
          for (int j = 0; j < p.kb; ++j, a16 += (uint32_t)kb_bytes >> 4) {
            const uint32_t b16 = a16 + ((uint32_t)a_bytes >> 4);
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (acc_ok)
                ptx::umma_bf16(d, desc0 | ((a16 + 2 * k) & 0x3FFFu), desc0 | ((b16 + 2 * k) & 0x3FFFu), idesc,
                               (i > 0 || j > 0 || k > 0) ? 1u : 0u);
          }
          ptx::umma_commit(&empty_bar[s]);
          if (++s == p.stages) {
            s = 0;
            ph ^= 1;
          }
        }
        ptx::umma_commit(&tmem_full_bar[acc]);
      }
    }
  } else {
    const int q = warp & 3, row = q * 32 + lane;   // TMEM lane quarter this warp may read; weight row of the tile
    const int half = p.tr / 2;
    float* s_up = reinterpret_cast<float*>(smem + (size_t)p.stages * stage_bytes);  // gate: [nb][tr / 2]
    uint32_t it = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++it) {
      const int g = tile / tps, r0 = (tile - g * tps) * tile_rows;
      const uint32_t acc = it & 1;
      if (!ptx::mbar_wait(&tmem_full_bar[acc], (it >> 1) & 1, &abort_flag)) {
        atomicOr(p.status, STATUS_TIMEOUT_EPI);
        abort_flag = 1;
      }
      __syncwarp();  // every lane polls by itself; the warp-wide tcgen05 instructions below need it whole again
      ptx::tc_fence_after_sync();
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + acc * 64;
      uint32_t v[64];
      const bool mine = q * 32 < p.tr && dbg::check(dbg::tmem_ok(taddr, tmem_base, 128, 64), p.status);
      if (mine) {
        ptx::tmem_ld_32x64(taddr, v);
        ptx::tmem_ld_wait();
      }
      ptx::tc_fence_before_sync();
      ptx::mbar_arrive(&tmem_empty_bar[acc]);
      bf16* o = p.out + (size_t)g * p.n * p.R + r0;
      if (GATE) {
        const bool up = row >= half && row < p.tr, gate = row < half && r0 + row < p.R;
        if (mine && up) {
#pragma unroll
          for (int j = 0; j < 64; ++j)
            if (j < p.n) s_up[j * half + row - half] = __uint_as_float(v[j]);
        }
        ptx::named_barrier(1, 128);
        if (mine && gate) {
#pragma unroll
          for (int j = 0; j < 64; ++j)
            if (j < p.n) {
              const float a = __uint_as_float(v[j]);
              o[(size_t)j * p.R + row] = __float2bfloat16_rn(a * sigmoid_fast(a) * s_up[j * half + row]);
            }
        }
        ptx::named_barrier(1, 128);  // the up values have been read
      } else if (mine && row < p.tr && r0 + row < p.R) {
#pragma unroll
        for (int j = 0; j < 64; ++j)
          if (j < p.n) o[(size_t)j * p.R + row] = __float2bfloat16_rn(__uint_as_float(v[j]));
      }
    }
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) ptx::tmem_dealloc(tmem_base, 128);
}

}  // namespace lory
