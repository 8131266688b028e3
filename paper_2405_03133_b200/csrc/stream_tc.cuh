// The merge (Eq. 2), and its adjoint for few segments, as streaming kernels: operands go from global memory to the
// fragments of warp-level matrix instructions, results from the accumulators to global memory.
//
// Both passes are bound by HBM.  Kernels that stage fixed tiles through TMA, shared memory and TMEM do not reach that
// bound, least of all with few segments: a tile then moves few bytes while its chain (TMA, barrier, MMA, TMEM load,
// staging, store) stays as long.  Here a warp works on a PIECE of 64 consecutive parameters of one matrix row with no barrier to any other
// warp, and 8 to 16 such warps per SM have their loads in flight at the same time.  Tensor throughput is no concern: an
// m16n8k16 takes 8.5 cycles of an SM quarter, and a piece needs 2 of them per 256 products of (segment, expert), a third
// of the time its bytes take or less.
//
// Fragment layout.  In m16n8k16 (g = lane / 4, t = lane % 4) a thread holds of B the column g at k = 2t, 2t+1, 2t+8,
// 2t+9 and of the accumulator rows g, g+8 at columns 2t, 2t+1.  Eight such instructions cover a piece if instruction j
// takes parameter 8 g + j as its column g: a thread then loads whole 16-byte vectors (eight parameters of one expert
// or segment), pairs two rows of them with byte permutes, and ends up with 16 CONSECUTIVE parameters of its two
// result rows, which leave as one 32-byte store per row, four lanes filling a 128-byte line.  Whole lines matter:
// with 16-byte stores (half a line per instruction) the store stream alone ran at 3.3 TB/s, with 32-byte ones at
// 5.3 TB/s (d = 2048, f = 5504, E = 32), and the adjoint took 1.30 instead of 0.95 ms.
#pragma once
#include "common.cuh"

namespace lory {

__device__ __forceinline__ void mma_bf16_16x8x16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
// 16 bytes that are read once
__device__ __forceinline__ uint4 ld_stream(const bf16* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
// 32 bytes, 32-byte aligned
__device__ __forceinline__ void st_32b(bf16* p, const uint4& a, const uint4& b) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z),
               "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
               : "memory");
}
__device__ __forceinline__ uint4 lds_16b(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
// 16 bytes global -> shared; the last 16 - bytes of them become zero
__device__ __forceinline__ void cp_async_16b(uint32_t dst, const bf16* src, uint32_t bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ uint32_t word_of(const uint4& v, int i) {
  return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w));
}
__device__ __forceinline__ uint32_t pack_pair(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}
// Two fp32 values as packed bf16 hi and lo parts (hi + lo keeps about 16 bits).
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& hi, uint32_t& lo) {
  const float ha = __bfloat162float(__float2bfloat16_rn(a)), hb = __bfloat162float(__float2bfloat16_rn(b));
  hi = pack_pair(ha, hb);
  lo = pack_pair(a - ha, b - hb);
}
// The A fragment (hi and lo) of lane `ln` for the 16 x 16 table val(row, col).
template <typename F>
__device__ __forceinline__ void a_fragment(int ln, F val, uint4& hi, uint4& lo) {
  const int g = ln >> 2, t = ln & 3;
  split_pair(val(g, 2 * t), val(g, 2 * t + 1), hi.x, lo.x);
  split_pair(val(g + 8, 2 * t), val(g + 8, 2 * t + 1), hi.y, lo.y);
  split_pair(val(g, 2 * t + 8), val(g, 2 * t + 9), hi.z, lo.z);
  split_pair(val(g + 8, 2 * t + 8), val(g + 8, 2 * t + 9), hi.w, lo.w);
}
// B fragments of a piece, one per instruction j, from the vectors of rows 2t, 2t+1, 2t+8, 2t+9.
__device__ __forceinline__ void b_fragments(const uint4 (&v)[4], uint32_t (&b)[8][2]) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t sel = (j & 1) ? 0x7632u : 0x5410u;
    b[j][0] = __byte_perm(word_of(v[0], j >> 1), word_of(v[1], j >> 1), sel);
    b[j][1] = __byte_perm(word_of(v[2], j >> 1), word_of(v[3], j >> 1), sel);
  }
}

// -----------------------------------------------------------------------------------------------------------
// Merge: Wbar_k[s, p] = sum_e w[s, e] W_k[e, p] into the blocked layout, A = (w_hi + w_lo), B = the experts, for any
// number of segments (with many of both the matrix instructions become the bound, and merge_tc.cuh takes over).
// KT = ceil(E / 16).  A warp loads U consecutive pieces of all experts into registers and then walks the segments, 16 at a
// time, with the weight fragments the routing step has prepared (they stay in L1).
// HBM-bound: algorithmic bytes 2 (E + S) per parameter.  The CTAs are small (two warps) and each does its pieces and
// ends, so the hardware hands out work as SMs get through theirs: SMs differ by 1.4 x in the rate at which they get
// writes out, and every persistent grid (the tcgen05 kernel this one replaced among them) waits for the slowest.
// Measured against that kernel: S = 8, E = 8, d = 1024, f = 2752: 160 -> 70 us; S = 128, E = 32: 535 -> 450 us (6.0 TB/s);
// S = 256, E = 32, d = 2048, f = 5504: 4.12 -> 3.49 ms; S = 64: 1.34 -> 1.03 ms.  With eight warps per CTA: 575 us
// instead of 450, with a persistent grid of the same CTAs: 600 us.
// -----------------------------------------------------------------------------------------------------------
struct StreamMergeParams {
  const bf16* src[3];
  bf16* dst[3];
  int R[3], C[3], Cb[3];   // rows and columns of the matrices; 64-column blocks per row
  unsigned piece_end[3];   // exclusive prefix sums of (rows rounded up to 64) * Cb: padded rows are written as zeros
  const uint4* w_frag;     // weight fragments of every segment (see w_frag_offset)
  int S, E;
};

template <int KT, int U, int NW>
__global__ void __launch_bounds__(32 * NW) merge_stream_kernel(const __grid_constant__ StreamMergeParams p) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const unsigned total = p.piece_end[2];
  const unsigned base = (blockIdx.x * NW + warp) * U;
  pdl_launch();
  pdl_wait();
  if (base >= total) return;
  uint4 v[U][KT][4];
  bf16* out[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const unsigned i = base + u;
    const int k = i < p.piece_end[0] ? 0 : (i < p.piece_end[1] ? 1 : 2);
    const unsigned l = i - (k == 0 ? 0u : p.piece_end[k - 1]);
    // the 64 rows of a 64 x 64 block are neighbours in this order
    const unsigned rb = (l >> 6) / p.Cb[k], cb = (l >> 6) - rb * p.Cb[k], r = rb * 64 + (l & 63);
    out[u] = p.dst[k] + ((size_t)rb * p.Cb[k] + cb) * p.S * 4096 + (r & 63) * 64 + t * 16;
    const int col = (int)cb * 64 + g * 8;
    const bool in = i < total && (int)r < p.R[k] && col < p.C[k];
    const bf16* src = p.src[k] + (size_t)r * p.C[k] + col;
    const size_t es = (size_t)p.R[k] * p.C[k];
#pragma unroll
    for (int kk = 0; kk < KT; ++kk)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = kk * 16 + 2 * t + (q & 1) + (q >> 1) * 8;
        v[u][kk][q] = make_uint4(0u, 0u, 0u, 0u);
        if (in && e < p.E) v[u][kk][q] = ld_stream(src + (size_t)e * es);
      }
  }
  uint32_t b[U][KT][8][2];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int kk = 0; kk < KT; ++kk) b_fragments(v[u][kk], b[u][kk]);
  const uint4* wf = p.w_frag + lane;
#pragma unroll 1
  for (int m = 0; m < p.S; m += 16, wf += KT * 64) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (u > 0 && base + u >= total) break;
      float acc[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll
      for (int kk = 0; kk < KT; ++kk) {
        const uint4 hi = __ldg(wf + kk * 64), lo = __ldg(wf + kk * 64 + 32);
#pragma unroll
        for (int j = 0; j < 8; ++j) mma_bf16_16x8x16(acc[j], hi, b[u][kk][j][0], b[u][kk][j][1]);
#pragma unroll
        for (int j = 0; j < 8; ++j) mma_bf16_16x8x16(acc[j], lo, b[u][kk][j][0], b[u][kk][j][1]);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int s = m + g + h * 8, c = 2 * h;
        if (s < p.S)
          st_32b(out[u] + (size_t)s * 4096,
                 make_uint4(pack_pair(acc[0][c], acc[1][c]), pack_pair(acc[2][c], acc[3][c]),
                            pack_pair(acc[4][c], acc[5][c]), pack_pair(acc[6][c], acc[7][c])),
                 make_uint4(pack_pair(acc[0][c + 1], acc[1][c + 1]), pack_pair(acc[2][c + 1], acc[3][c + 1]),
                            pack_pair(acc[4][c + 1], acc[5][c + 1]), pack_pair(acc[6][c + 1], acc[7][c + 1])));
      }
    }
  }
}

// -----------------------------------------------------------------------------------------------------------
// Adjoint of the merge, one pass over the per-segment weight gradients:
//   dW_k[e, p] = sum_s w[s, e] dWbar_k[s, p]      dw[s, e] += sum_p dWbar_k[s, p] W_k[e, p]
// for S <= 16 ST segments and E <= 16 ET experts.  ACC: dW_k receives its old value plus the sum.
// The rows of a piece (experts, segments, old gradients: 128 bytes each) come by cp.async into a ring of STG stages
// that belongs to ONE warp, so that the next pieces are on their way while one is worked on, at no cost in registers
// and without a barrier between warps (S = 16, E = 16, d = 2048, f = 5504: 548 us, 5.9 TB/s; loading straight into
// registers 710 us, the tcgen05 kernel 1.09 ms; with the old values read by the epilogue, as that kernel does,
// accumulation took 1.60 ms, here 0.70).
// The second product contracts over parameters: both its operands are rows of the piece, and any assignment of the
// 64 parameters to k positions will do, so a lane reads whole vectors (16-byte groups t and t + 4 of row g).  The dw
// sums stay in registers for the whole kernel and leave as one slab per CTA, the warps added in a fixed order.
// -----------------------------------------------------------------------------------------------------------
struct StreamAdjointParams {
  const bf16* dsrc[3];   // blocked per-segment gradients of a rectangle [R, C] of matrix k
  const bf16* wsrc[3];   // first element of the rectangle in the experts ...
  bf16* ddst[3];         // ... and in their gradients
  int R[3], C[3], Cb[3];
  long e_stride[3], row_stride[3];
  unsigned piece_end[3]; // exclusive prefix sums of R * Cb
  const float* w;        // [S, E]
  int S, E;
  int stages;            // ring stages in use (2 or 3)
  int slab_add;          // add to the slab (a launch that covers part of the parameters)
  float* dw_partial;     // [grid, S, E]
};

template <int ST, int ET, bool ACC>
struct AdjointStream {
  static constexpr int NW = 4;                          // warps per CTA
  static constexpr int STAGE = 16 * (ST + (ACC ? 2 : 1) * ET) * 128;
  static constexpr int FIXED = ET * ST * 1024 + ST * ET * 1024;  // weight fragments; dw sums
  static constexpr int ROOM = 224 * 1024;               // of an SM's shared memory
  static constexpr int fit(int ctas) { return (ROOM / ctas - 1024 - FIXED) / (NW * STAGE); }
  // CTAs per SM: three while the registers allow it (ST * ET <= 2), as long as every warp gets its two stages
  static constexpr int CTAS = ST * ET <= 2 && fit(3) >= 2 ? 3 : (fit(2) >= 2 ? 2 : 1);
  static constexpr int STG = fit(CTAS) > 3 ? 3 : fit(CTAS);   // at most; see stages
  static constexpr int SMEM = FIXED + NW * STG * STAGE;
  static_assert(STG >= 2, "a piece has to load while another is worked on");
};

// Where 16-byte chunk c of row r of a stage lies: c ^ stage_swizzle(r) within the row.  Conflict-free for the three ways a
// stage is accessed: whole rows (cp.async), rows 2i, 2i+1 at chunks 0..3 or 4..7, and rows 0, 2, 4, 6 (+1) at chunks 2i, 2i+1.
__device__ __forceinline__ int stage_swizzle(int row) { return (row & 6) ^ ((row & 1) << 2); }

template <int ST, int ET, bool ACC>
__global__ void __launch_bounds__(128, AdjointStream<ST, ET, ACC>::CTAS)
adjoint_stream_kernel(const __grid_constant__ StreamAdjointParams p) {
  using A = AdjointStream<ST, ET, ACC>;
  constexpr int NW = A::NW, STG = A::STG, NT = 32 * NW;
  extern __shared__ uint4 s_ring[];  // [warp][stage][experts, segments, old values][128 B]
  uint4* s_a = s_ring + NW * STG * A::STAGE / 16;            // [16 experts][16 segments][hi, lo][lane]
  float* s_dw = reinterpret_cast<float*>(s_a + ET * ST * 64);  // [16 ST][16 ET]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  pdl_launch();
  pdl_wait();
  for (int i = threadIdx.x; i < ET * ST * 32; i += NT) {
    const int ln = i & 31, m = (i >> 5) % ST, em = (i >> 5) / ST;
    a_fragment(ln, [&](int row, int col) {
      const int e = em * 16 + row, s = m * 16 + col;
      return (s < p.S && e < p.E) ? p.w[(size_t)s * p.E + e] : 0.f;
    }, s_a[((em * ST + m) * 2) * 32 + ln], s_a[((em * ST + m) * 2 + 1) * 32 + ln]);
  }
  for (int i = threadIdx.x; i < ST * ET * 256; i += NT) s_dw[i] = 0.f;
  // rows past the experts and segments are never loaded: they stay zero
  for (int i = threadIdx.x; i < NW * STG * A::STAGE / 16; i += NT) s_ring[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();

  const unsigned total = p.piece_end[2];
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(s_ring) + warp * (STG * A::STAGE);
  auto decode = [&](unsigned i, int& k, unsigned& r, unsigned& cb) {
    k = i < p.piece_end[0] ? 0 : (i < p.piece_end[1] ? 1 : 2);
    const unsigned l = i - (k == 0 ? 0u : p.piece_end[k - 1]);
    r = l / p.Cb[k];
    cb = l - r * p.Cb[k];
  };
  // starts the loads of piece i (if there is one); a group is committed either way, so that waits can count groups
  auto issue = [&](unsigned i, uint32_t stage) {
    if (i < total) {
      int k;
      unsigned r, cb;
      decode(i, k, r, cb);
      const int row0 = lane >> 3, c = lane & 7;   // four rows per instruction, eight lanes each
      const bf16* ds = p.dsrc[k] + ((size_t)(r >> 6) * p.Cb[k] + cb) * p.S * 4096 + (r & 63) * 64 + c * 8;
      const bool in = (int)(cb * 64 + c * 8) < p.C[k];   // columns past the matrix become zeros
      const uint32_t bytes = in ? 16u : 0u;
      const size_t off = (size_t)r * p.row_stride[k] + (in ? cb * 64 + c * 8 : 0);
      const uint32_t d0 = stage + row0 * 128 + ((c ^ stage_swizzle(row0)) << 4);
      const uint32_t d1 = stage + row0 * 128 + 512 + ((c ^ stage_swizzle(row0 + 4)) << 4);
#pragma unroll
      for (int j = 0; j < 4 * ET; ++j) {
        const int row = j * 4 + row0;
        if (row < p.E) cp_async_16b(((j & 1) ? d1 : d0) + (j >> 1) * 1024, p.wsrc[k] + off + (size_t)row * p.e_stride[k], bytes);
      }
#pragma unroll
      for (int j = 0; j < 4 * ST; ++j) {
        const int row = j * 4 + row0;
        if (row < p.S) cp_async_16b(((j & 1) ? d1 : d0) + (j >> 1) * 1024 + ET * 2048, ds + (size_t)row * 4096, 16u);
      }
      if (ACC) {
#pragma unroll
        for (int j = 0; j < 4 * ET; ++j) {
          const int row = j * 4 + row0;
          if (row < p.E)
            cp_async_16b(((j & 1) ? d1 : d0) + (j >> 1) * 1024 + (ET + ST) * 2048, p.ddst[k] + off + (size_t)row * p.e_stride[k], bytes);
        }
      }
    }
    cp_async_commit();
  };

  float d2[ST][2 * ET][4];
#pragma unroll
  for (int m = 0; m < ST; ++m)
#pragma unroll
    for (int n = 0; n < 2 * ET; ++n) d2[m][n][0] = d2[m][n][1] = d2[m][n][2] = d2[m][n][3] = 0.f;
  const unsigned first = blockIdx.x * NW + warp, step = gridDim.x * NW;
  const int stages = STG == 2 ? 2 : p.stages;
  for (int s = 0; s < stages - 1; ++s) issue(first + s * step, ring + s * A::STAGE);
  int cur = 0;
  for (unsigned i = first; i < total; i += step) {
    if (stages == 2) cp_async_wait<0>();
    else cp_async_wait<1>();
    __syncwarp();   // every lane's loads of this piece are visible, every lane is done with the stage refilled next
    issue(i + (stages - 1) * step, ring + (cur == 0 ? stages - 1 : cur - 1) * A::STAGE);
    const uint32_t st = ring + cur * A::STAGE;
    cur = cur + 1 == stages ? 0 : cur + 1;
    int k;
    unsigned r, cb;
    decode(i, k, r, cb);
    const uint32_t row_g = st + g * 128, c0 = (uint32_t)(t ^ stage_swizzle(g)) << 4, c1 = c0 ^ 64u;
    // dw += dWbar . W^T over these 64 parameters
#pragma unroll
    for (int m = 0; m < ST; ++m) {
      uint4 v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = lds_16b(row_g + (ET + m) * 2048 + (q & 1) * 1024 + ((q >> 1) ? c1 : c0));
#pragma unroll
      for (int n = 0; n < 2 * ET; ++n) {
        const uint4 w0 = lds_16b(row_g + n * 1024 + c0), w1 = lds_16b(row_g + n * 1024 + c1);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          mma_bf16_16x8x16(d2[m][n], make_uint4(word_of(v[0], q), word_of(v[1], q), word_of(v[2], q), word_of(v[3], q)),
                           word_of(w0, q), word_of(w1, q));
      }
    }
    // dW = (w_hi + w_lo)^T dWbar
    float acc[ET][8][4];
#pragma unroll
    for (int em = 0; em < ET; ++em)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[em][j][0] = acc[em][j][1] = acc[em][j][2] = acc[em][j][3] = 0.f;
#pragma unroll
    for (int m = 0; m < ST; ++m) {
      const uint32_t rows = st + (ET + m) * 2048 + t * 256;
      const uint32_t x0 = (uint32_t)(g ^ stage_swizzle(2 * t)) << 4, x1 = (uint32_t)(g ^ stage_swizzle(2 * t + 1)) << 4;
      const uint4 v[4] = {lds_16b(rows + x0), lds_16b(rows + 128 + x1), lds_16b(rows + 1024 + x0), lds_16b(rows + 1152 + x1)};
      uint32_t b[8][2];
      b_fragments(v, b);
#pragma unroll
      for (int em = 0; em < ET; ++em) {
        const uint4 hi = s_a[((em * ST + m) * 2) * 32 + lane], lo = s_a[((em * ST + m) * 2 + 1) * 32 + lane];
#pragma unroll
        for (int j = 0; j < 8; ++j) mma_bf16_16x8x16(acc[em][j], hi, b[j][0], b[j][1]);
#pragma unroll
        for (int j = 0; j < 8; ++j) mma_bf16_16x8x16(acc[em][j], lo, b[j][0], b[j][1]);
      }
    }
    bf16* dst = p.ddst[k] + (size_t)r * p.row_stride[k] + cb * 64 + t * 16;
    const int left = p.C[k] - (int)cb * 64 - t * 16;   // columns from this lane's first on
#pragma unroll
    for (int em = 0; em < ET; ++em)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int e = em * 16 + g + h * 8;
        if (e >= p.E || left <= 0) continue;
        uint4 o[2];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const int c = 2 * h + half;
          uint4 old = make_uint4(0u, 0u, 0u, 0u);
          if (ACC) old = lds_16b(row_g + (ET + ST + em) * 2048 + h * 1024 + (((2 * t + half) ^ stage_swizzle(g)) << 4));
          uint32_t w[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float a0 = acc[em][2 * q][c], a1 = acc[em][2 * q + 1][c];
            if (ACC) {
              const uint32_t ow = word_of(old, q);
              const float2 of = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&ow));
              a0 += of.x;
              a1 += of.y;
            }
            w[q] = pack_pair(a0, a1);
          }
          o[half] = make_uint4(w[0], w[1], w[2], w[3]);
        }
        bf16* q = dst + (size_t)e * p.e_stride[k];
        if (left >= 16 && (reinterpret_cast<uintptr_t>(q) & 31) == 0) {
          st_32b(q, o[0], o[1]);
        } else {
          *reinterpret_cast<uint4*>(q) = o[0];
          if (left > 8) *reinterpret_cast<uint4*>(q + 8) = o[1];
        }
      }
  }
  cp_async_wait<0>();
  for (int w = 0; w < NW; ++w) {
    if (warp == w) {
#pragma unroll
      for (int m = 0; m < ST; ++m)
#pragma unroll
        for (int n = 0; n < 2 * ET; ++n)
#pragma unroll
          for (int c = 0; c < 4; ++c)
            s_dw[(m * 16 + g + (c >> 1) * 8) * (16 * ET) + n * 8 + 2 * t + (c & 1)] += d2[m][n][c];
    }
    __syncthreads();
  }
  float* slab = p.dw_partial + (size_t)blockIdx.x * p.S * p.E;
  for (int i = threadIdx.x; i < p.S * p.E; i += NT) {
    const float v = s_dw[(i / p.E) * (16 * ET) + i % p.E];
    slab[i] = p.slab_add ? slab[i] + v : v;
  }
}

}  // namespace lory
