// Fused per-ray pass of one GO-Surf step with the decoders on the tcgen05 tensor cores.
//
// What it computes (same as the paper's step, Sec. 3.1-3.4): multi-level trilinear gather,
// geometry and colour decoders, NeuS compositing, the rgb / depth / sdf / free-space losses
// and, in the same pass, their reverse mode down to every grid feature and decoder weight.
//
// Mapping.  A "group" of 8 warps owns one M = 128 tensor-core tile, two threads per tile row:
// warps w and w + 4 of the group render one ray, and its 32-sample chunk j fills tile rows
// 32w..32w+31, which are exactly the tensor-memory lanes that warps w (mod 4) may read.  The
// lower half's threads hold the first half of a layer's units and grid levels 0 and 3, the upper
// half's the other units and levels 1 and 2.  Each decoder layer of a chunk is one MMA phase:
// the threads write their sample's activation row into the tensor-memory A operand, one thread
// issues the MMA(s) against the shared-memory weight tile (K-major, no swizzle), the result lands
// in tensor memory and every thread reads its columns back with tcgen05.ld.  Forward: 3 phases
// per chunk (the colour output layer on CUDA cores).  Reverse: the stored activations (or the
// forward phases again), then 3 adjoint phases; the decoder weight gradients are products over
// the tile's samples, accumulated in tensor memory.  FP32 form: each operand is split into three
// bfloat16 parts and the six leading part products are accumulated in FP32 (FP32-grade accuracy
// on BF16 tensor cores).  Compositing and its adjoint are warp scans over the ray's chunks, by
// the lower half; grid gradients are scattered with 16-byte vector reductions.
//
// What bounds it: the L1 / shared-memory data path (62 % busy over the whole kernel at 8192 x 96
// before the operands moved to tensor memory, in bursts: the phases of a group load it in turn)
// and each group's serial chain; DRAM and the tensor cores are below 20 %.  Hence two threads per
// row (half the chain at the same shared and tensor memory), the phases' A operands in tensor
// memory, two groups of 128 registers (three at 80 registers measured slower with a reverse pass: 607
// against 476 us, at the same data path), the weight gradients' part pairs in as few products as the
// tile layout allows.  What does not fit 128 registers goes to local memory, through the same data
// path: with a reverse pass 62 bytes stored and 168 loaded a thread at three chunks, 230 and 412 at
// five (the BF16 form 44 and 96 at three); forward only with two groups 0 to 8, with three at 80
// registers 68 and 76 at three chunks, 124 and 140 at five.  Render call, 8192 x 96, stored: one thread
// per row and three groups 523 us, two threads and two groups 476 us, A operands in tensor memory 451 us;
// forward only, 8192 x 132: 251, 223, 195 us, and 187 us with three groups (forward_groups says when).
#pragma once
#include "gs_internal.h"
#include <cuda_bf16.h>

#include "gs_tc.cuh"

namespace gs {

// Operand precisions.  Every operand is split into `planes` bfloat16 parts
// x = x0 + x1 + x2 (x0 = bf16(x), x1 = bf16(x - x0), x2 = bf16(x - x0 - x1): 24 significant
// bits) and a product is the sum of the part products with i + j < planes, accumulated in
// FP32 by the tensor core: 6 MMAs per K step give FP32-grade products (the dropped terms
// are below 2^-24 relative), 1 MMA per step is the plain BF16 form.
struct PrecBF16x3 {
  static constexpr int es = 2;      // bytes per operand element
  static constexpr int kmma = 16;   // K per MMA instruction
  static constexpr int planes = 3;
};
struct PrecBF16 {
  static constexpr int es = 2;
  static constexpr int kmma = 16;
  static constexpr int planes = 1;
};

constexpr int kTiles = 6;
// weight (B) tiles: {N, K} of the decoder contractions on the tensor core
//   0 W1  32x16 | 1 W2 16x32 | 2 W3 32x16 (col 15 zero)
//   3 W3^T 16x32 (row 15 zero) | 4 W2^T 32x16 | 5 W1^T 16x32
__host__ __device__ constexpr int wN(int i) { return (i == 0 || i == 2 || i == 4) ? 32 : 16; }
__host__ __device__ constexpr int wK(int i) { return (i == 0 || i == 2 || i == 4) ? 16 : 32; }
template <class P>
__host__ __device__ constexpr uint32_t wBytes(int i) { return (uint32_t)(wN(i) * wK(i) * P::es); }
template <class P>
__host__ __device__ constexpr uint32_t wOff(int i) {
  uint32_t o = 0;
  for (int k = 0; k < i; ++k) o += wBytes<P>(k);
  return o;
}
template <class P>
__host__ __device__ constexpr uint32_t wTotal() { return wOff<P>(kTiles); }

// tensor-memory columns of one group: the phases' results (N = 32 in cX, N = 16 in cY; each is
// read back before the next phase that writes its columns), then the decoder weight gradients,
// accumulated over all of the group's tiles (M = 64 layout: row m in lane 32 (m / 16) + m % 16)
// and the phases' A operand: part p of a K-column row in columns cA + p K / 2 ..
// (a forward-only call has no weight gradients: its operand follows the results)
constexpr uint32_t cX = 0, cY = 32, cW1 = 48, cW2 = 72, cW3 = 112;
template <bool BWD>
constexpr uint32_t cA = BWD ? 128 : 48;
template <bool BWD>
constexpr uint32_t kGroupCols = cA<BWD> + 48;
// tcgen05.alloc takes a power of two >= 32 columns
__host__ __device__ constexpr uint32_t tmem_cols(uint32_t columns) {
  uint32_t c = 32;
  while (c < columns) c <<= 1;
  return c;
}

constexpr int kGroupThreads = 128;  // a tile group of one thread per tile row
constexpr int kTileThreads = 256;   // the compact render kernel's tile group: two threads per tile row
constexpr int kSums = 8;            // running sums of a compositing warp: 4 losses, kappa, the colour seeds
constexpr uint32_t kMbarLimit = 1u << 20;  // bounded MMA-completion wait (tries of up to 2 us: ~2 s)

// Shared memory per tile group: adjoint tile | partner planes of the weight-gradient products (an
// activation tile of up to 40 columns; that widest one goes with a 16-column adjoint tile, which
// fills half of its space, and starts there) | (BF16 form) the colour layer's staging rows |
// barriers.  The phases' own A operands are in tensor memory: from shared memory every product
// read its 4 KB again, and the shared-memory data path, which the loads and stores of both
// caches go through too, is what binds this kernel.
// The adjoint tile holds the two leading parts side by side (part p of a K-column tile takes the
// 16-byte column chunks p K / 8 .. of a row): read MN-major, one M = 64 product then takes both
// parts of a 32-unit adjoint as 64 rows, two products per 16 samples (one per part of the
// partner) where the part pairs by themselves took three.  An M = 64 read of a narrower tile runs
// into the next rows (or what follows the tile), for D rows that nobody reads.
template <class P>
struct TcLayout {
  static constexpr uint32_t a_bytes = 128u * 32u * P::es;  // one part, K = 32
  static constexpr int side = P::planes < 2 ? 1 : 2;       // parts side by side
  static constexpr uint32_t b_bytes = 128u * 40u * P::es;
  static constexpr int b_planes = P::planes < 2 ? P::planes : 2;
  static constexpr uint32_t b_off = a_bytes * side;                            // partner tile
  static constexpr uint32_t b_wide = b_off - (side > 1 ? a_bytes : 0u);        // the 40-column one
  static constexpr uint32_t stage_off = b_off + (b_bytes * 3 / 5) * b_planes;  // after 24 columns
  static constexpr uint32_t stage_bytes = P::planes < 2 ? 128u * 32u * 4u : 0u;
  static constexpr uint32_t tiles = stage_off + stage_bytes;
  static constexpr uint32_t runs = 8u * 33u * 36u * 4u;  // the run reduction's rows over the whole space
  static constexpr uint32_t bar_off = ((tiles > runs ? tiles : runs) + 127u) / 128u * 128u;
  static constexpr uint32_t group_bytes = bar_off + 128;
  static_assert(b_wide + b_bytes * b_planes <= bar_off, "the wide partner tile fits");
  static constexpr uint32_t row_stride(int K) { return (uint32_t)side * (uint32_t)K * 16u; }  // per 8 rows
};

// Lanes come here from polls and branches of their own (a phase's one polling lane, lane 0's sums);
// bar.sync is an .aligned instruction, which a whole warp has to execute together.
template <int T = kGroupThreads>
__device__ __forceinline__ void group_sync(int g) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "n"(T) : "memory");
}

// ---- operand rows ---------------------------------------------------------------------
// bf16 parts of x (round to nearest even; the differences are exact in binary32)
template <int PL>
__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16 (&p)[PL]) {
  float r = x;
#pragma unroll
  for (int i = 0; i < PL; ++i) {
    p[i] = __float2bfloat16_rn(r);
    r = r - __bfloat162float(p[i]);
  }
}

// r -= the two bfloat16 values in w, exactly (they are r's leading bits): one packed operation
__device__ __forceinline__ void sub_parts(float2& r, uint32_t w) {
  const float2 h = make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
  const float2 m1 = make_float2(-1.0f, -1.0f);
  asm("fma.rn.f32x2 %0, %1, %2, %0;"
      : "+l"(reinterpret_cast<uint64_t&>(r))
      : "l"(reinterpret_cast<const uint64_t&>(h)), "l"(reinterpret_cast<const uint64_t&>(m1)));
}
// the NPL bf16 parts of 2 W consecutive values, W words a part; pairs of values are rounded
// together (one cvt.rn.bf16x2 per pair and part)
template <int NPL, int W>
__device__ __forceinline__ void split_words(const float* v, uint32_t (&w)[NPL][W]) {
#pragma unroll
  for (int q = 0; q < W; ++q) {
    float2 r = make_float2(v[2 * q], v[2 * q + 1]);
#pragma unroll
    for (int pl = 0; pl < NPL; ++pl) {
      const __nv_bfloat162 b = __floats2bfloat162_rn(r.x, r.y);
      w[pl][q] = *reinterpret_cast<const uint32_t*>(&b);
      if (pl + 1 < NPL) sub_parts(r, w[pl][q]);
    }
  }
}
// 8 values as 16-byte chunk `c` of row `row` of a K-major no-swizzle tile of K columns
template <int NPL, int K, uint32_t PLANE_BYTES>
__device__ __forceinline__ void store_chunk(uint8_t* planes, int row, int c, const float* v) {
  constexpr uint32_t sbo = (uint32_t)(K * 2 / 16) * 128u;
  uint32_t w[NPL][4];
  split_words<NPL, 4>(v, w);
  const uint32_t off = tc::core_offset((uint32_t)row, (uint32_t)c, 128u, sbo);
#pragma unroll
  for (int pl = 0; pl < NPL; ++pl)
    *reinterpret_cast<uint4*>(planes + pl * PLANE_BYTES + off) = make_uint4(w[pl][0], w[pl][1], w[pl][2], w[pl][3]);
}
// 4 values as the columns 4 q .. 4 q + 3 of the row
template <int NPL, int K, uint32_t PLANE_BYTES>
__device__ __forceinline__ void store_quarter(uint8_t* planes, int row, int q, const float4& v4) {
  constexpr uint32_t sbo = (uint32_t)(K * 2 / 16) * 128u;
  const float v[4] = {v4.x, v4.y, v4.z, v4.w};
  uint32_t w[NPL][2];
  split_words<NPL, 2>(v, w);
  const uint32_t off = tc::core_offset((uint32_t)row, (uint32_t)(q >> 1), 128u, sbo) + (uint32_t)(q & 1) * 8u;
#pragma unroll
  for (int pl = 0; pl < NPL; ++pl) *reinterpret_cast<uint2*>(planes + pl * PLANE_BYTES + off) = make_uint2(w[pl][0], w[pl][1]);
}
// The compact kernel's operand rows: 2 W values of a K-column row from column 2 w0 on, all parts into
// tensor memory (ta: the part-0 column of the thread's lane) and, with TILE, the leading parts
// into the adjoint tile as well (whole 16-byte chunks: W a multiple of 4)
template <class P, int K, bool TILE, int W>
__device__ __forceinline__ void put_operand(uint32_t ta, uint8_t* tile, int row, int w0, const float* v) {
  using L = TcLayout<P>;
  uint32_t w[P::planes][W];
  split_words<P::planes, W>(v, w);
#pragma unroll
  for (int pl = 0; pl < P::planes; ++pl) tc::tmem_st(ta + (uint32_t)(pl * (K / 2) + w0), w[pl]);
  if constexpr (TILE) {
#pragma unroll
    for (int pl = 0; pl < L::side; ++pl)
#pragma unroll
      for (int c = 0; c < W / 4; ++c)
        *reinterpret_cast<uint4*>(tile + tc::core_offset((uint32_t)row, (uint32_t)(pl * (K / 8) + w0 / 4 + c), 128u,
                                                         L::row_stride(K))) =
            make_uint4(w[pl][4 * c], w[pl][4 * c + 1], w[pl][4 * c + 2], w[pl][4 * c + 3]);
  }
}
// K values as row `row`, one plane per bf16 part
template <int NPL, int K, uint32_t PLANE_BYTES>
__device__ __forceinline__ void store_row_planes(uint8_t* planes, int row, const float* v) {
#pragma unroll
  for (int c = 0; c < K / 8; ++c) store_chunk<NPL, K, PLANE_BYTES>(planes, row, c, v + 8 * c);
}

// one element of a weight tile (planes `wplane` bytes apart)
template <class P>
__device__ __forceinline__ void store_w(uint8_t* planes, uint32_t wplane, int K, int n, int k, float v) {
  const uint32_t sbo = (uint32_t)(K * P::es / 16) * 128u;
  const uint32_t off = tc::core_offset((uint32_t)n, (uint32_t)(k * P::es / 16), 128u, sbo) + (uint32_t)(k * P::es % 16);
  __nv_bfloat16 e[P::planes];
  split_bf16<P::planes>(v, e);
#pragma unroll
  for (int pl = 0; pl < P::planes; ++pl) *reinterpret_cast<__nv_bfloat16*>(planes + pl * wplane + off) = e[pl];
}

// Decoder weight gradients on the tensor core: D[64][N] (+)= sum over the tile's 128 samples
// of A[s][m] B[s][n], both operands read MN-major from the sample-row tiles the phases write
// (core-matrix stride along K = the tile's row-group stride, along M/N = 128 bytes).  Part
// products i + j < SUM, i < APL, j < BPL, smallest first; `acc` false on the first tile.
template <int APL, int BPL, int SUM, int N>
__device__ __forceinline__ void issue_mma_dw(uint32_t d, uint32_t a0, uint32_t a_plane, uint32_t a_kstride,
                                             uint32_t b0, uint32_t b_plane, uint32_t b_kstride, bool acc) {
  constexpr uint32_t idesc = tc::instr_desc(64, N) | (1u << 15) | (1u << 16);
  uint32_t alo = tc::desc_lo(a0, a_kstride), blo = tc::desc_lo(b0, b_kstride);
#pragma unroll 2
  for (int s = 0; s < 8; ++s) {  // K = 128 samples, 16 per MMA
#pragma unroll
    for (int sum = SUM - 1; sum >= 0; --sum)
#pragma unroll
      for (int i = 0; i <= sum; ++i) {
        const int j = sum - i;
        if (i >= APL || j >= BPL) continue;
        tc::mma_bf16(d, tc::desc_of(alo + ((i * a_plane) >> 4), tc::desc_hi(128u)),
                     tc::desc_of(blo + ((j * b_plane) >> 4), tc::desc_hi(128u)), idesc, acc ? 1u : 0u);
        acc = true;
      }
    alo += (2u * a_kstride) >> 4;
    blo += (2u * b_kstride) >> 4;
  }
}

// The compact kernel's phase product: D[128][N] = A[128][K] B[N][K]^T, A in tensor memory.  The operand
// descriptors of a series are the first one's plus constants: built from their addresses each, the
// issuing thread spent about 15 instructions per MMA, which the whole group waits for.
template <class P, int N, int K>
__device__ __forceinline__ void tile_mma(uint32_t d, uint32_t ta, uint32_t b0, uint32_t wplane) {
  constexpr uint32_t idesc = tc::instr_desc(128, N);
  const uint32_t blo = tc::desc_lo(b0, 128u);
  bool first = true;
#pragma unroll
  for (int s = 0; s < K / P::kmma; ++s) {
    // smallest part products first
#pragma unroll
    for (int sum = P::planes - 1; sum >= 0; --sum)
#pragma unroll
      for (int i = 0; i <= sum; ++i) {
        const uint32_t bo = (uint32_t)(sum - i) * wplane + (uint32_t)s * 256u;
        tc::mma_bf16_ta(d, ta + (uint32_t)(i * (K / 2) + s * 8), tc::desc_of(blo + (bo >> 4), tc::desc_hi(K * 16u)), idesc,
                        first ? 0u : 1u);
        first = false;
      }
  }
}
// Its weight-gradient product: D[64][N] (+)= sum over the tile's 128 samples of A[s][m] B[s][n], both
// operands read MN-major; m over the adjoint tile's KA columns of part 0, then of part 1 (rows KA ..
// 2 KA - 1, added to the first KA at the end), n over the partner tile's N columns, one product
// per partner part.  `acc` false on the first tile.
template <class P, int N, int KA>
__device__ __forceinline__ void tile_mma_dw(uint32_t d, uint32_t a0, uint32_t b0, bool acc) {
  using L = TcLayout<P>;
  constexpr uint32_t idesc = tc::instr_desc(64, N) | (1u << 15) | (1u << 16);
  constexpr uint32_t ra = L::row_stride(KA), rb = N * 16u;
  const uint32_t alo = tc::desc_lo(a0, ra), blo = tc::desc_lo(b0, rb);
#pragma unroll
  for (int s = 0; s < 8; ++s)  // K = 128 samples, 16 per product
#pragma unroll
    for (int j = L::b_planes - 1; j >= 0; --j) {
      tc::mma_bf16(d, tc::desc_of(alo + ((s * 2u * ra) >> 4), tc::desc_hi(128u)),
                   tc::desc_of(blo + ((s * 2u * rb + j * L::b_bytes) >> 4), tc::desc_hi(128u)), idesc,
                   acc || s > 0 || j < L::b_planes - 1 ? 1u : 0u);
    }
}

// per-group MMA machinery
struct Group {
  uint64_t* mbar;     // completion of the phase MMAs (issued by a lane of the group's first warp)
  uint64_t* mbar_dw;  // completion of the weight-gradient MMAs (a lane of its second warp)
  int* abort;
  uint32_t tcol;      // tensor-memory address of this group's column 0
  uint32_t phase;     // parity of the next completion on mbar
  uint32_t phase_dw;  // ... on mbar_dw
  bool dw_pending;    // weight-gradient MMAs may still read the operand tiles
  int g, gt;
};

// ---- the compact render kernel's tile groups ------------------------------------------------
// A tile group's barriers: the phase's products done, its weight-gradient products done; and whether a
// bounded wait ran out
struct TileBars {
  uint64_t done, dw;
  int abort;
};
template <class P, int TYPE, bool BWD>  // 0..2 the forward layers, 3..5 the adjoints b3, b2, b1
__device__ __forceinline__ void issue_phase(uint32_t tcol, uint32_t sw) {
  constexpr uint32_t wplane = wTotal<P>();
  if constexpr (TYPE == 0) tile_mma<P, 32, 16>(tcol + cX, tcol + cA<BWD>, sw + wOff<P>(0), wplane);
  if constexpr (TYPE == 1) tile_mma<P, 16, 32>(tcol + cY, tcol + cA<BWD>, sw + wOff<P>(1), wplane);
  if constexpr (TYPE == 2) tile_mma<P, 32, 16>(tcol + cX, tcol + cA<BWD>, sw + wOff<P>(2), wplane);
  if constexpr (TYPE == 3) tile_mma<P, 16, 32>(tcol + cY, tcol + cA<BWD>, sw + wOff<P>(3), wplane);
  if constexpr (TYPE == 4) tile_mma<P, 32, 16>(tcol + cX, tcol + cA<BWD>, sw + wOff<P>(4), wplane);
  if constexpr (TYPE == 5) tile_mma<P, 16, 32>(tcol + cY, tcol + cA<BWD>, sw + wOff<P>(5), wplane);
}
template <class P, int TYPE>
__device__ __forceinline__ void issue_phase_dw(uint32_t tcol, uint32_t sa, bool acc) {
  const uint32_t sb = sa + (TYPE == 4 ? TcLayout<P>::b_wide : TcLayout<P>::b_off);
  if constexpr (TYPE == 3) tile_mma_dw<P, 16, 32>(tcol + cW3, sa, sb, acc);
  if constexpr (TYPE == 4) tile_mma_dw<P, 40, 16>(tcol + cW2, sa, sb, acc);
  if constexpr (TYPE == 5) tile_mma_dw<P, 24, 32>(tcol + cW1, sa, sb, acc);
}

// what a thread of a group tracks of its barriers
struct Tile {
  TileBars* bars;
  int g, w8;                // the group, this thread's warp in it (uniform)
  uint32_t ph_done, ph_dw;  // parities of the next completions
  bool dw_pending;          // weight-gradient products may still read the tiles
};
// A bounded wait of the group ran out (every thread reads the same between two group barriers): the
// group leaves its loop at the next phase_wait.
__device__ __forceinline__ bool failed(const Tile& T) { return *reinterpret_cast<volatile int*>(&T.bars->abort) != 0; }
// Operand rows of this warp written -> once all warps have met, one thread of warp 0 issues the
// phase's products and (adjoint phases) one of warp 4 the weight-gradient products that
// read the same tiles.
template <class P, int TYPE, bool BWD>
__device__ __forceinline__ void phase_issue(Tile& T, uint32_t tcol, uint32_t sa, uint32_t sw, bool dw_acc) {
  tc::tmem_st_wait();
  if (TYPE >= 3) tc::fence_smem_async();
  tc::fence_before_sync();
  group_sync<kTileThreads>(T.g);
  tc::fence_after_sync();
  if (T.w8 == 0) {
    if (tc::elect_one()) {
      issue_phase<P, TYPE, BWD>(tcol, sw);
      tc::mma_commit(&T.bars->done);
    }
    __syncwarp();
  } else if (TYPE >= 3 && T.w8 == 4) {
    if (tc::elect_one()) {
      issue_phase_dw<P, TYPE>(tcol, sa, dw_acc);
      tc::mma_commit(&T.bars->dw);
    }
    __syncwarp();
  }
  if (TYPE >= 3) T.dw_pending = true;
}
// a thread of the group waits for the products (bounded) while the others park on the hardware
// barrier; false (for every thread) if they never complete
__device__ __forceinline__ bool phase_wait(Tile& T) {
  if (T.w8 == 1 && tc::elect_one() && !tc::mbar_wait(&T.bars->done, T.ph_done, kMbarLimit))
    atomicOr(&T.bars->abort, 1);
  T.ph_done ^= 1u;
  group_sync<kTileThreads>(T.g);
  tc::fence_after_sync();
  return !failed(T);
}
// no weight-gradient product reads the tiles.  Every lane polls by itself and may leave at another
// try than its neighbours; the warp goes on together, as the tcgen05 instructions that follow require.
__device__ __forceinline__ void tiles_free(Tile& T) {
  if (T.dw_pending) {
    if (!tc::mbar_wait(&T.bars->dw, T.ph_dw, kMbarLimit)) atomicOr(&T.bars->abort, 1);
    T.ph_dw ^= 1u;
    T.dw_pending = false;
    __syncwarp();
    tc::fence_after_sync();
  }
}
// The end of a group's work, called by all of its threads: no product of the group is in flight any
// more.  After a bounded wait that ran out, the status word takes `bit` and one thread waits once
// more (bounded) for the products that may still run: what follows reuses the tiles' space and
// releases the tensor memory that they read and write.  The CTA meets after this call and before
// either.  false if a wait ran out.
// Weight-gradient products may be owed twice: the wait that ran out before a phase, and that phase's
// own.  Then the first has parity ph_dw (the parity flips at every wait) and the second the other one;
// owed once, only the other one blocks.  What is not owed runs to its limit.
__device__ __forceinline__ bool tile_end(Tile& T, int* status, int bit) {
  tiles_free(T);
  group_sync<kTileThreads>(T.g);
  if (!failed(T)) return true;
  if (T.w8 == 0 && tc::elect_one()) {
    atomicOr(status, bit);
    tc::mbar_wait(&T.bars->done, T.ph_done ^ 1u, kMbarLimit);
    tc::mbar_wait(&T.bars->dw, T.ph_dw, kMbarLimit);
    tc::mbar_wait(&T.bars->dw, T.ph_dw ^ 1u, kMbarLimit);
  }
  __syncwarp();
  return false;
}

// every thread of the group: bounded wait until the weight-gradient MMAs are done with the tiles
__device__ __forceinline__ void dw_wait(Group& G) {
  if (!G.dw_pending) return;
  if (!tc::mbar_wait(G.mbar_dw, G.phase_dw, kMbarLimit)) *reinterpret_cast<volatile int*>(G.abort) = 1;
  G.phase_dw ^= 1u;
  G.dw_pending = false;
  __syncwarp();
  tc::fence_after_sync();
}
// the issuing thread waits for the MMA (bounded) while the other threads of the group park on
// the hardware barrier; false (for every thread) if it never completed
template <int T = kGroupThreads>
__device__ __forceinline__ bool mma_phase_wait(Group& G) {
  if (G.gt == 0 && !tc::mbar_wait(G.mbar, G.phase, kMbarLimit)) *reinterpret_cast<volatile int*>(G.abort) = 1;
  G.phase ^= 1u;
  group_sync<T>(G.g);
  tc::fence_after_sync();
  return *reinterpret_cast<volatile int*>(G.abort) == 0;
}

__device__ __forceinline__ uint32_t lane_addr(const Group& G, uint32_t col, int warp_g) {
  return G.tcol + col + ((uint32_t)(32 * warp_g) << 16);
}

// ---- gather / scatter -------------------------------------------------------------------
// The 8 corners of one cell at (runtime) level l, summed in corner order k = 4 bx + 2 by + bz:
// a float4 of features from the FP32 grid (`bf16` nullptr) or its bfloat16 copy
__device__ __forceinline__ float4 level_features(const GridDesc& g, const float* __restrict__ theta, int l,
                                                 const float x[3]) {
  const Cell c = locate(g, l, x);
  float w[8];
  corner_weights(c.f, w);
  const long long nx = g.dims[l][0], nxy = nx * g.dims[l][1];
  const float4* p = reinterpret_cast<const float4*>(theta + g.off[l]) + c.vtx;
  const float4 *p1 = p + nxy, *p2 = p + nx, *p3 = p2 + nxy;
  const float4 v[8] = {__ldg(p),     __ldg(p1),     __ldg(p2),     __ldg(p3),
                       __ldg(p + 1), __ldg(p1 + 1), __ldg(p2 + 1), __ldg(p3 + 1)};
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int k = 0; k < 8; ++k) f4fma(s, w[k], v[k]);
  return s;
}
__device__ __forceinline__ float4 level_features_bf16(const GridDesc& g, const uint16_t* __restrict__ copy, int l,
                                                      const float x[3]) {
  const Cell c = locate(g, l, x);
  float w[8];
  corner_weights(c.f, w);
  const long long nx = g.dims[l][0], nxy = nx * g.dims[l][1];
  const uint2* p = reinterpret_cast<const uint2*>(copy + g.off[l]) + c.vtx;
  const uint2 *p1 = p + nxy, *p2 = p + nx, *p3 = p2 + nxy;
  const uint2 u[8] = {__ldg(p),     __ldg(p1),     __ldg(p2),     __ldg(p3),
                      __ldg(p + 1), __ldg(p1 + 1), __ldg(p2 + 1), __ldg(p3 + 1)};
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int k = 0; k < 8; ++k)
    f4fma(s, w[k], make_float4(__uint_as_float(u[k].x << 16), __uint_as_float(u[k].x & 0xFFFF0000u),
                               __uint_as_float(u[k].y << 16), __uint_as_float(u[k].y & 0xFFFF0000u)));
  return s;
}

// The finest level's corners by plain loads, all eight in flight: lane i takes them in the order
// i, i + 1, .. (mod 8; corner c = vertex (x + (c & 1), y + (c >> 1 & 1), z + (c >> 2)))
struct FineCorners {
  float4 v[8];
  float f[3];
};
__device__ __forceinline__ void fine_corners_load(const GridDesc& g, const float* __restrict__ theta, const float x[3],
                                                  FineCorners& q) {
  constexpr int l = kLevels - 1;
  const Cell c = locate(g, l, x);
  const int lane = threadIdx.x & 31;
  const long long nx = g.dims[l][0], nxy = nx * g.dims[l][1];
  const float4* base = reinterpret_cast<const float4*>(theta + g.off[l]) + c.vtx;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int cc = (k + lane) & 7;
    q.v[k] = __ldg(base + (cc & 1) + ((cc & 2) ? nx : 0) + ((cc & 4) ? nxy : 0));
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) q.f[a] = c.f[a];
}
__device__ __forceinline__ float4 fine_corners_sum(const FineCorners& q) {
  const int lane = threadIdx.x & 31;
  const float f0 = q.f[0], f1 = q.f[1], f2 = q.f[2];
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int cc = (k + lane) & 7;
    const float w = (((cc & 1) ? f0 : 1.0f - f0) * ((cc & 2) ? f1 : 1.0f - f1)) * ((cc & 4) ? f2 : 1.0f - f2);
    f4fma(s, w, q.v[k]);
  }
  return s;
}

// staging floats per warp of the run-reduced scatter: 32 rows of 36 floats, then the 32 keys
constexpr int kScatterStage = 33 * 36;

// 16-byte vector reduction into global memory (fire and forget; no kernel here reads the result,
// so other memory operations may move across it)
__device__ __forceinline__ void red_add_f4(float4* p, float4 v) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
}

// The deferred Eikonal record of a sample (gs_batch.eik): at level l its corner c also receives
// q_l (a . dw_c/df), the grid part of the Eikonal gradient (Supp. Sec. 1), in the same reduction.
struct EikSeed {
  const float4* er;  // the sample's record in plane 0 (planes `es` float4 apart: q_l of the four levels, then a); nullptr: none
  long long es;
  float a[3];
  bool any;  // some lane of the warp has one
};
__device__ __forceinline__ EikSeed eik_seed(const float4* er, long long es) {
  EikSeed e{er, es, {0.f, 0.f, 0.f}, __any_sync(0xffffffffu, er != nullptr) != 0};
  if (er != nullptr) {
    const float4 a4 = __ldg(er + 4 * es);
    e.a[0] = a4.x;
    e.a[1] = a4.y;
    e.a[2] = a4.z;
  }
  return e;
}
// this level's q and a . dw_c/df (zeros without a record)
__device__ __forceinline__ float4 eik_level(const EikSeed& e, int l, const Cell& cc, float (&dd)[8]) {
  float4 q4 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int k = 0; k < 8; ++k) dd[k] = 0.f;
  if (e.any) {  // warp-uniform
    if (e.er != nullptr) q4 = __ldg(e.er + l * e.es);
    float dw[8][3];
    corner_weight_grads(cc.f, cc.clamped, dw);
#pragma unroll
    for (int k = 0; k < 8; ++k) dd[k] = e.a[0] * dw[k][0] + e.a[1] * dw[k][1] + e.a[2] * dw[k][2];
  }
  return q4;
}

// Adjoint of the gather at a coarse level (0 or 1): dtheta_l[corner] += w_c dz_l.  A warp's lanes
// hold consecutive samples of one ray, so the cells they fall in are visited monotonically and
// equal cells form contiguous (long) runs of lanes.  The 8 weighted corner vectors are summed
// over each run through shared memory: every lane stages its 32 values as a row, lane c walks the
// 32 rows summing component c (corner c / 4, feature c % 4), and at the end of each run the four
// features of a corner are gathered into one lane, which issues one 16-byte reduction (8 per
// run).  st: the warp's kScatterStage floats.
__device__ __forceinline__ void scatter_runs(const GridDesc& g, float* grad, int l, const float x[3], float4 g4,
                                             bool valid, float* st, const EikSeed& e) {
  const int lane = threadIdx.x & 31;
  const Cell cc = locate(g, l, x);
  float wc[8], dd[8];
  corner_weights(cc.f, wc);
  const float4 q4 = eik_level(e, l, cc, dd);
  float4* gl = reinterpret_cast<float4*>(grad + g.off[l]);
  const int key = valid ? (int)cc.vtx : -1;  // the coarse levels have fewer than 2^31 vertices
  const int next = __shfl_down_sync(0xffffffffu, key, 1);
  const unsigned ends = __ballot_sync(0xffffffffu, lane == 31 || next != key || key < 0);  // a run's last lane
  float* rw = st + lane * 36;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    float4 cv = f4scale(g4, wc[k]);
    if (e.any) f4fma(cv, dd[k], q4);
    *reinterpret_cast<float4*>(rw + 4 * k) = cv;
  }
  st[32 * 36 + lane] = __int_as_float(key);  // the keys after the rows
  __syncwarp();
  const long long coff = corner_offset(g, l, lane >> 2);
  float acc = 0.f;
#pragma unroll 1
  for (int i0 = 0; i0 < 32; i0 += 8) {
    float v[8];  // eight rows in flight
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = st[(i0 + q) * 36 + lane];
    const unsigned e8 = ends >> i0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      acc += v[q];
      if ((e8 >> q) & 1u) {  // uniform: the run holding row i0 + q ends there
        const float a1 = __shfl_down_sync(0xffffffffu, acc, 1), a2 = __shfl_down_sync(0xffffffffu, acc, 2),
                    a3 = __shfl_down_sync(0xffffffffu, acc, 3);
        const int ki = __float_as_int(st[32 * 36 + i0 + q]);
        if ((lane & 3) == 0 && ki >= 0) red_add_f4(gl + (long long)ki + coff, make_float4(acc, a1, a2, a3));
        acc = 0.f;
      }
    }
  }
  __syncwarp();
}

// The same at a fine level, where runs are short: every lane issues its 8 corners' 16-byte
// reductions directly (staging them there measured slower).  A zero vector adds nothing: samples
// whose dL/dz_l is exactly zero (saturated opacity and no active loss term) issue none.
// PAIRED: lane pairs (2i, 2i + 1) take turns on each other's samples so that in one reduction
// instruction the pair adds a cell's two x-neighbouring corners of one sample, 32 contiguous
// bytes (one sector when the cell's x index is even): a quarter fewer L2 reduction requests for
// 18 shuffles per lane.
template <bool PAIRED>
__device__ __forceinline__ void scatter_direct(const GridDesc& g, float* grad, int l, const float x[3], float4 g4,
                                               bool valid, const EikSeed& e) {
  const int lane = threadIdx.x & 31;
  const bool give = valid && (g4.x != 0.f || g4.y != 0.f || g4.z != 0.f || g4.w != 0.f || e.er != nullptr);
  if (!PAIRED && !give && !e.any) return;
  const Cell cc = locate(g, l, x);
  float wc[8], dd[8];
  corner_weights(cc.f, wc);
  const float4 q4 = eik_level(e, l, cc, dd);
  const long long nx = g.dims[l][0], nxy = nx * g.dims[l][1];
  float4* gl = reinterpret_cast<float4*>(grad + g.off[l]);
  if constexpr (PAIRED) {
    // corners k and k + 4 are the x-neighbours v and v + 1.  The even lane sends its upper
    // corner's vector and receives the odd lane's lower one; then the even lane adds the lower
    // corners (its own sample's, then its partner's) and the odd lane the upper ones (its
    // partner's, then its own), so each instruction covers one sample's pair.
    const bool odd = (lane & 1) != 0;
    const long long pv = __shfl_xor_sync(0xffffffffu, cc.vtx, 1);
    float4* q0 = gl + (odd ? pv : cc.vtx) + (odd ? 1 : 0);  // first instruction: the even lane's sample
    float4* q1 = gl + (odd ? cc.vtx : pv) + (odd ? 1 : 0);  // second: the odd lane's
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float4 lo4 = make_float4(0.f, 0.f, 0.f, 0.f), hi4 = lo4;
      if (give) {
        lo4 = f4scale(g4, wc[k]);
        hi4 = f4scale(g4, wc[k + 4]);
        if (e.any) {
          f4fma(lo4, dd[k], q4);
          f4fma(hi4, dd[k + 4], q4);
        }
      }
      const float4 snd = odd ? lo4 : hi4;
      float4 rcv;
      rcv.x = __shfl_xor_sync(0xffffffffu, snd.x, 1);
      rcv.y = __shfl_xor_sync(0xffffffffu, snd.y, 1);
      rcv.z = __shfl_xor_sync(0xffffffffu, snd.z, 1);
      rcv.w = __shfl_xor_sync(0xffffffffu, snd.w, 1);
      const long long off = ((k & 2) ? nx : 0) + ((k & 1) ? nxy : 0);  // the lower corner; the upper one is + 1
      const float4 c0 = odd ? rcv : lo4, c1 = odd ? hi4 : rcv;
      if (c0.x != 0.f || c0.y != 0.f || c0.z != 0.f || c0.w != 0.f) red_add_f4(q0 + off, c0);
      if (c1.x != 0.f || c1.y != 0.f || c1.z != 0.f || c1.w != 0.f) red_add_f4(q1 + off, c1);
    }
  } else if (give) {
    float4* p0 = gl + cc.vtx;
    float4* const row[4] = {p0, p0 + nxy, p0 + nx, p0 + nx + nxy};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      float4 cv = f4scale(g4, wc[k]);
      if (e.any) f4fma(cv, dd[k], q4);
      red_add_f4(row[k & 3] + (k >> 2), cv);
    }
  }
}

template <int N>
__device__ __forceinline__ float pick_tc(const float (&arr)[N], int j) {
  float v = arr[0];
#pragma unroll
  for (int q = 1; q < N; ++q)
    if (q == j) v = arr[q];
  return v;
}

struct RenderTcArgs {
  GridDesc g;
  const float* theta;
  const uint16_t* theta_bf16;  // BF16 form: grid copy read by the gathers
  int R, N;
  const float *o, *r, *rgb, *D, *t;
  const uint8_t* cls;
  const int* counts;
  const float* dloss;
  float lam[5];
  float kappa_fs;
  float* grad;
  float* loss_part;
  float* mlp_part;
  float *rgb_hat, *d_hat, *wsum;
  int* status;      // device status word (bit 1: an MMA never completed)
  // Stored activations (store mode): written by every forward pass, read by every backward pass
  // in place of the gather and the recomputed decoder phases.  nullptr: recompute.
  float* store;
  float* w_out;  // [R][N] rendering weights, written by forward passes when not nullptr
  float* dz_out; // [R][N][16] dL/dz of every sample, written by backward passes when not nullptr
  // deferred Eikonal records ([5][R][N] float4 planes, eik_stride = R N) of the free-space
  // samples, added to their grid scatter by backward passes; nullptr: none
  const float4* eik;
  long long eik_stride;
};

// Stored activations of one chunk (n <= 32 consecutive samples of a ray from sample s on): 25
// planes of n float4, one after the other from float4 index 25 s on, lane i's four fields in
// element i of a plane, so a warp moves one contiguous line per plane and a chunk's 400 n bytes
// lie together (the planes of all samples apart, 12 MB each at 8192 x 96, a chunk touched 25
// pages).  Planes: z by level [4] | a1 = ReLU layer-1 output [8] | h [4] | a2 = ReLU layer-2
// output [8] | c, phi.
constexpr int kPz = 0, kPa1 = 4, kPh = 12, kPa2 = 16, kPc = 24;
static_assert((kPc + 1) * 4 == kStoreFloatsPerSample, "the store holds every field");
struct StoreRef {
  float4* p;  // this lane's element of plane 0
  int n;      // samples of the chunk
  __device__ __forceinline__ float4& operator[](int plane) const { return p[plane * n]; }
};
template <int NP>
__device__ __forceinline__ void put_planes(const StoreRef& s, int first, const float* v) {
#pragma unroll
  for (int q = 0; q < NP; ++q) s[first + q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}
template <int NP>
__device__ __forceinline__ void get_planes(const StoreRef& s, int first, bool get, float* v) {
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    const float4 u = get ? s[first + q] : make_float4(0.f, 0.f, 0.f, 0.f);
    v[4 * q] = u.x;
    v[4 * q + 1] = u.y;
    v[4 * q + 2] = u.z;
    v[4 * q + 3] = u.w;
  }
}

// NeuS compositing of one ray by one warp (lane = sample within the chunk), the losses of Sec.
// 3.2-3.4 and, with BWD, the adjoint down to each sample's seeds: dL/d(colour pre-activations)
// and dL/dphi into xch[128 j] of chunk j.  kc: the loss terms' scales (rgb, depth, sdf, fs) and
// the sharpness; sums: the warp's NS running sums (the four losses, dL/dkappa, the colour seeds';
// a ninth, the SDF seeds', is only the paper architecture's).
template <int NCH, bool FWD, bool BWD, int NS, class Args>
__device__ __forceinline__ void composite_ray(const Args& a, int ray, bool has_ray, const float (&tt)[NCH],
                                              const float (&ph)[NCH], const float (&col)[NCH][3],
                                              const int (&clv)[NCH], const float4& seen, const float* kc, float4* xch,
                                              float* sums) {
  const int lane = threadIdx.x & 31, N = a.N;
  const float D = seen.w, I[3] = {seen.x, seen.y, seen.z}, s_sharp = kc[4];
  float l_rgb = 0.f, l_d = 0.f, l_sdf = 0.f, l_fs = 0.f, g_kappa = 0.f, db4[3] = {0.f, 0.f, 0.f}, sum_d = 0.f;
  // ================= NeuS opacity, transmittance, weights (Sec. 3.2) =================
  float Ph[NCH], PhN[NCH], al[NCH], T[NCH], w[NCH];
#pragma unroll
  for (int j = 0; j < NCH; ++j) Ph[j] = (has_ray && 32 * j + lane < N) ? sigmoidf_(s_sharp * ph[j]) : 0.f;
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    float nx = __shfl_down_sync(0xffffffffu, Ph[j], 1);
    const float nx0 = (j + 1 < NCH) ? __shfl_sync(0xffffffffu, Ph[j + 1 < NCH ? j + 1 : j], 0) : 0.f;
    if (lane == 31) nx = nx0;
    PhN[j] = nx;
    float q = 0.f;
    if (has_ray && 32 * j + lane < N - 1) q = (Ph[j] - nx) / fmaxf(Ph[j], 1e-6f);
    al[j] = q > 0.f ? q : 0.f;
  }
  float carry = 1.0f;
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    float inc = 1.0f - al[j];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float y = __shfl_up_sync(0xffffffffu, inc, off);
      if (lane >= off) inc *= y;
    }
    float exc = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) exc = 1.0f;
    T[j] = carry * exc;
    carry *= __shfl_sync(0xffffffffu, inc, 31);
    w[j] = T[j] * al[j];
  }
  if (FWD && a.w_out != nullptr && has_ray) {
#pragma unroll
    for (int j = 0; j < NCH; ++j)
      if (32 * j + lane < N) a.w_out[(size_t)ray * N + 32 * j + lane] = w[j];
  }
  float ch[3] = {0.f, 0.f, 0.f}, dh = 0.f, ws = 0.f;
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
#pragma unroll
    for (int k = 0; k < 3; ++k) ch[k] = fmaf(w[j], col[j][k], ch[k]);
    dh = fmaf(w[j], tt[j], dh);
    ws += w[j];
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) ch[k] = warp_sum(ch[k]);
  dh = warp_sum(dh);
  ws = warp_sum(ws);
  if (FWD && has_ray) {
    if (lane == 0) {
      float e2 = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) e2 = fmaf(I[k] - ch[k], I[k] - ch[k], e2);
      l_rgb += e2;
      if (D > 0.f) l_d += fabsf(D - dh);
      if (a.rgb_hat) {
        a.rgb_hat[3 * ray] = ch[0];
        a.rgb_hat[3 * ray + 1] = ch[1];
        a.rgb_hat[3 * ray + 2] = ch[2];
      }
      if (a.d_hat) a.d_hat[ray] = dh;
      if (a.wsum) a.wsum[ray] = ws;
    }
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      const int si = 32 * j + lane;
      if (si >= N) continue;
      const int cl = clv[j];
      const float b = __fsub_rn(D, tt[j]);
      if (cl == CLS_TR) l_sdf += fabsf(ph[j] - b);
      else if (cl == CLS_FS) l_fs += fmaxf(fmaxf(0.f, expf(-a.kappa_fs * ph[j]) - 1.0f), ph[j] - b);
    }
  }
  if constexpr (BWD) {

  // ================= adjoint of compositing: dL/dalpha_k = T_k (e_k - U_k) =================
  float gc[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) gc[k] = has_ray ? kc[0] * (ch[k] - I[k]) : 0.f;
  const float gd = (has_ray && D > 0.f) ? kc[1] * ((dh > D) ? 1.f : (dh < D ? -1.f : 0.f)) : 0.f;
  float e[NCH], U[NCH];
#pragma unroll
  for (int j = 0; j < NCH; ++j) e[j] = gc[0] * col[j][0] + gc[1] * col[j][1] + gc[2] * col[j][2] + gd * tt[j];
  float cA = 0.f;
#pragma unroll
  for (int j = NCH - 1; j >= 0; --j) {
    float A = al[j] * e[j], B = 1.0f - al[j];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float A2 = __shfl_down_sync(0xffffffffu, A, off), B2 = __shfl_down_sync(0xffffffffu, B, off);
      if (lane + off < 32) {
        A = fmaf(B, A2, A);
        B *= B2;
      }
    }
    float eA = __shfl_down_sync(0xffffffffu, A, 1), eB = __shfl_down_sync(0xffffffffu, B, 1);
    if (lane == 31) {
      eA = 0.f;
      eB = 1.f;
    }
    U[j] = fmaf(eB, cA, eA);
    const float A0 = __shfl_sync(0xffffffffu, A, 0), B0 = __shfl_sync(0xffffffffu, B, 0);
    cA = fmaf(B0, cA, A0);
  }
  float dnext_prev = 0.f;
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    const int si = 32 * j + lane;
    const bool valid = has_ray && si < N;
    const float dal = T[j] * (e[j] - U[j]);
    float dself = 0.f, dnext = 0.f;
    if (valid && si < N - 1) {
      const float den = fmaxf(Ph[j], 1e-6f);
      if (Ph[j] - PhN[j] > 0.f) {
        dnext = -dal / den;
        dself = (Ph[j] > 1e-6f) ? dal * PhN[j] / (Ph[j] * Ph[j]) : dal * 1e6f;
      }
    }
    float recv = __shfl_up_sync(0xffffffffu, dnext, 1);
    const float last = __shfl_sync(0xffffffffu, dnext, 31);
    if (lane == 0) recv = dnext_prev;
    dnext_prev = last;
    const float dPh = dself + recv;
    const float dsig = Ph[j] * (1.0f - Ph[j]);
    float d = dPh * s_sharp * dsig;
    if (valid) {
      g_kappa = fmaf(dPh * dsig * s_sharp, ph[j], g_kappa);
      const int cl = clv[j];
      const float b = __fsub_rn(D, tt[j]);
      if (cl == CLS_TR) {
        const float df = ph[j] - b;
        d += kc[2] * (df > 0.f ? 1.f : (df < 0.f ? -1.f : 0.f));
      } else if (cl == CLS_FS) {
        const float ex = expf(-a.kappa_fs * ph[j]) - 1.0f, lin = ph[j] - b;
        int arg = 0;
        float top = 0.f;
        if (ex > top) {
          top = ex;
          arg = 1;
        }
        if (lin > top) arg = 2;
        d += kc[3] * (arg == 1 ? -a.kappa_fs * (ex + 1.0f) : (arg == 2 ? 1.0f : 0.0f));
      }
    } else {
      d = 0.f;
    }
    // the reverse pass's seeds of the sample: the colour pre-activations' (w gc c (1 - c)) and phi's
    float dp[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) dp[k] = valid ? w[j] * gc[k] * col[j][k] * (1.0f - col[j][k]) : 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) db4[k] += dp[k];
    xch[j * 128] = make_float4(dp[0], dp[1], dp[2], d);
    sum_d += d;
  }
  }  // BWD
  {
    float q[9] = {l_rgb, l_d, l_sdf, l_fs, g_kappa, db4[0], db4[1], db4[2], sum_d};
#pragma unroll
    for (int k = 0; k < NS; ++k) q[k] = warp_sum(q[k]);
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < NS; ++k) sums[k] += q[k];
    }
  }
}

// the forward-only instantiation ends each ray-quad before its reverse pass, which the front
// end reports as unreachable code there
#pragma nv_diag_suppress 128
template <class P, int NCH, int GR, bool FWD, bool BWD>
__global__ void __launch_bounds__(GR * kTileThreads, 1) render_tc_kernel(const __grid_constant__ RenderTcArgs a) {
  using L = TcLayout<P>;
  // a forward-only call writes no tiles: its groups have only their barriers in shared memory
  static_assert(sizeof(TileBars) <= 128, "a group's barriers");
  constexpr uint32_t kGroupBytes = BWD ? L::group_bytes : 128u, kBarOff = BWD ? L::bar_off : 0u;
  extern __shared__ __align__(1024) uint8_t smem[];
  constexpr uint32_t wplane = wTotal<P>();  // one bf16 part of all weight tiles
  // tile groups | weight tiles | exchange rows [GR][NCH][128] float4 | rays | accumulators, biases
  uint8_t* gbase = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem) + 127) & ~uintptr_t(127));
  uint8_t* wt0 = gbase + (size_t)GR * kGroupBytes;
  float4* xch0 = reinterpret_cast<float4*>(wt0 + wplane * P::planes);
  float4* rays0 = xch0 + (size_t)GR * NCH * 128;
  float* sums0 = reinterpret_cast<float*>(rays0 + GR * 20);  // [GR][4][kSums]: a compositing warp's running sums
  float* bias = sums0 + GR * 4 * kSums;  // b1[32] b2[16] b3[32] b4[4] kappa
  float* w4f = bias + 88;         // W4 [3][32] in FP32: the colour output layer runs on CUDA cores
  float* kc = w4f + 96;           // loss scales of rgb, depth, sdf, fs; sharpness
  uint32_t* tslot = reinterpret_cast<uint32_t*>(kc + 8);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform
  const int gi = warp >> 3, w8 = warp & 7, half = w8 >> 2, wq = w8 & 3;
  const int row = 32 * wq + lane;  // tile row of this thread's sample
  uint8_t* const tileA = gbase + (size_t)gi * kGroupBytes;
  uint8_t* const tileB = tileA + L::b_off;
  Tile T;
  T.bars = reinterpret_cast<TileBars*>(tileA + kBarOff);
  T.ph_done = T.ph_dw = 0;
  T.w8 = w8;
  T.g = gi;
  T.dw_pending = false;

  // ---- CTA set-up: weight tiles, biases, accumulators, barriers, tensor memory ----
  const float* mlp = a.theta + a.g.n_grid;
  for (int m = 0; m < kTiles; ++m) {
    const int Nn = wN(m), K = wK(m);
    for (int e = tid; e < Nn * K; e += blockDim.x) {
      const int n = e / K, k = e % K;
      float v = 0.f;
      switch (m) {
        case 0: v = mlp[oW1 + n * kZ + k]; break;
        case 1: v = mlp[oW2 + n * kH1 + k]; break;
        case 2: v = k < kHF ? mlp[oW3 + n * kHF + k] : 0.f; break;
        case 3: v = n < kHF ? mlp[oW3 + k * kHF + n] : 0.f; break;
        case 4: v = mlp[oW2 + k * kH1 + n]; break;
        default: v = mlp[oW1 + k * kZ + n]; break;
      }
      store_w<P>(wt0 + wOff<P>(m), wplane, K, n, k, v);
    }
  }
  for (int i = tid; i < 96; i += blockDim.x) w4f[i] = mlp[oW4 + i];
  for (int i = tid; i < 88; i += blockDim.x) {
    float v = 0.f;
    if (i < 32) v = mlp[ob1 + i];
    else if (i < 48) v = mlp[ob2 + i - 32];
    else if (i < 80) v = mlp[ob3 + i - 48];
    else if (i < 83) v = mlp[ob4 + i - 80];
    else if (i == 84) v = mlp[oKappa];
    bias[i] = v;
  }
  if (tid < GR * 4 * kSums) sums0[tid] = 0.f;
  if (w8 == 0 && lane == 0) {
    tc::mbar_init(&T.bars->done, 1);
    tc::mbar_init(&T.bars->dw, 1);
    tc::fence_mbar_init();
    T.bars->abort = 0;
  }
  if (tid == 0) {
    float wt[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) wt[k] = a.dloss[k] + a.lam[k] * a.dloss[5];
    const int n_d = a.counts[0], n_tr = a.counts[1], n_fs = a.counts[2];
    kc[0] = a.R > 0 ? wt[0] * 2.0f / (float)a.R : 0.f;
    kc[1] = n_d > 0 ? wt[1] / (float)n_d : 0.0f;
    kc[2] = n_tr > 0 ? wt[2] / (float)n_tr : 0.0f;
    kc[3] = n_fs > 0 ? wt[3] / (float)n_fs : 0.0f;
    kc[4] = expf(mlp[oKappa]);
  }
  static_assert(tmem_cols(GR * kGroupCols<BWD>) <= 512, "tensor memory holds 512 columns");
  if (warp == 0) tc::tmem_alloc(tslot, tmem_cols(GR * kGroupCols<BWD>));
  tc::fence_smem_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem0 = __shfl_sync(0xffffffffu, *tslot, 0);
  const int N = a.N, quads = (a.R + 3) / 4;
  const bool stored = a.store != nullptr;
  const bool fphases = FWD || !stored;  // the forward layers run before the compositing
  bool alive = true;
  bool dw_acc = false;  // the weight-gradient accumulators hold a first tile (accumulate from then on)
  // dW4[.][16 half + lane % 16] over this warp's samples of parity lane / 16
  float w4acc[3] = {0.f, 0.f, 0.f};

  const uint32_t sw = tc::smem_u32(wt0), sa = tc::smem_u32(gbase) + (uint32_t)gi * kGroupBytes;
  const uint32_t tcol = tmem0 + (uint32_t)gi * kGroupCols<BWD>;
  const uint32_t tq = tcol + ((uint32_t)(32 * wq) << 16), ta = tq + cA<BWD>;  // this warp's lanes
  const float* b1 = bias + 16 * half;  // this half's units
  const float* b2 = bias + 32;
  const float* b3 = bias + 48 + 16 * half;
  const float* b4 = bias + 80;
  const float* w4h = w4f + 16 * half;
  float4* xch = xch0 + (size_t)gi * NCH * 128;
  float4* rays = rays0 + (gi * 8 + w8) * 2;                     // this warp's ray: o, r
  float4* tint = rays0 + GR * 8 * 2 + gi * 4 + wq;              // its colour and depth (written by the upper half)
  const int l_lo = half ? 1 : 0, l_hi = half ? 2 : 3;  // this half's grid levels (coarse, fine)

  // this half's features of the sample at x into the A operand (levels' columns 4 l .. 4 l + 3)
  auto gather_store = [&](const float x[3], bool valid, float4& zl, float4& zh) {
    zl = zh = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) {
      if constexpr (P::planes > 1) {
        if (half == 0) {
          FineCorners fc;
          fine_corners_load(a.g, a.theta, x, fc);
          zl = level_features(a.g, a.theta, 0, x);
          zh = fine_corners_sum(fc);
        } else {
          zh = level_features(a.g, a.theta, 2, x);
          zl = level_features(a.g, a.theta, 1, x);
        }
      } else {
        zh = level_features_bf16(a.g, a.theta_bf16, l_hi, x);
        zl = level_features_bf16(a.g, a.theta_bf16, l_lo, x);
      }
    }
    __syncwarp();
    const float lo4[4] = {zl.x, zl.y, zl.z, zl.w}, hi4[4] = {zh.x, zh.y, zh.z, zh.w};
    put_operand<P, 16, false, 2>(ta, nullptr, row, 2 * l_lo, lo4);
    put_operand<P, 16, false, 2>(ta, nullptr, row, 2 * l_hi, hi4);
  };
  auto position = [&](float t, float x[3]) {
    const float4 o4 = rays[0], r4 = rays[1];
    const float o[3] = {o4.x, o4.y, o4.z}, r[3] = {r4.x, r4.y, r4.z};
    sample_pos(o, r, t, x);
  };
  // this half's 8 columns of [h | 0] from the 16 outputs [phi, h] of the second layer
  auto hidden_row = [&](const float (&u)[16], float (&h)[8]) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float lo = u[k + 1] + b2[k + 1], hi = k < 7 ? u[k < 7 ? k + 9 : 0] + b2[k < 7 ? k + 9 : 0] : 0.f;
      h[k] = half == 0 ? lo : hi;
    }
  };

  // ray-quads are dealt group-major (quad = round * G + group * CTAs + CTA): a batch with fewer
  // quads than tile groups spreads over all SMs, and so does the last, partial round
  for (int quad = gi * (int)gridDim.x + (int)blockIdx.x; quad < quads && alive; quad += (int)gridDim.x * GR) {
    const int ray = quad * 4 + wq;
    const bool has_ray = ray < a.R;
    const int rr = has_ray ? ray : 0;
    // every sample depth of the ray up front: one memory round trip instead of one per chunk
    float tt[NCH];
#pragma unroll
    for (int q = 0; q < NCH; ++q) {
      const int si = 32 * q + lane;
      tt[q] = has_ray && si < N ? a.t[(size_t)rr * N + si] : 0.f;
    }
    __syncwarp();
    if (lane < 6) reinterpret_cast<float*>(rays)[lane < 3 ? lane : lane + 1] = lane < 3 ? a.o[3 * rr + lane] : a.r[3 * rr + lane - 3];
    __syncwarp();
    float ph[NCH], col[NCH][3];

    // ================= forward: gather, then 3 decoder phases per chunk =================
#pragma unroll 1
    for (int j = 0; j < NCH && alive; ++j) {
      const int si = 32 * j + lane;
      const bool valid = has_ray && si < N;
      const StoreRef sp{reinterpret_cast<float4*>(a.store) + ((size_t)rr * N + 32 * j) * 25 + lane, min(32, N - 32 * j)};
      if (!fphases) {  // stored by the forward pass: no decoder phases here
        if (half != 0) {
          xch[j * 128 + row].w = __int_as_float(valid ? (int)a.cls[(size_t)rr * N + si] : 0);
          if (j == 0 && lane == 0) *tint = make_float4(a.rgb[3 * rr], a.rgb[3 * rr + 1], a.rgb[3 * rr + 2], has_ray ? a.D[rr] : 0.f);
          continue;
        }
        const float4 c4 = valid ? sp[kPc] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < NCH; ++q)
          if (q == j) {
            ph[q] = c4.w;
            col[q][0] = c4.x;
            col[q][1] = c4.y;
            col[q][2] = c4.z;
          }
        continue;
      }
      const bool put = FWD && stored && valid;
      int cl = 0;
      float4 i4 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (half != 0) {  // the compositing's other inputs, fetched by the half that does not composite
        if (valid) cl = (int)a.cls[(size_t)rr * N + si];
        if (j == 0 && lane == 0) i4 = make_float4(a.rgb[3 * rr], a.rgb[3 * rr + 1], a.rgb[3 * rr + 2], has_ray ? a.D[rr] : 0.f);
      }
      float4 zl, zh;
      {
        float x[3];
        position(pick_tc(tt, j), x);
        gather_store(x, valid, zl, zh);
      }
      phase_issue<P, 0, BWD>(T, tcol, sa, sw, dw_acc);
      if (put) {
        sp[kPz + l_lo] = zl;
        sp[kPz + l_hi] = zh;
      }
      if (!(alive = phase_wait(T))) break;
      float v[16];
      tc::tmem_ld16(tq + cX + 16 * half, v);
      tc::tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = fmaxf(v[k] + b1[k], 0.f);
      put_operand<P, 32, false, 8>(ta, nullptr, row, 8 * half, v);
      phase_issue<P, 1, BWD>(T, tcol, sa, sw, dw_acc);
      if (put) put_planes<4>(sp, kPa1 + 4 * half, v);
      if (!(alive = phase_wait(T))) break;
      float u[16];
      tc::tmem_ld16(tq + cY, u);
      tc::tmem_ld_wait();
      const float phi = u[0] + b2[0];
      float h[8];
      hidden_row(u, h);
      put_operand<P, 16, false, 4>(ta, nullptr, row, 4 * half, h);
      phase_issue<P, 2, BWD>(T, tcol, sa, sw, dw_acc);
      if (put) put_planes<2>(sp, kPh + 2 * half, h);
      if (!(alive = phase_wait(T))) break;
      tc::tmem_ld16(tq + cX + 16 * half, v);
      tc::tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = fmaxf(v[k] + b3[k], 0.f);
      if (put) put_planes<4>(sp, kPa2 + 4 * half, v);
      // this half's part of the colour pre-activations W4 a2 + b4
      float c3[3];
#pragma unroll
      for (int n = 0; n < 3; ++n) {
        float s = half == 0 ? b4[n] : 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) s = fmaf(w4h[32 * n + k], v[k], s);
        c3[n] = s;
      }
      if (half != 0) {
        xch[j * 128 + row] = make_float4(c3[0], c3[1], c3[2], __int_as_float(cl));
        if (j == 0 && lane == 0) *tint = i4;
      }
      // keep per-chunk values in registers (compile-time index via a selector loop)
#pragma unroll
      for (int q = 0; q < NCH; ++q)
        if (q == j) {
          ph[q] = valid ? phi : 0.f;
          col[q][0] = c3[0];
          col[q][1] = c3[1];
          col[q][2] = c3[2];
        }
    }
    if (!alive) break;
    // the upper half's parts of the colours, the classes, the observed colour and depth
    group_sync<kTileThreads>(gi);

    if (half == 0) {  // ---- compositing and its adjoint: the lower half, a warp per ray ----
    int clv[NCH];  // sample classes
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      const bool valid = has_ray && 32 * j + lane < N;
      const float4 p4 = xch[j * 128 + row];
      clv[j] = __float_as_int(p4.w);
      if (fphases) {
        col[j][0] = valid ? sigmoidf_(col[j][0] + p4.x) : 0.f;
        col[j][1] = valid ? sigmoidf_(col[j][1] + p4.y) : 0.f;
        col[j][2] = valid ? sigmoidf_(col[j][2] + p4.z) : 0.f;
        if (FWD && stored && valid)
          reinterpret_cast<float4*>(a.store)[((size_t)rr * N + 32 * j) * 25 + kPc * min(32, N - 32 * j) + lane] =
              make_float4(col[j][0], col[j][1], col[j][2], ph[j]);
      }
    }
    const float4 in4 = *tint;
    composite_ray<NCH, FWD, BWD, kSums>(a, ray, has_ray, tt, ph, col, clv, in4, kc, xch + row,
                                        sums0 + (gi * 4 + wq) * kSums);
    }  // lower half
    if constexpr (!BWD) continue;
    group_sync<kTileThreads>(gi);  // the reverse pass's seeds

    // ================= reverse, chunk by chunk: (recompute,) 3 adjoint phases =================
#pragma unroll 1
    for (int j = 0; j < NCH && alive; ++j) {
      const int si = 32 * j + lane;
      const bool valid = has_ray && si < N;
      const StoreRef sp{reinterpret_cast<float4*>(a.store) + ((size_t)rr * N + 32 * j) * 25 + lane, min(32, N - 32 * j)};
      const bool get = stored && valid;
      float v[16], h[8], a1[16];
      float4 zl, zh;
      if (stored) {  // stored activations: a2 and h now, a1 and z where they are used
        get_planes<4>(sp, kPa2 + 4 * half, get, v);
        get_planes<2>(sp, kPh + 2 * half, get, h);
      } else {
        // recompute the decoders (the same phases as the forward)
        {
          float x[3];
          position(pick_tc(tt, j), x);
          gather_store(x, valid, zl, zh);
        }
        phase_issue<P, 0, BWD>(T, tcol, sa, sw, dw_acc);
        if (!(alive = phase_wait(T))) break;
        tc::tmem_ld16(tq + cX + 16 * half, a1);
        tc::tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 16; ++k) a1[k] = fmaxf(a1[k] + b1[k], 0.f);
        put_operand<P, 32, false, 8>(ta, nullptr, row, 8 * half, a1);
        phase_issue<P, 1, BWD>(T, tcol, sa, sw, dw_acc);
        if (!(alive = phase_wait(T))) break;
        float u[16];
        tc::tmem_ld16(tq + cY, u);
        tc::tmem_ld_wait();
        hidden_row(u, h);
        put_operand<P, 16, false, 4>(ta, nullptr, row, 4 * half, h);
        phase_issue<P, 2, BWD>(T, tcol, sa, sw, dw_acc);
        if (!(alive = phase_wait(T))) break;
        tc::tmem_ld16(tq + cX + 16 * half, v);
        tc::tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = fmaxf(v[k] + b3[k], 0.f);
      }
      const float4 seed = xch[j * 128 + row];  // dL/d(colour pre-activations), dL/dphi
      tiles_free(T);  // stage the colour layer's rows there
      // --- b4 on CUDA cores: da2 = dpre W4 (3 x 32); dW4 (+)= sum over the warp's samples ---
      {
        // This warp's 16 a2 columns, 64 bytes a row (the 16-byte pieces rotated against bank
        // conflicts), in the part of the adjoint tile that only this warp writes: of each 8-row group
        // of a K = 32 tile, its half's 256 bytes of a part hold 4 staged rows.  The BF16 form's
        // one part is too small: its rows have their own space.
        constexpr uint32_t kBlk = P::planes > 1 ? L::row_stride(32) : 256u, kPl = P::planes > 1 ? 512u : 1024u;
        uint8_t* st = P::planes > 1 ? tileA + wq * 4 * L::row_stride(32) + half * 256 : tileA + L::stage_off + w8 * 2048;
        float* rw = reinterpret_cast<float*>(st + (lane >> 4) * kPl + ((lane >> 2) & 3) * kBlk + (lane & 3) * 64);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<float4*>(rw + 4 * ((q + (lane >> 1)) & 3)) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        __syncwarp();
        const int hi = lane >> 4, un = lane & 15;  // rows 2 i + hi, unit un of the half
        const float4* sd = xch + j * 128 + 32 * wq + hi;
        uint32_t rot[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) rot[i] = (uint32_t)((((un >> 2) + i) & 3) * 16 + (un & 3) * 4 + hi * 64);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const uint32_t off = (uint32_t)(i >> 3) * kPl + (uint32_t)((i >> 1) & 3) * kBlk + (uint32_t)(i & 1) * 128u;
          const float a2v = *reinterpret_cast<const float*>(st + off + rot[i & 3]);
          const float4 d4 = sd[2 * i];
          w4acc[0] = fmaf(d4.x, a2v, w4acc[0]);
          w4acc[1] = fmaf(d4.y, a2v, w4acc[1]);
          w4acc[2] = fmaf(d4.z, a2v, w4acc[2]);
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 16; ++k) {  // dy2 = mask2 (.) (dpre W4)
          const float d = fmaf(seed.x, w4h[k], fmaf(seed.y, w4h[32 + k], seed.z * w4h[64 + k]));
          v[k] = v[k] > 0.f ? d : 0.f;
        }
      }
      put_operand<P, 32, true, 8>(ta, tileA, row, 8 * half, v);
      if (half != 0) h[7] = 1.f;  // ones column: the bias gradient db3 lands in column 15 of dW3
      store_chunk<L::b_planes, 16, L::b_bytes>(tileB, row, half, h);
      // --- b3: dh = dy2 W3;  dW3, db3 (+)= dy2^T [h | 1] ---
      phase_issue<P, 3, BWD>(T, tcol, sa, sw, dw_acc);
      if (stored) get_planes<4>(sp, kPa1 + 4 * half, get, a1);
      if (!(alive = phase_wait(T))) break;
      {
        float u[16], dout[8];
        tc::tmem_ld16(tq + cY, u);
        tc::tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 8; ++k) dout[k] = half == 0 ? (k == 0 ? (valid ? seed.w : 0.f) : u[k > 0 ? k - 1 : 0]) : u[k + 7];
        tiles_free(T);
        put_operand<P, 16, true, 4>(ta, tileA, row, 4 * half, dout);
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) store_chunk<L::b_planes, 40, L::b_bytes>(tileA + L::b_wide, row, 2 * half + c, a1 + 8 * c);
      const float one8[8] = {1.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (half != 0) store_chunk<L::b_planes, 40, L::b_bytes>(tileA + L::b_wide, row, 4, one8);
      // --- b2: da1 = dout W2;  dW2^T, db2 (+)= [a1 | 1]^T dout ---
      phase_issue<P, 4, BWD>(T, tcol, sa, sw, dw_acc);
      if (stored) {
        zl = get ? sp[kPz + l_lo] : make_float4(0.f, 0.f, 0.f, 0.f);
        zh = get ? sp[kPz + l_hi] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      if (!(alive = phase_wait(T))) break;
      tc::tmem_ld16(tq + cX + 16 * half, v);
      tc::tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = a1[k] > 0.f ? v[k] : 0.f;  // dy1
      tiles_free(T);
      put_operand<P, 32, true, 8>(ta, tileA, row, 8 * half, v);
      store_quarter<L::b_planes, 24, L::b_bytes>(tileB, row, l_lo, zl);
      store_quarter<L::b_planes, 24, L::b_bytes>(tileB, row, l_hi, zh);
      if (half != 0) store_chunk<L::b_planes, 24, L::b_bytes>(tileB, row, 2, one8);
      // --- b1: dz = dy1 W1;  dW1, db1 (+)= dy1^T [z | 1] ---
      phase_issue<P, 5, BWD>(T, tcol, sa, sw, dw_acc);
      if (!(alive = phase_wait(T))) break;
      dw_acc = true;
      float4 gl4, gh4;  // dL/dz at this half's levels
      {
        float u[16];
        tc::tmem_ld16(tq + cY, u);
        tc::tmem_ld_wait();
        gl4 = half == 0 ? make_float4(u[0], u[1], u[2], u[3]) : make_float4(u[4], u[5], u[6], u[7]);
        gh4 = half == 0 ? make_float4(u[12], u[13], u[14], u[15]) : make_float4(u[8], u[9], u[10], u[11]);
      }
      if (!valid) gl4 = gh4 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (a.dz_out != nullptr && valid) {  // dL/dz of this sample (camera-pose gradients)
        float4* dzo = reinterpret_cast<float4*>(a.dz_out + ((size_t)rr * N + si) * kZ);
        dzo[l_lo] = gl4;
        dzo[l_hi] = gh4;
      }
      float x[3];
      position(pick_tc(tt, j), x);
      const float4* er = nullptr;
      if (a.eik != nullptr && valid && a.cls[(size_t)rr * N + si] == CLS_FS) er = a.eik + (size_t)rr * N + si;
      const EikSeed es = eik_seed(er, a.eik_stride);
      scatter_direct<(P::planes == 1)>(a.g, a.grad, l_hi, x, gh4, valid, es);
      tiles_free(T);  // their space holds the run reduction's staging rows
      {
        static_assert(L::runs == 8u * kScatterStage * 4u, "staging space");
        float* st = reinterpret_cast<float*>(tileA) + w8 * kScatterStage;
        scatter_runs(a.g, a.grad, l_lo, x, gl4, valid, st, es);
      }
      group_sync<kTileThreads>(gi);  // every warp is done with its rows before the tiles are rewritten
    }
  }

  // ---- epilogue: loss and decoder-gradient partials, tensor memory ----
  const bool done = tile_end(T, a.status, kStatusRender);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (BWD) {
    // each group's decoder gradients as a row over its tiles
    for (int i = tid; i < GR * kMlpPad; i += blockDim.x)
      reinterpret_cast<float*>(gbase + (size_t)(i / kMlpPad) * L::group_bytes)[i % kMlpPad] = 0.f;
    __syncthreads();
    float* macc = reinterpret_cast<float*>(tileA);
    if (half == 0 && dw_acc && done) {
      // The weight-gradient accumulators: warp w holds rows 16 w .. 16 w + 15 of every M = 64
      // product in its lanes 0..15.  Rows 32 .. 63 of dW1 and dW3 (16 .. 31 of dW2) are the
      // adjoints' second parts; without one they mean nothing.
      const bool mine = lane < 16 && (wq < 2 || P::planes > 1);
      const int m = (16 * wq + lane) & 31;
      float d[16];
      tc::tmem_ld16(tq + cW1, d);
      tc::tmem_ld_wait();
      if (mine) {
#pragma unroll
        for (int n = 0; n < 16; ++n) atomicAdd(macc + oW1 + m * kZ + n, d[n]);
      }
      tc::tmem_ld16(tq + cW1 + 16, d);
      tc::tmem_ld_wait();
      if (mine) atomicAdd(macc + ob1 + m, d[0]);
      tc::tmem_ld16(tq + cW3, d);
      tc::tmem_ld_wait();
      if (mine) {
#pragma unroll
        for (int n = 0; n < 15; ++n) atomicAdd(macc + oW3 + m * kHF + n, d[n]);
        atomicAdd(macc + ob3 + m, d[15]);
      }
      const bool mine2 = lane < 16 && (wq == 0 || (wq == 1 && P::planes > 1));  // row lane: output unit
      tc::tmem_ld16(tq + cW2, d);
      tc::tmem_ld_wait();
      if (mine2) {
#pragma unroll
        for (int n = 0; n < 16; ++n) atomicAdd(macc + oW2 + lane * kH1 + n, d[n]);
      }
      tc::tmem_ld16(tq + cW2 + 16, d);
      tc::tmem_ld_wait();
      if (mine2) {
#pragma unroll
        for (int n = 0; n < 16; ++n) atomicAdd(macc + oW2 + lane * kH1 + 16 + n, d[n]);
      }
      tc::tmem_ld16(tq + cW2 + 32, d);
      tc::tmem_ld_wait();
      if (mine2) atomicAdd(macc + ob2 + lane, d[0]);
    }
    // the colour layer's gradient, accumulated per warp on CUDA cores
#pragma unroll
    for (int n = 0; n < 3; ++n) atomicAdd(macc + oW4 + n * kH2 + 16 * half + (lane & 15), w4acc[n]);
    __syncthreads();
  } else {
    __syncthreads();
  }
  auto total = [&](int k) {  // running sum k over the compositing warps
    float v = 0.f;
#pragma unroll
    for (int q = 0; q < GR * 4; ++q) v += sums0[q * kSums + k];
    return v;
  };
  if (tid < kLossPad) a.loss_part[(size_t)blockIdx.x * kLossPad + tid] = tid < 4 ? total(tid) : 0.f;
  for (int i = tid; i < kMlpPad; i += blockDim.x) {
    float v = i == oKappa ? total(4) : (i >= ob4 && i < ob4 + kRGB ? total(5 + i - ob4) : 0.f);
    if (BWD) {
#pragma unroll
      for (int q = 0; q < GR; ++q) v += reinterpret_cast<const float*>(gbase + (size_t)q * L::group_bytes)[i];
    }
    a.mlp_part[(size_t)blockIdx.x * kMlpPad + i] = v;
  }
  __syncwarp();
  if (warp == 0) tc::tmem_dealloc(*tslot, tmem_cols(GR * kGroupCols<BWD>));
}
#pragma nv_diag_default 128

template <class P, int NCH, int GR, bool BWD>
constexpr size_t render_tc_smem() {
  using L = TcLayout<P>;
  static_assert(kMlpPad * 4 <= L::bar_off, "a group's decoder-gradient row fits over its tiles");
  return 128 + (size_t)GR * (BWD ? L::group_bytes : 128u) + wTotal<P>() * P::planes + (size_t)GR * NCH * 128 * 16 +
         GR * 20 * 16 + (GR * 4 * kSums + 88 + 96 + 8 + 4) * 4;
}

template <class P, int NCH, int GR, bool FWD, bool BWD>
gs_status launch_tc_t(const gs_ctx* ctx, RenderTcArgs& a, cudaStream_t st) {
  constexpr size_t smem = render_tc_smem<P, NCH, GR, BWD>();
  static_assert(smem <= 227u * 1024u, "shared memory per CTA");
  auto k = render_tc_kernel<P, NCH, GR, FWD, BWD>;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return GS_ERR_CUDA;
  k<<<ctx->render_ctas, GR * kTileThreads, smem, st>>>(a);
  return cudaPeekAtLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

template <class P, int NCH>
gs_status launch_tc_n(const gs_ctx* ctx, RenderTcArgs& a, int mode, cudaStream_t st) {
  constexpr int GR = kRenderGroups;  // tile groups in one CTA per SM
  if (mode == 1)
    return forward_groups(a.R, ctx->render_ctas, NCH, a.store != nullptr) == kForwardGroups
               ? launch_tc_t<P, NCH, kForwardGroups, true, false>(ctx, a, st)
               : launch_tc_t<P, NCH, kRenderGroups, true, false>(ctx, a, st);
  if (mode == 2) return launch_tc_t<P, NCH, GR, false, true>(ctx, a, st);
  return launch_tc_t<P, NCH, GR, true, true>(ctx, a, st);
}

}  // namespace gs
