// The paper's architecture (Sec. 3.1 Eq. SDF_MLP and Eq. COLOR_MLP, "Architecture Details") in
// one fused per-ray pass with both decoders on the tcgen05 tensor cores: phi = f_omega(V(x))
// with f_omega 16 -> 32 -> 32 -> 1, c = g_gamma(W_beta(x), d) with g_gamma 9 -> 32 -> 32 -> 3,
// NeuS compositing and the losses of Sec. 3.2-3.4, then their reverse mode down to both grids
// and every decoder weight.
//
// Mapping (as in the compact decoder's kernel).  A group of 8 warps owns one M = 128 tile, two
// threads per tile row: warps w and w + 4 render one ray and its 32-sample chunk j fills rows 32 w
// .. 32 w + 31.  The two decoders are independent given their inputs, so the lower half's threads
// run the geometry decoder (tile Ag) and the upper half's the colour decoder (tile Ac), each layer
// of both as one phase of two products:
//   forward  F1: [Z | U] -> H1 (K = 16),  F2: [A1 | R1] -> H2 (K = 32); the 32 -> 1 and
//            32 -> 3 output layers on CUDA cores;
//   reverse  (the forward recomputed: F1, F2), B1: [dY2 | dQ2] -> [dA1 | dR1] (K = 32),
//            B2: [dY1 | dQ1] -> [dZ | dU] (K = 32), each with the weight-gradient products
//            D[64][32] (+)= sum over the tile's samples of [x | 1]^T dy (MN-major operands,
//            accumulated in tensor memory over all of the group's tiles) issued by two other
//            warps; the output layers' gradients on CUDA cores.
// Grid level 1 goes with the upper half (its gather beside the colour corners, its run-reduced
// scatter beside the colour grid's), the other levels with the lower.  Compositing by the lower
// half.  Operands are split into three bfloat16 parts with the six leading part products
// accumulated in FP32 (two parts and three products in the weight-gradient products), as in the
// compact kernel's FP32 form.  Activations are stored by the forward pass (156 floats per sample,
// a chunk's together) and read back by the reverse pass, or recomputed there (no store).  Grid
// gradients: the geometry levels through the compact kernel's scatter (which also adds the
// deferred Eikonal records of the free-space samples), the colour grid (6 floats per finest-level
// vertex) with one 16-byte and one 8-byte reduction per corner; samples whose vectors are exactly
// zero issue none.  With one thread per row for both decoders the SM held 8 warps at 255 registers;
// 8192 x 96, stored: 974 us a call, then 854; with the operands in tensor memory 828 (recomputed
// 1160, 1047, 976).
#pragma once
#include "gs_paper.cuh"
#include "gs_render_tc.cuh"

namespace gs {
namespace ptc {

using paper::kC;
using paper::kH;
using paper::kU;
using P3 = PrecBF16x3;
constexpr int kPaperSums = kSums + 1;  // and the SDF seeds' (the output layer's bias)

// weight (B) tiles {N, K}:
//   0 gW1 32x16 | 1 cW1 32x16 (cols 9.. zero) | 2 gW2 32x32 | 3 cW2 32x32
//   4 gW2^T 32x32 | 5 cW2^T 32x32 | 6 gW1^T 16x32 | 7 cW1^T 16x32 (rows 9.. zero)
__host__ __device__ constexpr int tN(int i) { return i < 6 ? 32 : 16; }
__host__ __device__ constexpr int tK(int i) { return i < 2 ? 16 : 32; }
__host__ __device__ constexpr uint32_t tOff(int i) {
  uint32_t o = 0;
  for (int k = 0; k < i; ++k) o += (uint32_t)(tN(k) * tK(k) * 2);
  return o;
}
constexpr uint32_t kTW = tOff(8);  // one bfloat16 part of all eight tiles

// per group: A tiles Ag | Ac (3 parts of 128 x 32 each) | partner tiles Bg | Bc (2 parts each: a1,
// [r1 | 1] in B1, [z | 1], [u | 1] in B2; the geometry's second layer has its bias gradient from the
// output layer's loop, which leaves room for the exchange rows of 160 samples) | barriers.  The
// M = 64 reads of a partner tile run up to 512 bytes past its last part: into the next tile, the
// group's barriers and the next group (or, for the last group, the weight tiles).
constexpr uint32_t kAP = 128u * 32u * 2u;  // one part of an A tile
constexpr uint32_t kBPg = 128u * 32u * 2u, kBP = 128u * 40u * 2u;  // one part of a partner tile
constexpr uint32_t oAg = 0, oAc = 3 * kAP, oBg = 6 * kAP, oBc = oBg + 2 * kBPg, oBar = oBc + 2 * kBP;
constexpr uint32_t kPGroupBytes = oBar + 128;
constexpr int kPGroups = 2;  // tensor memory: 2 groups x 256 columns
constexpr int kPThreads = kPGroups * kTileThreads;

// tensor-memory columns of a group: phase outputs (geometry, colour), the weight-gradient
// accumulators (M = 64 layout: row m in lane 32 (m / 16) + m % 16), then the two leading parts of the
// phases' A operands (part p of a K-column row in columns p K / 2 ..; the third part, read by one
// product of six, has no columns left and stays in the A tile)
constexpr uint32_t cG = 0, cC = 32, cWg2 = 64, cWc2 = 96, cWg1 = 128, cWc1 = 160, cAg = 192, cAc = 224, kPCols = 256;
constexpr uint32_t kPTmem = 512;
static_assert(kPGroups * kPCols <= kPTmem, "tensor-memory columns");

// FP32 scalars of the decoders in shared memory
constexpr int sc_gb1 = 0, sc_gb2 = 32, sc_gw3 = 64, sc_gb3 = 96, sc_cb1 = 100, sc_cb2 = 132, sc_cW3 = 164,
              sc_cb3 = 260, sc_kappa = 263, kScal = 264;
static_assert(8u * kScatterStage * 4u <= 6u * kAP, "the run reduction's rows fit in the A tiles");

struct PaperTcArgs {
  GridDesc g;            // geometry levels; g.n_grid = decoder block offset (after the colour grid)
  long long colour_off;  // float offset of the colour grid (a multiple of 4)
  const float* theta;
  float* grad;
  const float *o, *r, *rgb, *D, *t;
  const uint8_t* cls;
  const int* counts;
  const float* dloss;
  float lam[5];
  float kappa_fs;
  float *rgb_hat, *d_hat, *wsum, *w_out;
  float* dz_out;                // [R][N][32] per-sample records for the pose gradient (may be nullptr)
  float *loss_part, *mlp_part;  // this kernel's partial rows, one per CTA
  int R, N;
  int* status;  // kStatusPaperRender: a tensor-core phase did not complete
  // deferred Eikonal records ([5][R N] float4 planes) of the free-space samples, added to their
  // geometry scatter; nullptr: none
  const float4* eik;
  long long eik_stride;
  // stored activations: written by forward passes, read by backward passes in place of the gathers
  // and the two recomputed phases; nullptr: recompute
  float* store;
};

// planes of one chunk's stored activations (StoreRef, 39 float4 a sample): z by level [4] | cf [2] |
// c, phi | a1 [8] | r1 [8] | a2 [8] | r2 [8]
constexpr int kQz = 0, kQu = 4, kQc = 6, kQa1 = 7, kQr1 = 15, kQa2 = 23, kQr2 = 31, kQPlanes = 39;
static_assert(kQPlanes * 4 == kPaperStoreFloatsPerSample, "the store holds every field");

__device__ __forceinline__ void red_add_f2(float* p, float a, float b) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b));
}

// the colour features cf at x: the finest cell's 8 corners, 6 floats per vertex
__device__ __forceinline__ void gather_colour(const PaperTcArgs& a, const float x[3], float cf[kC]) {
  constexpr int l = kLevels - 1;
  const Cell c = locate(a.g, l, x);
  const int nx = a.g.dims[l][0], ny = a.g.dims[l][1];
  const float f0 = c.f[0], f1 = c.f[1], f2 = c.f[2];
  const float* cg = a.theta + a.colour_off;
#pragma unroll
  for (int i = 0; i < kC; ++i) cf[i] = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {  // corner k: vertex (x + (k & 1), y + (k >> 1 & 1), z + (k >> 2))
    const long long v = c.vtx + (k & 1) + (long long)((k >> 1) & 1) * nx + (long long)(k >> 2) * nx * ny;
    // its 24 bytes lie in the 16-byte aligned 32-byte window that starts at them (even v) or 8
    // bytes before them (odd v): two loads and selects, no branch, so that the loads of all
    // corners are in flight together (past the last vertex the window reads the decoder block)
    const bool odd = (v & 1) != 0;
    const float4* q = reinterpret_cast<const float4*>(cg + 6 * v - (odd ? 2 : 0));
    const float4 A = __ldg(q), B = __ldg(q + 1);
    const float e[6] = {odd ? A.z : A.x, odd ? A.w : A.y, odd ? B.x : A.z,
                        odd ? B.y : A.w, odd ? B.z : B.x, odd ? B.w : B.y};
    const float w = (((k & 1) ? f0 : 1.0f - f0) * ((k & 2) ? f1 : 1.0f - f1)) * ((k & 4) ? f2 : 1.0f - f2);
#pragma unroll
    for (int i = 0; i < kC; ++i) cf[i] = fmaf(w, e[i], cf[i]);
  }
}

// colour-grid gradient of one sample: corner k of the finest cell += w_k dcf
__device__ __forceinline__ void scatter_colour(const PaperTcArgs& a, const float x[3], const float dcf[kC]) {
  const int l = kLevels - 1;
  const Cell c = locate(a.g, l, x);
  float w[8];
  corner_weights(c.f, w);
  float* cg = a.grad + a.colour_off;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const long long v = c.vtx + corner_offset(a.g, l, k);
    float* p = cg + 6 * v;
    float e[6];
#pragma unroll
    for (int q = 0; q < kC; ++q) e[q] = w[k] * dcf[q];
    if ((v & 1) == 0) {
      red_add_f4(reinterpret_cast<float4*>(p), make_float4(e[0], e[1], e[2], e[3]));
      red_add_f2(p + 4, e[4], e[5]);
    } else {
      red_add_f2(p, e[0], e[1]);
      red_add_f4(reinterpret_cast<float4*>(p + 2), make_float4(e[2], e[3], e[4], e[5]));
    }
  }
}

// Rows written by every thread of the group -> one thread of warp 0 issues the phase's products
// and, with DW, one of warps 4 and 5 each one decoder's weight-gradient products that read the same
// tiles (two commits to the dw barrier; the tiles are rewritten only after them)
template <bool DW, class F, class Fg, class Fc>
__device__ __forceinline__ void phase2(Tile& T, F mma, Fg dwg, Fc dwc) {
  tc::tmem_st_wait();
  tc::fence_smem_async();
  tc::fence_before_sync();
  group_sync<kTileThreads>(T.g);
  tc::fence_after_sync();
  if (T.w8 == 0) {
    if (tc::elect_one()) {
      mma();
      tc::mma_commit(&T.bars->done);
    }
    __syncwarp();
  } else if (DW && (T.w8 == 4 || T.w8 == 5)) {
    if (tc::elect_one()) {
      if (T.w8 == 4) dwg();
      else dwc();
      tc::mma_commit(&T.bars->dw);
    }
    __syncwarp();
  }
  if (DW) T.dw_pending = true;
}

// D[128][N] = A[128][K] B[N][K]^T over the six leading part products, smallest first: A's parts 0
// and 1 from tensor memory (ta), part 2 from the A tile at a0, B's parts kTW apart
template <int N, int K>
__device__ __forceinline__ void mma3(uint32_t d, uint32_t ta, uint32_t a0, uint32_t b0) {
  constexpr uint32_t sbo = K * 16u, idesc = tc::instr_desc(128, N);
  const uint32_t alo = tc::desc_lo(a0 + 2 * kAP, 128u), blo = tc::desc_lo(b0, 128u);
  bool first = true;
#pragma unroll
  for (int s = 0; s < K / 16; ++s) {
    const uint32_t off = (uint32_t)s * 256u;
#pragma unroll
    for (int sum = 2; sum >= 0; --sum)
#pragma unroll
      for (int i = 0; i <= sum; ++i) {
        const uint64_t bd = tc::desc_of(blo + (((sum - i) * kTW + off) >> 4), tc::desc_hi(sbo));
        if (i < 2) tc::mma_bf16_ta(d, ta + (uint32_t)(i * (K / 2) + s * 8), bd, idesc, first ? 0u : 1u);
        else tc::mma_bf16(d, tc::desc_of(alo + (off >> 4), tc::desc_hi(sbo)), bd, idesc, first ? 0u : 1u);
        first = false;
      }
  }
}
// 2 W values of a K-column operand row from column 2 w0 on: parts 0 and 1 into tensor memory and,
// for the weight-gradient products (DW), the A tile; part 2 into the A tile
template <int K, bool DW, int W>
__device__ __forceinline__ void put_row(uint32_t ta, uint8_t* tile, int row, int w0, const float* v) {
  uint32_t w[3][W];
  split_words<3, W>(v, w);
  tc::tmem_st(ta + (uint32_t)w0, w[0]);
  tc::tmem_st(ta + (uint32_t)(K / 2 + w0), w[1]);
#pragma unroll
  for (int pl = DW ? 0 : 2; pl < 3; ++pl) {
    uint8_t* t = tile + pl * kAP;
    if constexpr (W >= 4) {
#pragma unroll
      for (int c = 0; c < W / 4; ++c)
        *reinterpret_cast<uint4*>(t + tc::core_offset((uint32_t)row, (uint32_t)(w0 / 4 + c), 128u, K * 16u)) =
            make_uint4(w[pl][4 * c], w[pl][4 * c + 1], w[pl][4 * c + 2], w[pl][4 * c + 3]);
    } else {
      *reinterpret_cast<uint2*>(t + tc::core_offset((uint32_t)row, (uint32_t)(w0 / 4), 128u, K * 16u) + (uint32_t)(w0 & 3) * 4u) =
          make_uint2(w[pl][0], w[pl][1]);
    }
  }
}
// a whole row
template <int K, bool DW>
__device__ __forceinline__ void put_rows(uint32_t ta, uint8_t* tile, int row, const float* v) {
#pragma unroll
  for (int c = 0; c < K / 16; ++c) put_row<K, DW, 8>(ta, tile, row, 8 * c, v + 16 * c);
}

// the forward-only instantiation ends each ray-quad before its reverse pass, which the front
// end reports as unreachable code there
#pragma nv_diag_suppress 128
template <int NCH, bool FWD, bool BWD>
__global__ void __launch_bounds__(kPThreads, 1) paper_tc_kernel(const __grid_constant__ PaperTcArgs a) {
  using namespace paper;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  uint8_t* wt = base + kPGroups * kPGroupBytes;  // the eight weight tiles, 3 parts
  float4* xch0 = reinterpret_cast<float4*>(wt + 3 * kTW);  // exchange rows [kPGroups][NCH][128]
  float4* rays0 = xch0 + (size_t)kPGroups * NCH * 128;
  float* sc = reinterpret_cast<float*>(rays0 + kPGroups * 20);
  float* kc = sc + kScal;     // loss scales of rgb, depth, sdf, fs; sharpness
  float* sums0 = kc + 8;      // [kPGroups][4][kPaperSums]: a compositing warp's running sums
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sums0 + kPGroups * 4 * kPaperSums);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform
  const int gi = warp >> 3, w8 = warp & 7, half = w8 >> 2, wq = w8 & 3;
  const int row = 32 * wq + lane;  // tile row of this thread's sample
  uint8_t* gmem = base + (size_t)gi * kPGroupBytes;
  uint8_t* tileA = gmem + (half ? oAc : oAg);  // this half's decoder
  uint8_t* tileB = gmem + (half ? oBc : oBg);
  Tile T;
  T.bars = reinterpret_cast<TileBars*>(gmem + oBar);
  T.g = gi;
  T.w8 = w8;
  T.ph_done = T.ph_dw = 0;
  T.dw_pending = false;

  // ---- CTA set-up: weight tiles, scalars, accumulators, barriers, tensor memory ----
  const float* mlp = a.theta + a.g.n_grid;
  for (int m = 0; m < 8; ++m) {
    const int Nn = tN(m), K = tK(m);
    for (int e = tid; e < Nn * K; e += blockDim.x) {
      const int n = e / K, k = e % K;
      float v = 0.f;
      switch (m) {
        case 0: v = mlp[A_gW1 + n * kZ + k]; break;
        case 1: v = k < kU ? mlp[A_cW1 + n * kU + k] : 0.f; break;
        case 2: v = mlp[A_gW2 + n * kH + k]; break;
        case 3: v = mlp[A_cW2 + n * kH + k]; break;
        case 4: v = mlp[A_gW2 + k * kH + n]; break;
        case 5: v = mlp[A_cW2 + k * kH + n]; break;
        case 6: v = mlp[A_gW1 + k * kZ + n]; break;
        default: v = n < kU ? mlp[A_cW1 + k * kU + n] : 0.f; break;
      }
      store_w<P3>(wt + tOff(m), kTW, K, n, k, v);
    }
  }
  for (int i = tid; i < kScal; i += blockDim.x) {
    float v = 0.f;
    if (i < sc_gb2) v = mlp[A_gb1 + i];
    else if (i < sc_gw3) v = mlp[A_gb2 + i - sc_gb2];
    else if (i < sc_gb3) v = mlp[A_gw3 + i - sc_gw3];
    else if (i == sc_gb3) v = mlp[A_gb3];
    else if (i >= sc_cb1 && i < sc_cb2) v = mlp[A_cb1 + i - sc_cb1];
    else if (i >= sc_cb2 && i < sc_cW3) v = mlp[A_cb2 + i - sc_cb2];
    else if (i >= sc_cW3 && i < sc_cb3) v = mlp[A_cW3 + i - sc_cW3];
    else if (i >= sc_cb3 && i < sc_kappa) v = mlp[A_cb3 + i - sc_cb3];
    else if (i == sc_kappa) v = mlp[A_kappa];
    sc[i] = v;
  }
  if (tid < kPGroups * 4 * kPaperSums) sums0[tid] = 0.f;
  if (w8 == 0 && lane == 0) {
    tc::mbar_init(&T.bars->done, 1);
    tc::mbar_init(&T.bars->dw, 2);
    tc::fence_mbar_init();
    T.bars->abort = 0;
  }
  if (tid == 0) {
    float wt4[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) wt4[k] = a.dloss[k] + a.lam[k] * a.dloss[5];
    const int n_d = a.counts[0], n_tr = a.counts[1], n_fs = a.counts[2];
    kc[0] = a.R > 0 ? wt4[0] * 2.0f / (float)a.R : 0.f;
    kc[1] = n_d > 0 ? wt4[1] / (float)n_d : 0.0f;
    kc[2] = n_tr > 0 ? wt4[2] / (float)n_tr : 0.0f;
    kc[3] = n_fs > 0 ? wt4[3] / (float)n_fs : 0.0f;
    kc[4] = expf(mlp[A_kappa]);
  }
  if (warp == 0) tc::tmem_alloc(tslot, kPTmem);
  tc::fence_smem_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tcol = __shfl_sync(0xffffffffu, *tslot, 0) + (uint32_t)(gi * kPCols);
  const uint32_t tq = tcol + ((uint32_t)(32 * wq) << 16);      // this warp's lanes
  const uint32_t tx = tq + (half ? cC : cG), ta = tq + (half ? cAc : cAg);  // its decoder's phase output and operand
  const uint32_t sg = tc::smem_u32(base) + (uint32_t)gi * kPGroupBytes, sw = tc::smem_u32(wt);
  const float* hb1 = sc + (half ? sc_cb1 : sc_gb1);
  const float* hb2 = sc + (half ? sc_cb2 : sc_gb2);
  float4* xch = xch0 + (size_t)gi * NCH * 128;
  float4* rays = rays0 + (gi * 8 + w8) * 2;                     // this warp's ray: o, r
  float4* tint = rays0 + kPGroups * 8 * 2 + gi * 4 + wq;        // its colour and depth (written by the upper half)
  const int N = a.N, quads = (a.R + 3) / 4;
  const bool stored = a.store != nullptr;
  const bool fphases = FWD || !stored;  // the forward layers run before the compositing
  bool alive = true, dw_acc = false;
  // this lane's column of the output layers' gradients: gw3[lane], gb2[lane] over gw3[lane] (lower
  // half), cW3[.][lane] (upper)
  float oacc[3] = {0.f, 0.f, 0.f};

  auto position = [&](float t, float x[3]) {
    const float4 o4 = rays[0], r4 = rays[1];
    const float o[3] = {o4.x, o4.y, o4.z}, r[3] = {r4.x, r4.y, r4.z};
    sample_pos(o, r, t, x);
  };
  // u[9..15] = 0 and u[6..8] = the unit viewing direction, the colour decoder's last inputs
  auto view_inputs = [&](float (&u)[16]) {
    const float4 r4 = rays[1];
    const float rn = sqrtf(r4.x * r4.x + r4.y * r4.y + r4.z * r4.z);
    u[kC] = r4.x / rn;
    u[kC + 1] = r4.y / rn;
    u[kC + 2] = r4.z / rn;
#pragma unroll
    for (int k = kU; k < 16; ++k) u[k] = 0.f;
  };
  // this half's decoder inputs at x: u = z of the levels 0, 2, 3 (lower half; level 1's columns are
  // the upper half's z1) or the colour inputs (upper half), into the A tiles
  auto gather_store = [&](const float x[3], bool valid, float (&u)[16], float4& z1) {
#pragma unroll
    for (int k = 0; k < 16; ++k) u[k] = 0.f;
    z1 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) {
      if (half == 0) {
        FineCorners fc;
        fine_corners_load(a.g, a.theta, x, fc);
        const float4 z2 = level_features(a.g, a.theta, 2, x), z0 = level_features(a.g, a.theta, 0, x),
                     z3 = fine_corners_sum(fc);
        u[0] = z0.x, u[1] = z0.y, u[2] = z0.z, u[3] = z0.w;
        u[8] = z2.x, u[9] = z2.y, u[10] = z2.z, u[11] = z2.w;
        u[12] = z3.x, u[13] = z3.y, u[14] = z3.z, u[15] = z3.w;
      } else {
        gather_colour(a, x, u);
        z1 = level_features(a.g, a.theta, 1, x);
      }
    }
    tiles_free(T);
    __syncwarp();
    if (half == 0) {
      put_row<16, false, 2>(ta, tileA, row, 0, u);
      put_row<16, false, 4>(ta, tileA, row, 4, u + 8);
    } else {
      view_inputs(u);
      put_rows<16, false>(ta, tileA, row, u);
      const float q1[4] = {z1.x, z1.y, z1.z, z1.w};
      put_row<16, false, 2>(tq + cAg, gmem + oAg, row, 2, q1);
    }
  };
  auto nop = [] {};
  auto f1 = [&] {
    mma3<32, 16>(tcol + cG, tcol + cAg, sg + oAg, sw + tOff(0));
    mma3<32, 16>(tcol + cC, tcol + cAc, sg + oAc, sw + tOff(1));
  };
  auto f2 = [&] {
    mma3<32, 32>(tcol + cG, tcol + cAg, sg + oAg, sw + tOff(2));
    mma3<32, 32>(tcol + cC, tcol + cAc, sg + oAc, sw + tOff(3));
  };

  // ray-quads are dealt group-major, as in the compact kernel
  for (int quad = gi * (int)gridDim.x + (int)blockIdx.x; quad < quads && alive; quad += (int)gridDim.x * kPGroups) {
    const int ray = quad * 4 + wq;
    const bool has_ray = ray < a.R;
    const int rr = has_ray ? ray : 0;
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

    // ================= forward: gather, then F1 and F2 per chunk =================
#pragma unroll 1
    for (int j = 0; j < NCH && alive; ++j) {
      const int si = 32 * j + lane;
      const bool valid = has_ray && si < N;
      const StoreRef sp{reinterpret_cast<float4*>(a.store) + ((size_t)rr * N + 32 * j) * kQPlanes + lane, min(32, N - 32 * j)};
      int cl = 0;
      float4 i4 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (half != 0) {  // the compositing's other inputs, fetched by the half that does not composite
        if (valid) cl = (int)a.cls[(size_t)rr * N + si];
        if (j == 0 && lane == 0) i4 = make_float4(a.rgb[3 * rr], a.rgb[3 * rr + 1], a.rgb[3 * rr + 2], has_ray ? a.D[rr] : 0.f);
      }
      float c3[3] = {0.f, 0.f, 0.f}, phi = 0.f;
      if (fphases) {
        const bool put = FWD && stored && valid;
        float u[16], v[32];
        float4 z1;
        {
          float x[3];
          position(pick_tc(tt, j), x);
          gather_store(x, valid, u, z1);
        }
        phase2<false>(T, f1, nop, nop);
        if (put) {
          if (half == 0) {
            sp[kQz] = make_float4(u[0], u[1], u[2], u[3]);
            put_planes<2>(sp, kQz + 2, u + 8);
          } else {
            sp[kQz + 1] = z1;
            sp[kQu] = make_float4(u[0], u[1], u[2], u[3]);
            sp[kQu + 1] = make_float4(u[4], u[5], 0.f, 0.f);
          }
        }
        if (!(alive = phase_wait(T))) break;
        tc::tmem_ld32(tx, v);
        tc::tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = fmaxf(v[k] + hb1[k], 0.f);
        put_rows<32, false>(ta, tileA, row, v);
        phase2<false>(T, f2, nop, nop);
        if (put) put_planes<8>(sp, half ? kQr1 : kQa1, v);
        if (!(alive = phase_wait(T))) break;
        tc::tmem_ld32(tx, v);
        tc::tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = fmaxf(v[k] + hb2[k], 0.f);
        if (put) put_planes<8>(sp, half ? kQr2 : kQa2, v);
        if (half == 0) {
          phi = sc[sc_gb3];
#pragma unroll
          for (int k = 0; k < 32; ++k) phi = fmaf(sc[sc_gw3 + k], v[k], phi);
        } else {
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            float s = sc[sc_cb3 + i];
#pragma unroll
            for (int k = 0; k < 32; ++k) s = fmaf(sc[sc_cW3 + 32 * i + k], v[k], s);
            c3[i] = valid ? sigmoidf_(s) : 0.f;
          }
        }
      } else if (half == 0 && valid) {  // stored by the forward pass: phi and c only
        const float4 c4 = sp[kQc];
        c3[0] = c4.x;
        c3[1] = c4.y;
        c3[2] = c4.z;
        phi = c4.w;
      }
      if (half != 0) {
        xch[j * 128 + row] = make_float4(c3[0], c3[1], c3[2], __int_as_float(cl));
        if (j == 0 && lane == 0) *tint = i4;
      }
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
    group_sync<kTileThreads>(gi);  // the colours, the classes, the observed colour and depth are there

    if (half == 0) {  // ---- compositing and its adjoint: the lower half, a warp per ray ----
      int clv[NCH];
#pragma unroll
      for (int j = 0; j < NCH; ++j) {
        const float4 p4 = xch[j * 128 + row];
        clv[j] = __float_as_int(p4.w);
        if (fphases) {
          col[j][0] = p4.x;
          col[j][1] = p4.y;
          col[j][2] = p4.z;
          if (FWD && stored && has_ray && 32 * j + lane < N)
            reinterpret_cast<float4*>(a.store)[((size_t)rr * N + 32 * j) * kQPlanes + kQc * min(32, N - 32 * j) + lane] =
                make_float4(p4.x, p4.y, p4.z, ph[j]);
        }
      }
      const float4 in4 = *tint;
      composite_ray<NCH, FWD, BWD, kPaperSums>(a, ray, has_ray, tt, ph, col, clv, in4, kc, xch + row,
                                               sums0 + (gi * 4 + wq) * kPaperSums);
    }
    if constexpr (!BWD) continue;
    group_sync<kTileThreads>(gi);  // the reverse pass's seeds

    // ================= reverse, chunk by chunk: the stored activations (or F1, F2 again), B1, B2, scatter =================
#pragma unroll 1
    for (int j = 0; j < NCH && alive; ++j) {
      const int si = 32 * j + lane;
      const bool valid = has_ray && si < N;
      const StoreRef sp{reinterpret_cast<float4*>(a.store) + ((size_t)rr * N + 32 * j) * kQPlanes + lane, min(32, N - 32 * j)};
      const bool get = stored && valid;
      float v[32], h1[32], u[16];  // second layer's outputs, first layer's, the decoder's inputs
      float4 z1;
      if (stored) {  // no gather and no forward phases
        get_planes<8>(sp, half ? kQr2 : kQa2, get, v);
        get_planes<8>(sp, half ? kQr1 : kQa1, get, h1);
      } else {
        {
          float x[3];
          position(pick_tc(tt, j), x);
          gather_store(x, valid, u, z1);
        }
        phase2<false>(T, f1, nop, nop);
        if (!(alive = phase_wait(T))) break;
        tc::tmem_ld32(tx, h1);
        tc::tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 32; ++k) h1[k] = fmaxf(h1[k] + hb1[k], 0.f);
        put_rows<32, false>(ta, tileA, row, h1);
        phase2<false>(T, f2, nop, nop);
        if (!(alive = phase_wait(T))) break;
        tc::tmem_ld32(tx, v);
        tc::tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = fmaxf(v[k] + hb2[k], 0.f);
      }
      const float4 seed = xch[j * 128 + row];  // dL/d(colour pre-activations), dL/dphi
      tiles_free(T);
      {
        // output layers on CUDA cores: the warp's second-layer outputs staged as rows of 36 floats
        // in its own rows of the A tile's parts (2048 bytes of each: 14 rows), then lane = column
        uint8_t* st = tileA + wq * 2048;
        float* orow = reinterpret_cast<float*>(st + (lane / 14) * kAP + (lane % 14) * 144);
#pragma unroll
        for (int q = 0; q < 8; ++q)
          *reinterpret_cast<float4*>(orow + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        __syncwarp();
        const float4* sd = xch + j * 128 + 32 * wq;
#pragma unroll 1
        for (int p = 0; p < 3; ++p) {
          const float* r2 = reinterpret_cast<const float*>(st + p * kAP) + lane;
          const int n2 = p < 2 ? 14 : 4;
          if (half == 0) {
#pragma unroll 4
            for (int s2 = 0; s2 < n2; ++s2) {
              const float d = sd[14 * p + s2].w, a2 = r2[36 * s2];
              oacc[0] = fmaf(d, a2, oacc[0]);
              oacc[1] += a2 > 0.f ? d : 0.f;  // dy2 = [a2 > 0] gw3 dphi
            }
          } else {
#pragma unroll 4
            for (int s2 = 0; s2 < n2; ++s2) {
              const float4 d4 = sd[14 * p + s2];
              const float rv = r2[36 * s2];
              oacc[0] = fmaf(d4.x, rv, oacc[0]);
              oacc[1] = fmaf(d4.y, rv, oacc[1]);
              oacc[2] = fmaf(d4.z, rv, oacc[2]);
            }
          }
        }
        __syncwarp();
      }
      if (half == 0) {
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = v[k] > 0.f ? sc[sc_gw3 + k] * seed.w : 0.f;  // dy2
      } else {
#pragma unroll
        for (int k = 0; k < 32; ++k) {  // dq2 = m(r2) (.) cW3^T dpre
          const float d = fmaf(seed.x, sc[sc_cW3 + k], fmaf(seed.y, sc[sc_cW3 + 32 + k], seed.z * sc[sc_cW3 + 64 + k]));
          v[k] = v[k] > 0.f ? d : 0.f;
        }
      }
      put_rows<32, true>(ta, tileA, row, v);
      const float one8[8] = {1.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // ones column: the bias gradient lands in its row
      if (half == 0) {
        store_row_planes<2, 32, kBPg>(tileB, row, h1);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) store_chunk<2, 40, kBP>(tileB, row, c, h1 + 8 * c);
        store_chunk<2, 40, kBP>(tileB, row, 4, one8);
      }
      // B1: dA1 = dY2 gW2, dR1 = dQ2 cW2; dW2^T (+)= a1^T dY2 and the colour's [r1 | 1]^T dQ2
      phase2<true>(T, [&] {
        mma3<32, 32>(tcol + cG, tcol + cAg, sg + oAg, sw + tOff(4));
        mma3<32, 32>(tcol + cC, tcol + cAc, sg + oAc, sw + tOff(5));
      }, [&] {
        issue_mma_dw<2, 3, 2, 32>(tcol + cWg2, sg + oBg, kBPg, 4u * 128u, sg + oAg, kAP, 4u * 128u, dw_acc);
      }, [&] {
        issue_mma_dw<2, 3, 2, 32>(tcol + cWc2, sg + oBc, kBP, 5u * 128u, sg + oAc, kAP, 4u * 128u, dw_acc);
      });
      if (stored) {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        z1 = zero;
        if (half == 0) {
          get_planes<1>(sp, kQz, get, u);
          get_planes<2>(sp, kQz + 2, get, u + 8);
        } else {
          get_planes<2>(sp, kQu, get, u);
          if (get) z1 = sp[kQz + 1];
          view_inputs(u);
        }
      }
      if (!(alive = phase_wait(T))) break;
      tc::tmem_ld32(tx, v);
      tc::tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < 32; ++k) v[k] = h1[k] > 0.f ? v[k] : 0.f;  // dy1, dq1
      tiles_free(T);
      put_rows<32, true>(ta, tileA, row, v);
      if (half == 0) {
        store_quarter<2, 24, kBPg>(tileB, row, 0, make_float4(u[0], u[1], u[2], u[3]));
        store_chunk<2, 24, kBPg>(tileB, row, 1, u + 8);
        store_chunk<2, 24, kBPg>(tileB, row, 2, one8);
      } else {
        u[kU] = 1.f;
        store_row_planes<2, 16, kBP>(tileB, row, u);
        store_quarter<2, 24, kBPg>(gmem + oBg, row, 1, z1);
      }
      // B2: dZ = dY1 gW1, dU = dQ1 cW1; dW1, db1 (+)= [z | 1]^T dY1 and the colour's [u | 1]^T dQ1
      phase2<true>(T, [&] {
        mma3<16, 32>(tcol + cG, tcol + cAg, sg + oAg, sw + tOff(6));
        mma3<16, 32>(tcol + cC, tcol + cAc, sg + oAc, sw + tOff(7));
      }, [&] {
        issue_mma_dw<2, 3, 2, 32>(tcol + cWg1, sg + oBg, kBPg, 3u * 128u, sg + oAg, kAP, 4u * 128u, dw_acc);
      }, [&] {
        issue_mma_dw<2, 3, 2, 32>(tcol + cWc1, sg + oBc, kBP, 2u * 128u, sg + oAc, kAP, 4u * 128u, dw_acc);
      });
      if (!(alive = phase_wait(T))) break;
      dw_acc = true;
      float d[16];  // dz (lower half), du (upper half)
      tc::tmem_ld16(tx, d);
      float dz1[16];
      if (half != 0) tc::tmem_ld16(tq + cG, dz1);  // warp-uniform
      tc::tmem_ld_wait();
      float x[3];
      position(pick_tc(tt, j), x);
      const float4* er = nullptr;
      if (a.eik != nullptr && valid && a.cls[(size_t)rr * N + si] == CLS_FS) er = a.eik + (size_t)rr * N + si;
      const EikSeed es = eik_seed(er, a.eik_stride);
      if (valid && a.dz_out != nullptr) {  // the sample's record: dz (16), dcf (6), d direction (3), zeros (7)
        float4* rec = reinterpret_cast<float4*>(a.dz_out + ((size_t)rr * N + si) * 32);
        if (half == 0) {
#pragma unroll
          for (int q = 0; q < 4; ++q) rec[q] = make_float4(d[4 * q], d[4 * q + 1], d[4 * q + 2], d[4 * q + 3]);
        } else {
          rec[4] = make_float4(d[0], d[1], d[2], d[3]);
          rec[5] = make_float4(d[4], d[5], d[6], d[7]);
          rec[6] = make_float4(d[8], 0.f, 0.f, 0.f);
          rec[7] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      if (half == 0) {
        scatter_direct<false>(a.g, a.grad, 3, x, make_float4(d[12], d[13], d[14], d[15]), valid, es);
        scatter_direct<false>(a.g, a.grad, 2, x, make_float4(d[8], d[9], d[10], d[11]), valid, es);
      } else if (valid && (d[0] != 0.f || d[1] != 0.f || d[2] != 0.f || d[3] != 0.f || d[4] != 0.f || d[5] != 0.f)) {
        scatter_colour(a, x, d);  // a zero vector adds nothing
      }
      __syncwarp();
      tiles_free(T);  // their space holds the run reduction's staging rows
      {
        float4 g4 = half == 0 ? make_float4(d[0], d[1], d[2], d[3]) : make_float4(dz1[4], dz1[5], dz1[6], dz1[7]);
        if (!valid) g4 = make_float4(0.f, 0.f, 0.f, 0.f);
        scatter_runs(a.g, a.grad, half ? 1 : 0, x, g4, valid, reinterpret_cast<float*>(gmem) + w8 * kScatterStage, es);
      }
      group_sync<kTileThreads>(gi);  // every warp is done with its rows before the tiles are rewritten
    }
  }

  // ---- epilogue: loss sums, decoder-gradient partial row, tensor memory ----
  const bool done = tile_end(T, a.status, kStatusPaperRender) && alive;
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  float* prow = reinterpret_cast<float*>(base);  // the CTA's partial row, over group 0's tiles
  for (int i = tid; i < kPart; i += blockDim.x) prow[i] = 0.f;
  __syncthreads();
  if (BWD) {
    if (dw_acc && done) {
      // warp w (mod 4) holds rows 16 w .. 16 w + 15 of every M = 64 product in its lanes 0..15
      const int m = 16 * wq + lane, n1 = half ? kU : kZ;
      float d[32];
      tc::tmem_ld32(tq + (half ? cWc2 : cWg2), d);  // a1^T dY2, [r1 | 1]^T dQ2
      tc::tmem_ld_wait();
      if (lane < 16 && (m < 32 || (m == 32 && half != 0)))
#pragma unroll
        for (int n = 0; n < 32; ++n)
          atomicAdd(prow + (m < 32 ? (half ? A_cW2 : A_gW2) + n * kH + m : A_cb2 + n), d[n]);
      tc::tmem_ld32(tq + (half ? cWc1 : cWg1), d);  // [z | 1]^T dY1, [u | 1]^T dQ1
      tc::tmem_ld_wait();
      if (lane < 16 && m <= n1)
#pragma unroll
        for (int n = 0; n < 32; ++n)
          atomicAdd(prow + (m < n1 ? (half ? A_cW1 : A_gW1) + n * n1 + m : (half ? A_cb1 : A_gb1) + n), d[n]);
    }
    if (half == 0) {
      atomicAdd(prow + A_gw3 + lane, oacc[0]);
      atomicAdd(prow + A_gb2 + lane, oacc[1] * sc[sc_gw3 + lane]);
    } else {
#pragma unroll
      for (int i = 0; i < 3; ++i) atomicAdd(prow + A_cW3 + 32 * i + lane, oacc[i]);
    }
    __syncthreads();
  }
  auto total = [&](int k) {  // running sum k over the compositing warps
    float v = 0.f;
#pragma unroll
    for (int q = 0; q < kPGroups * 4; ++q) v += sums0[q * kPaperSums + k];
    return v;
  };
  for (int i = tid; i < kPart; i += blockDim.x) {
    float v = prow[i];
    if (i == A_kappa) v += total(4);
    else if (i >= A_cb3 && i < A_cb3 + 3) v += total(5 + i - A_cb3);
    else if (i == A_gb3) v += total(8);
    a.mlp_part[(size_t)blockIdx.x * kPart + i] = v;
  }
  if (tid < kLossPad) a.loss_part[(size_t)blockIdx.x * kLossPad + tid] = tid < 4 ? total(tid) : 0.f;
  __syncwarp();
  if (warp == 0) tc::tmem_dealloc(*tslot, kPTmem);
}
#pragma nv_diag_default 128

template <int NCH>
constexpr size_t paper_tc_smem() {
  constexpr size_t b = 128 + (size_t)kPGroups * kPGroupBytes + 3 * kTW + (size_t)kPGroups * NCH * 128 * 16 +
                       kPGroups * 20 * 16 + sizeof(float) * (kScal + 8 + kPGroups * 4 * kPaperSums) + 16;
  static_assert(b <= 227u * 1024u, "shared memory per CTA");
  return b;
}
static_assert(paper::kPart * 4 <= 3 * kAP, "the partial row fits in group 0's geometry tile");

template <int NCH>
gs_status launch_paper_tc(const PaperTcArgs& a, int mode, int ctas, cudaStream_t st) {
  constexpr size_t smem = paper_tc_smem<NCH>();
  auto k = mode == 1 ? paper_tc_kernel<NCH, true, false>
                     : (mode == 2 ? paper_tc_kernel<NCH, false, true> : paper_tc_kernel<NCH, true, true>);
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return GS_ERR_CUDA;
  k<<<ctas, kPThreads, smem, st>>>(a);
  return cudaPeekAtLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

}  // namespace ptc
}  // namespace gs
