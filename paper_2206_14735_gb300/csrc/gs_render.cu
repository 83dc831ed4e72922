// Loss / decoder-gradient combination, SDF query and cell lookup, and the dispatch of the
// fused render kernel over samples-per-ray (its instantiations live in gs_render_tc_n*.cu).
#include "gs_render_tc.cuh"

namespace gs {

extern template gs_status launch_tc_n<PrecBF16x3, 1>(const gs_ctx*, RenderTcArgs&, int, cudaStream_t);
extern template gs_status launch_tc_n<PrecBF16x3, 2>(const gs_ctx*, RenderTcArgs&, int, cudaStream_t);
extern template gs_status launch_tc_n<PrecBF16x3, 3>(const gs_ctx*, RenderTcArgs&, int, cudaStream_t);
extern template gs_status launch_tc_n<PrecBF16x3, 4>(const gs_ctx*, RenderTcArgs&, int, cudaStream_t);
extern template gs_status launch_tc_n<PrecBF16x3, 5>(const gs_ctx*, RenderTcArgs&, int, cudaStream_t);
extern template gs_status launch_tc_n<PrecBF16, 1>(const gs_ctx*, RenderTcArgs&, int, cudaStream_t);
extern template gs_status launch_tc_n<PrecBF16, 2>(const gs_ctx*, RenderTcArgs&, int, cudaStream_t);
extern template gs_status launch_tc_n<PrecBF16, 3>(const gs_ctx*, RenderTcArgs&, int, cudaStream_t);
extern template gs_status launch_tc_n<PrecBF16, 4>(const gs_ctx*, RenderTcArgs&, int, cudaStream_t);
extern template gs_status launch_tc_n<PrecBF16, 5>(const gs_ctx*, RenderTcArgs&, int, cudaStream_t);

// ------------------------------------------------------------------------------------
// combine per-CTA partials: losses in FP64, decoder gradients in a fixed order
// ------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) finalize_kernel(const float* loss_part, const float* mlp_part, int nparts,
                                                       const int* counts, int R, float l0, float l1, float l2,
                                                       float l3, float l4, float* loss, float* gmlp) {
  // decoder gradients: block b owns entries [32b, 32b + 32); warp w sums rows w, w + 8, ...,
  // then warp 0 adds the 8 warps' sums in a fixed order
  __shared__ float part[8][33];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  if (gmlp) {
    part[wid][lane] = i < GS_MLP_PARAMS ? column_sum8(mlp_part, kMlpPad, i, wid, nparts) : 0.f;
    __syncthreads();
    if (wid == 0 && i < GS_MLP_PARAMS) {
      float t = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) t += part[k][lane];
      gmlp[i] += t;
    }
  }
  // losses (FP64): lane l of warp 0 sums rows l, l + 32, ... of every term, then a warp sum
  if (loss && blockIdx.x == 0 && threadIdx.x < 32) {
    double s[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int p = lane; p < nparts; p += 32)
#pragma unroll
      for (int k = 0; k < 5; ++k) s[k] += (double)loss_part[(size_t)p * kLossPad + k];
#pragma unroll
    for (int k = 0; k < 5; ++k)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
    if (lane == 0) {
      const double den[5] = {(double)R, (double)counts[0], (double)counts[1], (double)counts[2], (double)counts[3]};
      const double lam[5] = {l0, l1, l2, l3, l4};
      double tot = 0.0;
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const double v = den[k] > 0 ? s[k] / den[k] : 0.0;
        loss[k] = (float)v;
        tot += lam[k] * v;
      }
      loss[5] = (float)tot;
    }
  }
}

// ------------------------------------------------------------------------------------
// SDF query and cell lookup
// ------------------------------------------------------------------------------------
// Bound by the latency of its gathers; W1's rows are read once, as 16-byte vectors, for a unit and its
// part of p.  Room, 4096 / 40000 / 300000 points with the gradient: 23 / 50 / 167 us with a read per use
// and 1.5 KB of spills, now 17 / 21 / 60 (blocks of 64 threads, each with its own copy of the decoder,
// took 19 / 23 / 66).
__global__ void __launch_bounds__(128) query_kernel(GridDesc g, const float* __restrict__ theta, const float* __restrict__ xq, int P,
                             float* sdf, float* grad) {
  __shared__ __align__(16) float sm[sb2 + 1];
  const float* mlp = theta + g.n_grid;
  for (int i = threadIdx.x; i <= sb2; i += blockDim.x) {
    float v = 0.0f;
    if (i < sb1) v = mlp[oW1 + i];
    else if (i < sW2) v = mlp[ob1 + i - sb1];
    else if (i < sb2) v = mlp[oW2 + i - sW2];
    else v = mlp[ob2];
    sm[i] = v;
  }
  __syncthreads();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  const float x[3] = {xq[3 * p], xq[3 * p + 1], xq[3 * p + 2]};
  float z[kZ], pz[kZ];  // pz = d phi / d z
  float4 J[kLevels][3];
  features_jacobian(g, theta, x, z, J);
#pragma unroll
  for (int k = 0; k < kZ; ++k) pz[k] = 0.f;
  float phi = sm[sb2];
#pragma unroll 4
  for (int j = 0; j < kH1; ++j) {
    float w[kZ];
    w1_row(sm, j, w);
    const float s = w1_dot(w, z, sm[sb1 + j]), mw = s > 0.f ? sm[sW2 + j] : 0.f;
    phi = fmaf(sm[sW2 + j], fmaxf(s, 0.f), phi);
#pragma unroll
    for (int k = 0; k < kZ; ++k) pz[k] = fmaf(w[k], mw, pz[k]);
  }
  sdf[p] = phi;
  if (grad) {
    float gxyz[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      float v = 0.f;
#pragma unroll
      for (int l = 0; l < kLevels; ++l) {
        v = fmaf(pz[4 * l], J[l][q].x, v);
        v = fmaf(pz[4 * l + 1], J[l][q].y, v);
        v = fmaf(pz[4 * l + 2], J[l][q].z, v);
        v = fmaf(pz[4 * l + 3], J[l][q].w, v);
      }
      gxyz[q] = v;
    }
    grad[3 * p] = gxyz[0];
    grad[3 * p + 1] = gxyz[1];
    grad[3 * p + 2] = gxyz[2];
  }
}

__global__ void voxel_index_kernel(GridDesc g, const float* __restrict__ xq, int P, long long* out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  const float x[3] = {xq[3 * p], xq[3 * p + 1], xq[3 * p + 2]};
#pragma unroll
  for (int l = 0; l < kLevels; ++l) out[(size_t)kLevels * p + l] = locate(g, l, x).vtx;
}

}  // namespace gs

using namespace gs;

gs_status gs_launch_render(const gs_ctx* ctx, const float* theta, const uint16_t* theta_bf16, const gs_batch* b,
                           const float* dloss, float* grad, float* rgb_hat, float* d_hat, float* wsum, int mode,
                           cudaStream_t st) {
  RenderTcArgs a;
  a.g = ctx->grid;
  a.theta = theta;
  a.theta_bf16 = theta_bf16;
  a.R = b->R;
  a.N = b->N;
  a.o = b->origin;
  a.r = b->dir;
  a.rgb = b->rgb;
  a.D = b->depth;
  a.t = b->t;
  a.cls = b->cls;
  a.counts = b->counts;
  a.dloss = dloss;
  for (int k = 0; k < 5; ++k) a.lam[k] = ctx->cfg.lam[k];
  a.kappa_fs = ctx->cfg.kappa_fs;
  a.grad = grad;
  a.loss_part = ctx->loss_part;
  a.mlp_part = ctx->mlp_part;
  a.rgb_hat = rgb_hat;
  a.d_hat = d_hat;
  a.wsum = wsum;
  a.status = ctx->status;
  a.store = ctx->store;
  a.w_out = b->w;
  a.dz_out = b->dz;
  a.eik = reinterpret_cast<const float4*>(b->eik);
  a.eik_stride = (long long)b->R * b->N;
  const int nch = (b->N + 31) / 32;
  if (ctx->cfg.precision == GS_PREC_BF16) {
    switch (nch) {
      case 1: return launch_tc_n<PrecBF16, 1>(ctx, a, mode, st);
      case 2: return launch_tc_n<PrecBF16, 2>(ctx, a, mode, st);
      case 3: return launch_tc_n<PrecBF16, 3>(ctx, a, mode, st);
      case 4: return launch_tc_n<PrecBF16, 4>(ctx, a, mode, st);
      case 5: return launch_tc_n<PrecBF16, 5>(ctx, a, mode, st);
      default: return GS_ERR_UNSUPPORTED;
    }
  }
  switch (nch) {
    case 1: return launch_tc_n<PrecBF16x3, 1>(ctx, a, mode, st);
    case 2: return launch_tc_n<PrecBF16x3, 2>(ctx, a, mode, st);
    case 3: return launch_tc_n<PrecBF16x3, 3>(ctx, a, mode, st);
    case 4: return launch_tc_n<PrecBF16x3, 4>(ctx, a, mode, st);
    case 5: return launch_tc_n<PrecBF16x3, 5>(ctx, a, mode, st);
    default: return GS_ERR_UNSUPPORTED;
  }
}

gs_status gs_launch_finalize(const gs_ctx* ctx, const gs_batch* b, float* loss, float* grad, int mode,
                             cudaStream_t st) {
  const float* l = ctx->cfg.lam;
  float* gmlp = (mode & 2) ? grad + ctx->grid.n_grid : nullptr;
  float* lo = (mode & 1) ? loss : nullptr;
  finalize_kernel<<<(GS_MLP_PARAMS + 31) / 32, 256, 0, st>>>(ctx->loss_part, ctx->mlp_part, ctx->n_parts,
                                                                b->counts, b->R, l[0], l[1], l[2], l[3], l[4], lo,
                                                                gmlp);
  return cudaPeekAtLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

gs_status gs_launch_query(const gs_ctx* ctx, const float* theta, const float* x, int P, float* sdf, float* grad,
                          cudaStream_t st) {
  if (P > 0) query_kernel<<<(P + 127) / 128, 128, 0, st>>>(ctx->grid, theta, x, P, sdf, grad);
  return cudaPeekAtLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

gs_status gs_launch_voxel_index(const gs_ctx* ctx, const float* x, int P, long long* out, cudaStream_t st) {
  if (P > 0) voxel_index_kernel<<<(P + 127) / 128, 128, 0, st>>>(ctx->grid, x, P, out);
  return cudaPeekAtLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}
