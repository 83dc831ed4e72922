// SDF-gradient smoothness term (Sec. 3.3, Eq. smoothness_loss) and its second-order adjoint
// (Supp. Sec. 1): L_smooth = mean_p || grad phi(x_p) - grad phi(x_p + eps_p) ||^2 over S_g.
//
// grad_x phi = sum_l (1/v_l) J_l(x)^T p_l with p = d phi/d z = W1^T (m (.) W2[0,:]^T), m the
// ReLU mask (the decoder is piecewise linear, so p does not depend on z almost everywhere).
// For an adjoint a = dL/d(grad phi) at a point y:
//   d/d theta_{l,c,k} = p_{l,k} (1/v_l) (a . dw_c/df)       (Supp. Eq. second_order_theta)
//   d/d W1 = (m (.) W2[0,:]) j^T,  d/d W2[0,:] = m (.) (W1 j), j_k = a . d z_k / d x.
// One lane per evaluation; a warp stages its 32 evaluations' vectors and reduces the decoder
// gradients as 4x4 tiles.
//
// Bound by latency: 4096 points are one pass of every warp, in the render kernel's shadow only where that
// leaves SMs idle.  Hence one visit of the corners for z and dz/dx (three before: features, gradient
// and adjoint each gathered again), W1's rows read once as 16-byte vectors for the unit, its mask
// and its part of p, and the points dealt over the blocks first; 230 registers, no spill.  The term by
// itself, forward and backward, 300 / 4096 / 20000 / 100000 points: 43 / 49 / 133 / 507 us with three
// visits (192 registers), now 36 / 44 / 96 / 330; forward only, where that form spilled 948 bytes, 35 /
// 36 / 92 / 342 and now 27 / 27 / 49 / 140.
#include <algorithm>

#include "gs_internal.h"

namespace gs {

constexpr int kSmoothWarps = 2;  // static shared memory stays under 48 KB
constexpr int kSt = 84;  // staged row: mw2[32] | j[16] | u[32] (+4 pad), stride = 20 mod 32 banks
constexpr int sMw2 = 0, sJ = 32, sU = 48;

struct SmoothRunArgs {
  GridDesc g;
  const float* theta;
  int P;
  const float *xs, *eps;
  const uint8_t* valid;
  const int* counts;
  const float* dloss;
  float lam4;
  float* grad;
  float* loss_part;  // rows for this kernel's CTAs
  float* mlp_part;
};

__device__ __forceinline__ float4 ldv(const float* p) { return *reinterpret_cast<const float4*>(p); }

template <bool FWD, bool BWD>
__global__ void __launch_bounds__(kSmoothWarps * 32, 1) smooth_kernel(SmoothRunArgs a) {
  __shared__ __align__(16) float sm[kSmemMlp];
  __shared__ __align__(16) float acc[kMlpPad + kLossPad];
  __shared__ __align__(16) float stage[kSmoothWarps][32 * kSt];
  const float* mlp = a.theta + a.g.n_grid;
  for (int i = threadIdx.x; i < kSmemMlp; i += blockDim.x) {
    float v = 0.0f;
    if (i < sb1) v = mlp[oW1 + i];
    else if (i < sW2) v = mlp[ob1 + i - sb1];
    else if (i < sb2) v = mlp[oW2 + i - sW2];
    sm[i] = v;
  }
  for (int i = threadIdx.x; i < kMlpPad + kLossPad; i += blockDim.x) acc[i] = 0.0f;
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* st = stage[warp];
  const int n_g = a.counts[3];
  const float k_sm = n_g > 0 ? (a.dloss[4] + a.lam4 * a.dloss[5]) * 2.0f / (float)n_g : 0.0f;
  float l_sm = 0.f;

  // one lane per gradient evaluation: lanes 2q and 2q+1 evaluate point q at x and x + eps
#pragma unroll 1
  for (int base = (warp * gridDim.x + blockIdx.x) * 16; base < a.P; base += gridDim.x * kSmoothWarps * 16) {
    const int p = base + (lane >> 1), e = lane & 1;
    const bool valid = p < a.P && a.valid[p];
    float y[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) y[k] = valid ? (e == 0 ? a.xs[3 * p + k] : __fadd_rn(a.xs[3 * p + k], a.eps[3 * p + k])) : 0.f;
    float4 J[kLevels][3];
    float pz[kZ];           // p = d phi / d z
    unsigned mask = 0;      // ReLU mask m (bit j = unit j on)
    float* row = st + lane * kSt;
    {
      float z[kZ];
      features_jacobian(a.g, a.theta, y, z, J);
#pragma unroll
      for (int k = 0; k < kZ; ++k) pz[k] = 0.f;
#pragma unroll 2
      for (int j4 = 0; j4 < kH1; j4 += 4) {
        float mw[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float w[kZ];
          w1_row(sm, j4 + q, w);
          const bool on = w1_dot(w, z, sm[sb1 + j4 + q]) > 0.f;
          mw[q] = on ? sm[sW2 + j4 + q] : 0.f;
          mask |= (on ? 1u : 0u) << (j4 + q);
#pragma unroll
          for (int k = 0; k < kZ; ++k) pz[k] = fmaf(w[k], mw[q], pz[k]);
        }
        if (BWD) *reinterpret_cast<float4*>(row + sMw2 + j4) = make_float4(mw[0], mw[1], mw[2], mw[3]);
      }
    }
    float gq[3] = {0.f, 0.f, 0.f};  // grad_x phi = sum_l (dz_l/dx)^T p_l
#pragma unroll
    for (int l = 0; l < kLevels; ++l)
#pragma unroll
      for (int q = 0; q < 3; ++q)
        gq[q] += pz[4 * l] * J[l][q].x + pz[4 * l + 1] * J[l][q].y + pz[4 * l + 2] * J[l][q].z + pz[4 * l + 3] * J[l][q].w;
    float dg[3];  // g(x) - g(x + eps), on both lanes of the pair
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float other = __shfl_xor_sync(0xffffffffu, gq[q], 1);
      dg[q] = e == 0 ? gq[q] - other : other - gq[q];
    }
    if (FWD && valid && e == 0) l_sm += dg[0] * dg[0] + dg[1] * dg[1] + dg[2] * dg[2];
    if constexpr (!BWD) continue;
    const float sgn = e == 0 ? 1.f : -1.f;
    const float av[3] = {valid ? sgn * k_sm * dg[0] : 0.f, valid ? sgn * k_sm * dg[1] : 0.f,
                         valid ? sgn * k_sm * dg[2] : 0.f};
    float jv[kZ];  // j_l = a . dz_l/dx
#pragma unroll
    for (int l = 0; l < kLevels; ++l) {
      const float4 d0 = J[l][0], d1 = J[l][1], d2 = J[l][2];
      jv[4 * l] = av[0] * d0.x + av[1] * d1.x + av[2] * d2.x;
      jv[4 * l + 1] = av[0] * d0.y + av[1] * d1.y + av[2] * d2.y;
      jv[4 * l + 2] = av[0] * d0.z + av[1] * d1.z + av[2] * d2.z;
      jv[4 * l + 3] = av[0] * d0.w + av[1] * d1.w + av[2] * d2.w;
    }
    if (valid) {  // the direct term d/d theta_{l,c,k} = p_{l,k} (1/v_l) (a . dw_c/df)
#pragma unroll
      for (int l = 0; l < kLevels; ++l) {
        const Cell c = locate(a.g, l, y);
        float dw[8][3];
        corner_weight_grads(c.f, c.clamped, dw);
        const float iv = a.g.inv_voxel[l];
        const float4 p4 = make_float4(pz[4 * l], pz[4 * l + 1], pz[4 * l + 2], pz[4 * l + 3]);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float ad = (av[0] * dw[k][0] + av[1] * dw[k][1] + av[2] * dw[k][2]) * iv;
          atomicAdd(reinterpret_cast<float4*>(a.grad + a.g.off[l]) + c.vtx + corner_offset(a.g, l, k), f4scale(p4, ad));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      *reinterpret_cast<float4*>(row + sJ + 4 * q) = make_float4(jv[4 * q], jv[4 * q + 1], jv[4 * q + 2], jv[4 * q + 3]);
    // d/d W2[0][j] = m_j (W1 j)_j
#pragma unroll 2
    for (int j4 = 0; j4 < kH1; j4 += 4) {
      float u[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float w[kZ];
        w1_row(sm, j4 + q, w);
        u[q] = w1_dot(w, jv, 0.f);
        if (!((mask >> (j4 + q)) & 1u)) u[q] = 0.f;
      }
      *reinterpret_cast<float4*>(row + sU + j4) = make_float4(u[0], u[1], u[2], u[3]);
    }
    __syncwarp();
    {  // dW1[32][16] += mw2 (x) j over the warp's 32 evaluations
      const int i0 = 4 * (lane >> 2), j0 = 4 * (lane & 3);
      float t[4][4] = {};
#pragma unroll 4
      for (int s2 = 0; s2 < 32; ++s2) {
        const float4 av4 = ldv(st + s2 * kSt + sMw2 + i0), bv4 = ldv(st + s2 * kSt + sJ + j0);
        const float ar[4] = {av4.x, av4.y, av4.z, av4.w}, br[4] = {bv4.x, bv4.y, bv4.z, bv4.w};
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int q = 0; q < 4; ++q) t[x][q] = fmaf(ar[x], br[q], t[x][q]);
      }
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int q = 0; q < 4; ++q) atomicAdd(acc + oW1 + (i0 + x) * kZ + j0 + q, t[x][q]);
      float u = 0.f;  // dW2[0][lane] += sum_s u_s[lane]
#pragma unroll 4
      for (int s2 = 0; s2 < 32; ++s2) u += st[s2 * kSt + sU + lane];
      atomicAdd(acc + oW2 + lane, u);
    }
    __syncwarp();
  }
  if (FWD) {
    l_sm = warp_sum(l_sm);
    if (lane == 0) atomicAdd(acc + kMlpPad + 4, l_sm);
  }
  __syncthreads();
  if (threadIdx.x < kLossPad) a.loss_part[(size_t)blockIdx.x * kLossPad + threadIdx.x] = acc[kMlpPad + threadIdx.x];
  for (int i = threadIdx.x; i < kMlpPad; i += blockDim.x) a.mlp_part[(size_t)blockIdx.x * kMlpPad + i] = acc[i];
}

// ------------------------------------------------------------------------------------
// Reverse mode of the SDF query: grad += sum_p dsdf_p d phi(x_p)/d theta
//                                        + dgrad_p . d grad_x phi(x_p)/d theta.
// First order (Sec. 3.1): d phi/d z = p, so the grid gets p_{l,f} w_c and the decoder the
// usual dense-layer terms.  Second order (Supp. Sec. 1, as in the smoothness adjoint): with
// a = dgrad_p and j_k = a . d z_k/d x, the grid gets p_{l,f} (1/v_l)(a . d w_c/d f) and the
// decoder d/d W1 = (m (.) W2[0,:]) j^T, d/d W2[0,:] = m (.) (W1 j).  Combined per point:
//   dW1 += (m (.) W2[0,:]) (dsdf z + j)^T,  db1 += dsdf (m (.) W2[0,:]),
//   dW2[0,:] += dsdf a1 + m (.) (W1 j),     db2[0] += dsdf.
// One lane per point; the decoder gradients are reduced per warp as in the smoothness kernel.
// ------------------------------------------------------------------------------------
struct QueryBwdArgs {
  GridDesc g;
  const float* theta;
  const float* x;
  int P;
  const float* dsdf;   // [P] or nullptr
  const float* dgrad;  // [P][3] or nullptr
  float* grad;
};

// Large calls are bound by the reductions, 32 of 16 bytes a point, most of all by the ones that meet on
// the few vertices of the coarse levels.  Those come last, when the warps have drifted apart, and five
// CTAs per SM share them: 40000 / 300000 points of the room 101 / 515 us with the coarse levels first
// and eight CTAs, now 87 / 486; of the cube, whose levels are all crowded, 105 / 508, now 99 / 511.
constexpr int kQueryBwdCtasPerSm = 5;
__global__ void __launch_bounds__(kSmoothWarps * 32) query_backward_kernel(QueryBwdArgs a) {
  __shared__ __align__(16) float sm[kSmemMlp];
  __shared__ __align__(16) float acc[kH1 * kZ + kH1 + kH1 + 4];  // dW1 | db1 | dW2[0,:] | db2[0]
  __shared__ __align__(16) float stage[kSmoothWarps][32 * kSt];
  constexpr int aW1 = 0, ab1 = kH1 * kZ, aW2 = ab1 + kH1, ab2 = aW2 + kH1, kAcc = ab2 + 4;
  const float* mlp = a.theta + a.g.n_grid;
  for (int i = threadIdx.x; i < kSmemMlp; i += blockDim.x) {
    float v = 0.0f;
    if (i < sb1) v = mlp[oW1 + i];
    else if (i < sW2) v = mlp[ob1 + i - sb1];
    else if (i < sb2) v = mlp[oW2 + i - sW2];
    sm[i] = v;
  }
  for (int i = threadIdx.x; i < kAcc; i += blockDim.x) acc[i] = 0.0f;
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* st = stage[warp];
  float db2 = 0.f;
  for (int base = (blockIdx.x * kSmoothWarps + warp) * 32; base < a.P; base += gridDim.x * kSmoothWarps * 32) {
    const int p = base + lane;
    const bool valid = p < a.P;
    float y[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) y[k] = valid ? a.x[3 * p + k] : 0.f;
    const float ds = (valid && a.dsdf) ? a.dsdf[p] : 0.f;
    float av[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) av[k] = (valid && a.dgrad) ? a.dgrad[3 * p + k] : 0.f;
    float z[kZ], jv[kZ], pz[kZ];
    {
      float4 J[kLevels][3];
      features_jacobian(a.g, a.theta, y, z, J);
#pragma unroll
      for (int l = 0; l < kLevels; ++l) {
        const float4 d0 = J[l][0], d1 = J[l][1], d2 = J[l][2];
        jv[4 * l] = av[0] * d0.x + av[1] * d1.x + av[2] * d2.x;
        jv[4 * l + 1] = av[0] * d0.y + av[1] * d1.y + av[2] * d2.y;
        jv[4 * l + 2] = av[0] * d0.z + av[1] * d1.z + av[2] * d2.z;
        jv[4 * l + 3] = av[0] * d0.w + av[1] * d1.w + av[2] * d2.w;
        pz[4 * l] = pz[4 * l + 1] = pz[4 * l + 2] = pz[4 * l + 3] = 0.f;
      }
    }
    float* row = st + lane * kSt;
#pragma unroll 2
    for (int j4 = 0; j4 < kH1; j4 += 4) {
      float mw[4], u[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float w[kZ];
        w1_row(sm, j4 + q, w);
        const float s = w1_dot(w, z, sm[sb1 + j4 + q]), wj = w1_dot(w, jv, 0.f);
        mw[q] = s > 0.f ? sm[sW2 + j4 + q] : 0.f;
        u[q] = fmaf(ds, fmaxf(s, 0.f), s > 0.f ? wj : 0.f);
#pragma unroll
        for (int k = 0; k < kZ; ++k) pz[k] = fmaf(w[k], mw[q], pz[k]);
      }
      *reinterpret_cast<float4*>(row + sMw2 + j4) = make_float4(mw[0], mw[1], mw[2], mw[3]);
      *reinterpret_cast<float4*>(row + sU + j4) = make_float4(u[0], u[1], u[2], u[3]);
    }
    if (valid) {
#pragma unroll
      for (int l = kLevels - 1; l >= 0; --l) {  // the crowded coarse levels last
        const Cell c = locate(a.g, l, y);
        float dw[8][3], w[8];
        corner_weights(c.f, w);
        corner_weight_grads(c.f, c.clamped, dw);
        const float iv = a.g.inv_voxel[l];
        const float4 p4 = make_float4(pz[4 * l], pz[4 * l + 1], pz[4 * l + 2], pz[4 * l + 3]);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float coef = ds * w[k] + (av[0] * dw[k][0] + av[1] * dw[k][1] + av[2] * dw[k][2]) * iv;
          atomicAdd(reinterpret_cast<float4*>(a.grad + a.g.off[l]) + c.vtx + corner_offset(a.g, l, k), f4scale(p4, coef));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      *reinterpret_cast<float4*>(row + sJ + 4 * q) =
          make_float4(fmaf(ds, z[4 * q], jv[4 * q]), fmaf(ds, z[4 * q + 1], jv[4 * q + 1]),
                      fmaf(ds, z[4 * q + 2], jv[4 * q + 2]), fmaf(ds, z[4 * q + 3], jv[4 * q + 3]));
    row[80] = ds;
    db2 += ds;
    __syncwarp();
    {  // dW1[32][16] += mw2 (x) (ds z + j) over the warp's 32 points; dW2[0][lane], db1[lane]
      const int i0 = 4 * (lane >> 2), j0 = 4 * (lane & 3);
      float t[4][4] = {};
#pragma unroll 4
      for (int s2 = 0; s2 < 32; ++s2) {
        const float4 av4 = ldv(st + s2 * kSt + sMw2 + i0), bv4 = ldv(st + s2 * kSt + sJ + j0);
        const float ar[4] = {av4.x, av4.y, av4.z, av4.w}, br[4] = {bv4.x, bv4.y, bv4.z, bv4.w};
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int q = 0; q < 4; ++q) t[x][q] = fmaf(ar[x], br[q], t[x][q]);
      }
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int q = 0; q < 4; ++q) atomicAdd(acc + aW1 + (i0 + x) * kZ + j0 + q, t[x][q]);
      float u = 0.f, b = 0.f;
#pragma unroll 4
      for (int s2 = 0; s2 < 32; ++s2) {
        u += st[s2 * kSt + sU + lane];
        b = fmaf(st[s2 * kSt + 80], st[s2 * kSt + sMw2 + lane], b);
      }
      atomicAdd(acc + aW2 + lane, u);
      atomicAdd(acc + ab1 + lane, b);
    }
    __syncwarp();
  }
  db2 = warp_sum(db2);
  if (lane == 0) atomicAdd(acc + ab2, db2);
  __syncthreads();
  float* gm = a.grad + a.g.n_grid;
  for (int i = threadIdx.x; i < kAcc; i += blockDim.x) {
    const float v = acc[i];
    if (v == 0.f) continue;
    if (i < ab1) atomicAdd(gm + oW1 + i, v);
    else if (i < aW2) atomicAdd(gm + ob1 + i - ab1, v);
    else if (i < ab2) atomicAdd(gm + oW2 + i - aW2, v);  // row 0 of W2
    else if (i == ab2) atomicAdd(gm + ob2, v);
  }
}

}  // namespace gs

using namespace gs;

gs_status gs_launch_query_backward(const gs_ctx* ctx, const float* theta, const float* x, int P, const float* dsdf,
                                   const float* dgrad, float* grad, cudaStream_t st) {
  if (P <= 0 || (!dsdf && !dgrad)) return GS_OK;
  QueryBwdArgs a;
  a.g = ctx->grid;
  a.theta = theta;
  a.x = x;
  a.P = P;
  a.dsdf = dsdf;
  a.dgrad = dgrad;
  a.grad = grad;
  const int per = kSmoothWarps * 32;
  const int blocks = (int)std::min<long long>(((long long)P + per - 1) / per, (long long)kQueryBwdCtasPerSm * ctx->num_sms);
  query_backward_kernel<<<blocks, per, 0, st>>>(a);
  return cudaPeekAtLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

gs_status gs_launch_smooth(const gs_ctx* ctx, const float* theta, const gs_batch* b, const float* dloss, float* grad,
                           int mode, cudaStream_t st) {
  if (b->P <= 0) return GS_OK;
  SmoothRunArgs a;
  a.g = ctx->grid;
  a.theta = theta;
  a.P = b->P;
  a.xs = b->xs;
  a.eps = b->eps;
  a.valid = b->valid;
  a.counts = b->counts;
  a.dloss = dloss;
  a.lam4 = ctx->cfg.lam[4];
  a.grad = grad;
  a.loss_part = ctx->loss_part + (size_t)ctx->render_ctas * kLossPad;
  a.mlp_part = ctx->mlp_part + (size_t)ctx->render_ctas * kMlpPad;
  if (mode == 1) smooth_kernel<true, false><<<kSmoothCtas, kSmoothWarps * 32, 0, st>>>(a);
  else if (mode == 2) smooth_kernel<false, true><<<kSmoothCtas, kSmoothWarps * 32, 0, st>>>(a);
  else smooth_kernel<true, true><<<kSmoothCtas, kSmoothWarps * 32, 0, st>>>(a);
  return cudaPeekAtLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}
