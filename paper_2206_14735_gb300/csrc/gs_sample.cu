// Ray batch sampling, sample placement and bound classes (Sec. 3.2-3.4), and the
// near-surface smoothness points S_g (Sec. 3.3).  Every value here is computed with
// explicitly rounded binary32 operations so that it is reproducible bit for bit.
#include "gs_sample.cuh"

namespace gs {

struct SampleArgs {
  FramesDev fr;
  uint64_t seed;
  uint32_t step;
  int R, Ns, Ng;
  float near_m, far_m, guide_half, trunc;
  long long* pix;
  float *o, *r, *rgb, *D, *t;
  uint8_t* cls;
  int* counts;
};

struct SmoothArgs {
  FramesDev fr;
  uint64_t seed;
  uint32_t step;
  int P;
  float trunc, delta_s;
  float *xs, *eps;
  uint8_t* valid;
  int* counts;
};

// S_g: back-projected observed depth of a random valid pixel (up to 8 draws) jittered by
// +-t per axis; eps of length delta_s in a direction drawn by rejection from [-1,1]^3.
__device__ __forceinline__ void sample_smooth_point(const SmoothArgs& a, int p) {
  int nv = 0;
  if (p < a.P) {
    const uint64_t pre = draw_prefix(a.seed, 1, a.step, (uint64_t)p);
    const long long npix = (long long)a.fr.F * a.fr.H * a.fr.W;
    long long px = -1;
    for (int tr = 0; tr < 8; ++tr) {
      const long long q = (long long)(draw_slot(pre, (uint64_t)tr) % (uint64_t)npix);
      if (a.fr.depth[q] > 0.0f) {
        px = q;
        break;
      }
    }
    if (px < 0) {
      a.valid[p] = 0;
#pragma unroll
      for (int k = 0; k < 3; ++k) a.xs[3 * p + k] = a.eps[3 * p + k] = 0.0f;
    } else {
      nv = 1;
      a.valid[p] = 1;
      float o[3], r[3], rgb[3], D;
      pixel_ray(a.fr, px, o, r, rgb, &D);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float u = unif24(draw_slot(pre, 16 + (uint64_t)k));
        const float base = __fadd_rn(o[k], __fmul_rn(D, r[k]));
        const float jit = __fmul_rn(a.trunc, __fsub_rn(__fmul_rn(2.0f, u), 1.0f));
        a.xs[3 * p + k] = __fadd_rn(base, jit);
      }
      float v[3] = {1.0f, 0.0f, 0.0f}, n2 = 1.0f;
      for (int tr = 0; tr < 16; ++tr) {
        float w[3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
          w[k] = __fsub_rn(__fmul_rn(2.0f, unif24(draw_slot(pre, 32 + 3 * (uint64_t)tr + k))), 1.0f);
        const float q = __fadd_rn(__fadd_rn(__fmul_rn(w[0], w[0]), __fmul_rn(w[1], w[1])), __fmul_rn(w[2], w[2]));
        if (q >= 0.01f && q <= 1.0f) {
          v[0] = w[0];
          v[1] = w[1];
          v[2] = w[2];
          n2 = q;
          break;
        }
      }
      const float sc = __fdiv_rn(a.delta_s, __fsqrt_rn(n2));
#pragma unroll
      for (int k = 0; k < 3; ++k) a.eps[3 * p + k] = __fmul_rn(v[k], sc);
    }
  }
  nv = __reduce_add_sync(0xffffffffu, nv);
  if ((threadIdx.x & 31) == 0 && nv) atomicAdd(a.counts + 3, nv);
}

__global__ void __launch_bounds__(128) sample_smooth_kernel(SmoothArgs a) {
  sample_smooth_point(a, blockIdx.x * blockDim.x + threadIdx.x);
}

// One warp per ray, its samples over the lanes, and behind the rays' blocks one thread per
// smoothness point.  A thread per ray drew and merged its 96 samples one after the other on 8 blocks
// or 64: 28.7 us a call at 1024 x 64 and 33.2 us at 8192 x 96 with 4096 points; now 12.3 and 16.5.  The
// counts are summed over a block first: one atomic per warp and count was 24 us of atomics on four
// words at 8192 rays.
// The two sorted lists merge by rank: a stratified sample follows the guided ones below it, a
// guided one the stratified ones up to it (ties stratified first), so a sample's place is its own
// index plus one binary search in the other list.  Both searches ask the merge's own question,
// "stratified <= guided", so the places are all different for any depths (an infinite guide_half
// makes the guided ones NaN, which go first).
constexpr int kSampleWarps = 16;
__global__ void __launch_bounds__(kSampleWarps * 32) sample_rays_kernel(SampleArgs a, SmoothArgs sm, int ray_blocks) {
  __shared__ float list[kSampleWarps][GS_MAX_SAMPLES];
  if ((int)blockIdx.x >= ray_blocks) {
    sample_smooth_point(sm, ((int)blockIdx.x - ray_blocks) * blockDim.x + threadIdx.x);
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * kSampleWarps + warp;
  int nd = 0, ntr = 0, nfs = 0;
  if (i < a.R) {
    const uint64_t pre = draw_prefix(a.seed, 0, a.step, (uint64_t)i);
    const long long npix = (long long)a.fr.F * a.fr.H * a.fr.W;
    const long long p = (long long)(draw_slot(pre, 0) % (uint64_t)npix);
    float o[3], r[3], rgb[3], D;
    pixel_ray(a.fr, p, o, r, rgb, &D);
    if (lane == 0) {
      a.pix[i] = p;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        a.o[3 * i + k] = o[k];
        a.r[3 * i + k] = r[k];
        a.rgb[3 * i + k] = rgb[k];
      }
      a.D[i] = D;
      nd = D > 0.0f;
    }
    const int N = a.Ns + a.Ng;
    float* ti = a.t + (size_t)i * N;
    uint8_t* ci = a.cls + (size_t)i * N;
    if (D > 0.0f) {
      // N_s strata of [near, far] (slots 1 ..) and N_g strata of [D - g, D + g], merged by depth
      const float delta = __fdiv_rn(__fsub_rn(a.far_m, a.near_m), (float)a.Ns);
      const float gstep = __fdiv_rn(__fmul_rn(2.0f, a.guide_half), (float)a.Ng);
      const float g0 = __fsub_rn(D, a.guide_half);
      float* l = list[warp];
      for (int k = lane; k < N; k += 32) {
        const float u = unif24(draw_slot(pre, 1 + (uint64_t)k));
        l[k] = k < a.Ns ? __fadd_rn(a.near_m, __fmul_rn(__fadd_rn((float)k, u), delta))
                        : __fadd_rn(g0, __fmul_rn(__fadd_rn((float)(k - a.Ns), u), gstep));
      }
      __syncwarp();
      for (int k = lane; k < N; k += 32) {
        const bool strat = k < a.Ns;
        const float tk = l[k];
        int lo = strat ? a.Ns : 0, hi = strat ? N : a.Ns;  // first of the other list that comes after
        const int base = lo;
        while (lo < hi) {
          const int m = (lo + hi) >> 1;
          if (strat ? !(tk <= l[m]) : l[m] <= tk) lo = m + 1;
          else hi = m;
        }
        const int at = (strat ? k : k - a.Ns) + lo - base;
        ti[at] = tk;
        const int c = sample_class(D, tk, a.trunc);
        ci[at] = (uint8_t)c;
        ntr += c == CLS_TR;
        nfs += c == CLS_FS;
      }
    } else {
      const float delta = __fdiv_rn(__fsub_rn(a.far_m, a.near_m), (float)N);
      for (int k = lane; k < N; k += 32) {
        const float u = unif24(draw_slot(pre, 1 + (uint64_t)k));
        ti[k] = __fadd_rn(a.near_m, __fmul_rn(__fadd_rn((float)k, u), delta));
        ci[k] = (uint8_t)CLS_NONE;
      }
    }
  }
  add_counts_per_block(a.counts, nd, ntr, nfs);
}

}  // namespace gs

using namespace gs;

static SmoothArgs smooth_args(const gs_ctx* ctx, const gs_frames* f, uint64_t seed, uint32_t step, const gs_batch* b) {
  FramesDev fr{f->F, f->H, f->W, f->rgb, f->depth, f->c2w, f->fx, f->fy, f->cx, f->cy};
  return SmoothArgs{fr, seed, step, b->P, ctx->cfg.trunc, ctx->cfg.delta_s, b->xs, b->eps, b->valid, b->counts};
}

gs_status gs_launch_sample_smooth(const gs_ctx* ctx, const gs_frames* f, uint64_t seed, uint32_t step,
                                  const gs_batch* b, cudaStream_t st) {
  if (b->P > 0) sample_smooth_kernel<<<(b->P + 127) / 128, 128, 0, st>>>(smooth_args(ctx, f, seed, step, b));
  return cudaPeekAtLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

gs_status gs_launch_sample(const gs_ctx* ctx, const gs_frames* f, uint64_t seed, uint32_t step, const gs_batch* b,
                           cudaStream_t st) {
  FramesDev fr{f->F, f->H, f->W, f->rgb, f->depth, f->c2w, f->fx, f->fy, f->cx, f->cy};
  if (cudaMemsetAsync(b->counts, 0, 4 * sizeof(int), st) != cudaSuccess) return GS_ERR_CUDA;
  SampleArgs a{fr,     seed,   step,   b->R,   ctx->cfg.n_strat, ctx->cfg.n_guided, ctx->cfg.near_m,
               ctx->cfg.far_m, ctx->cfg.guide_half, ctx->cfg.trunc, (long long*)b->pix, b->origin, b->dir,
               b->rgb, b->depth, b->t, b->cls, b->counts};
  const int ray_blocks = (b->R + kSampleWarps - 1) / kSampleWarps, blocks = ray_blocks + (b->P + kSampleWarps * 32 - 1) / (kSampleWarps * 32);
  if (blocks > 0) sample_rays_kernel<<<blocks, kSampleWarps * 32, 0, st>>>(a, smooth_args(ctx, f, seed, step, b), ray_blocks);
  return cudaPeekAtLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}
