// Direct transform core shared by k_dft (k_dft.cu) and k_dft_partials (wst_noalloc.cu):
// the exact dirty image at a few pixels (the conjugate of Eq. 1 summed over the
// visibilities), phases u l + v m + w (n-1) formed from float-float l, m, n-1 with the
// whole cycles taken out product by product (phase_frac) before an FP32 sincospi, so a
// phase of thousands of cycles keeps the accuracy of one below a cycle.
#pragma once

#include "wst_internal.cuh"

namespace wst {

constexpr int kDftPix = 8;  // pixels per CTA (every thread evaluates all of them)
constexpr int kDftThreads = 256;

struct PixelLMN {
  ff l, m, t;
};

__device__ __forceinline__ ff ff_from_double(double d) {
  float2 s = ff_split(d);
  return {s.x, s.y};
}

// u l + v m + w t modulo whole cycles, as one FP32 number of magnitude about 1/2 or less.
// Each product's leading part is exact as p + e (the product and its fused residual), and
// p - rint(p) is exact, so the whole cycles leave each product before any sum is rounded;
// the residuals and the low words' products are small and summed in FP32.  The sum of the
// three fractions is exact unless a product is itself below a cycle or two; its error is
// then at most 2^-24 cycle, that of the FP32 argument sincospi takes.  The kernels are bound
// by FP32 issue; float-float products and sums of the whole phase took 1360 us for 2e5
// visibilities at 2048 pixels, this (with the pixels' set-up once per CTA) 825 us, at an
// error against FP64 of 2.7e-7 instead of 3.1e-7.
__device__ __forceinline__ float phase_frac(float u, float v, float w, const ff &l, const ff &m, const ff &t) {
  const float pu = __fmul_rn(u, l.hi), pv = __fmul_rn(v, m.hi), pw = __fmul_rn(w, t.hi);
  float e = __fmaf_rn(u, l.lo, __fmaf_rn(u, l.hi, -pu));
  e = __fmaf_rn(v, m.lo, __fadd_rn(e, __fmaf_rn(v, m.hi, -pv)));
  e = __fmaf_rn(w, t.lo, __fadd_rn(e, __fmaf_rn(w, t.hi, -pw)));
  const float a = __fsub_rn(pu, rintf(pu)), b = __fsub_rn(pv, rintf(pv)), c = __fsub_rn(pw, rintf(pw));
  const float s = __fadd_rn(__fadd_rn(a, b), c);
  return __fadd_rn(__fsub_rn(s, rintf(s)), e);
}

// exp(2 pi i phi) of a phase given in cycles
__device__ __forceinline__ float2 cis_cycles(float phi) {
  float s, c;
  sincospif(2.0f * phi, &s, &c);
  return make_float2(c, s);
}

// The CTA's share of out_i = sum_j w_j V_j exp(2 pi i (u_j l_i + v_j m_i + w_j (n_i - 1)))
// for the kDftPix pixels pix0 .. pix0 + kDftPix - 1 (those below n_pix): the visibilities
// j = blockIdx.x * kDftThreads + threadIdx.x + k * gridDim.x * kDftThreads, skipping any
// with a non-finite coordinate, value or weight.  Pixels outside the unit sphere get 0.
// Thread i < kDftPix returns the CTA's sum for pixel pix0 + i (summed in a fixed order:
// a warp butterfly, then the warps in index order); other threads return 0.  Every
// thread of the CTA must call it (it synchronises the CTA).
__device__ __forceinline__ float2 dft_cta_partial(int64_t n_vis, const float *__restrict__ u,
                                                  const float *__restrict__ v, const float *__restrict__ w,
                                                  const float2 *__restrict__ vis, const float *__restrict__ weight,
                                                  int n, double dl, int64_t n_pix, const int32_t *__restrict__ pa,
                                                  const int32_t *__restrict__ pb, int64_t pix0) {
  // the pixels' l, m, n - 1: one thread each (the FP64 root and division are slow here,
  // and every thread of the CTA needs the same eight)
  __shared__ PixelLMN s_px[kDftPix];
  __shared__ bool s_valid[kDftPix];
  if (threadIdx.x < kDftPix) {
    const int64_t q = pix0 + threadIdx.x;
    bool valid = false;
    PixelLMN p;
    p.l = p.m = p.t = {0.0f, 0.0f};
    if (q < n_pix) {
      const double l = (double)(pa[q] - n / 2) * dl, m = (double)(pb[q] - n / 2) * dl;
      const double r2 = l * l + m * m;
      if (r2 < 1.0) {
        valid = true;
        p.l = ff_from_double(l);
        p.m = ff_from_double(m);
        p.t = ff_from_double(-r2 / (1.0 + sqrt(1.0 - r2)));
      }
    }
    s_px[threadIdx.x] = p;
    s_valid[threadIdx.x] = valid;
  }
  __syncthreads();
  PixelLMN px[kDftPix];
#pragma unroll
  for (int i = 0; i < kDftPix; ++i) px[i] = s_px[i];
  float2 acc[kDftPix];
#pragma unroll
  for (int i = 0; i < kDftPix; ++i) acc[i] = make_float2(0.0f, 0.0f);
  for (int64_t j = (int64_t)blockIdx.x * kDftThreads + threadIdx.x; j < n_vis;
       j += (int64_t)gridDim.x * kDftThreads) {
    const float uf = u[j], vf = v[j], wf = w[j];
    float2 val = vis[j];
    const float wt = weight ? weight[j] : 1.0f;
    if (!(isfinite(uf) && isfinite(vf) && isfinite(wf) && isfinite(val.x) && isfinite(val.y) && isfinite(wt)))
      continue;
    val = make_float2(val.x * wt, val.y * wt);
#pragma unroll
    for (int i = 0; i < kDftPix; ++i) {
      const float2 e = cis_cycles(phase_frac(uf, vf, wf, px[i].l, px[i].m, px[i].t));
      acc[i].x = fmaf(val.x, e.x, fmaf(-val.y, e.y, acc[i].x));
      acc[i].y = fmaf(val.x, e.y, fmaf(val.y, e.x, acc[i].y));
    }
  }
  __shared__ float2 red[kDftThreads / 32][kDftPix];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < kDftPix; ++i) {
    float x = acc[i].x, y = acc[i].y;
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
      y += __shfl_xor_sync(0xFFFFFFFFu, y, o);
    }
    if (lane == 0) red[wid][i] = make_float2(x, y);
  }
  __syncthreads();
  float2 s = make_float2(0.0f, 0.0f);
  if (threadIdx.x < kDftPix && s_valid[threadIdx.x])
    for (int k = 0; k < kDftThreads / 32; ++k) s = make_float2(s.x + red[k][threadIdx.x].x, s.y + red[k][threadIdx.x].y);
  return s;
}

}  // namespace wst
