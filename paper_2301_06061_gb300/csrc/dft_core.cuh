// Direct transform core shared by k_dft (k_dft.cu) and k_dft_partials (wst_noalloc.cu):
// the exact dirty image at a few pixels (the conjugate of Eq. 1 summed over the
// visibilities), phases u l + v m + w (n-1) formed in float-float (l, m, n-1 carried as
// float-float) and reduced modulo one cycle before the FP32 sine and cosine (cis_small,
// cis_any), so a phase of thousands of cycles keeps the accuracy of one below a cycle.
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

// exp(2 pi i (u l + v m + w t)) for |u|, |v|, |w| <= kCisMax and |l|, |m|, |t| <= 1
//
// The phase as a float-float sum without its renormalisations: the products u l.hi with their
// exact remainders (two_prod), summed exactly (two_sum); the remainders and the low words'
// products go into one low word.  s + M, M = 1.5 2^22, rounds the high word (below 2^21 in
// size) to a multiple of 1/2 whose last bit is its parity; what is left, at most 1/4, and
// the low word are added with the phase's one rounding: 1.5e-8 cycle at most, 3.3e-9 rms (the
// phase as a float-float reduced to half a cycle: 3.0e-8, 6.5e-9).  The kernel is bound by
// instruction issue, most of it on the FP32 pipe: 2e5 visibilities at 2048 pixels and 25
// sources 766 us.  With whole float-float operations and sincospi (cis_any), part of it on a
// slower pipe, 1367 us; with each product rounded after its half cycles are taken out and
// plain sums, phases 7e-8 cycle off, 640 us.
constexpr float kCisMax = 0x1p+19f;
__device__ __forceinline__ float2 cis_small(float u, float v, float w, const ff &l, const ff &m, const ff &t) {
  constexpr float M = 6291456.0f;
  const float pu = __fmul_rn(u, l.hi), pv = __fmul_rn(v, m.hi), pw = __fmul_rn(w, t.hi);
  const float eu = __fmaf_rn(u, l.lo, __fmaf_rn(u, l.hi, -pu));
  const float ev = __fmaf_rn(v, m.lo, __fmaf_rn(v, m.hi, -pv));
  const float ew = __fmaf_rn(w, t.lo, __fmaf_rn(w, t.hi, -pw));
  const ff a = two_sum(pu, pv), b = two_sum(a.hi, pw);
  const float e = __fadd_rn(__fadd_rn(eu, ev), __fadd_rn(ew, __fadd_rn(a.lo, b.lo)));
  const float ts = __fadd_rn(b.hi, M);
  return cis_octant(__fadd_rn(__fsub_rn(b.hi, __fsub_rn(ts, M)), e), 2u * __float_as_uint(ts));
}

// phi = u l + v m + w t with exact float products (two_prod) and float-float sums
__device__ __forceinline__ ff phase_ff(float u, float v, float w, const ff &l, const ff &m, const ff &t) {
  const ff a = ff_mul({u, 0.0f}, l), b = ff_mul({v, 0.0f}, m), c = ff_mul({w, 0.0f}, t);
  return ff_add(ff_add(a, b), c);
}
// the same for any size
static __device__ __noinline__ float2 cis_any(float u, float v, float w, ff l, ff m, ff t) {
  return cis_cycles_ff(phase_ff(u, v, w, l, m, t));
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
    auto add = [&](float2 &s, float2 e) {
      s.x = fmaf(val.x, e.x, fmaf(-val.y, e.y, s.x));
      s.y = fmaf(val.x, e.y, fmaf(val.y, e.x, s.y));
    };
    if (fmaxf(fmaxf(fabsf(uf), fabsf(vf)), fabsf(wf)) <= kCisMax) {
#pragma unroll
      for (int i = 0; i < kDftPix; ++i) add(acc[i], cis_small(uf, vf, wf, px[i].l, px[i].m, px[i].t));
    } else {
#pragma unroll
      for (int i = 0; i < kDftPix; ++i) add(acc[i], cis_any(uf, vf, wf, px[i].l, px[i].m, px[i].t));
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
