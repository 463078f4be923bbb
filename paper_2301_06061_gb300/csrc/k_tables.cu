// Plan tables built on the device at plan creation: FFT twiddles, the grid
// correction 1/Ghat(nu) and the l^2 terms of the phase screen (section 2, Eq. 2-3).
#include <math.h>

#include "wst_internal.cuh"

namespace wst {

KernelParams kernel_params(const wst_plan_s *p) {
  KernelParams k;
  k.kind = p->cfg.kernel;
  k.support = p->W;
  k.half = 0.5f * (float)p->W;
  double s = p->cfg.kparam;
  k.inv2s2 = (k.kind == WST_KERNEL_GAUSS) ? (float)(1.0 / (2.0 * s * s)) : 0.0f;
  k.l2c = (k.kind == WST_KERNEL_GAUSS) ? (float)(1.4426950408889634 / (2.0 * s * s)) : 0.0f;
  k.beta = (k.kind == WST_KERNEL_ES) ? (float)s : 0.0f;
  k.two_over_w = 2.0f / (float)p->W;
  k.table = p->ktable;
  k.table_len = p->cfg.ktable_len;
  k.table_scale = (k.kind == WST_KERNEL_TABLE) ? (float)((double)(p->cfg.ktable_len - 1) / p->W) : 0.0f;
  k.tap_table = p->ktap;
  k.table_max = p->kmax;
  k.per_cell = p->ktap ? (p->cfg.ktable_len - 1) / p->W : 0;
  return k;
}

// Tap-major copy of a kernel table with L - 1 = W pc samples: row i, 0 <= i <= pc, holds
// every tap's sample at sub-cell position i / pc, so the samples that bracket the W taps of
// one visibility (all at the same sub-cell offset) are two neighbouring rows.
__global__ void k_tap_table(const float *t, float *tap, int W, int pc) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= kTapRow * (pc + 1)) return;
  const int i = idx / kTapRow, a = idx % kTapRow;
  tap[idx] = a < W ? t[a * pc + i] : 0.0f;
}

cudaError_t build_tap_table(wst_plan_s *p) {
  if (!p->ktap) return cudaSuccess;
  const int pc = (p->cfg.ktable_len - 1) / p->W;
  k_tap_table<<<(kTapRow * (pc + 1) + 255) / 256, 256, 0, p->stream>>>(p->ktable, p->ktap, p->W, pc);
  p->launches += 1;
  return cudaGetLastError();
}

// half-wave table exp(+2 pi i m / N), m < N/2, rounded once from FP64
__global__ void k_twiddles(float2 *tw, int n) {
  int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= n / 2) return;
  double s, c;
  sincospi(2.0 * (double)m / (double)n, &s, &c);
  tw[m] = make_float2((float)c, (float)s);
}

// l_a^2 with l_a = (a - N/2) * fov/N, as float-float and FP64
__global__ void k_l2(float2 *l2ff, double *l2d, int n, double dl) {
  int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= n) return;
  double l = (double)(a - n / 2) * dl;
  double l2 = l * l;
  l2ff[a] = ff_split(l2);
  l2d[a] = l2;
}

// 1/Ghat(nu_a), nu_a = (a - n/2)/n, Ghat(nu) = int_{-W/2}^{W/2} G(x) cos(2 pi nu x) dx by
// composite Simpson in FP64: 256 panels per cell for analytic kernels; for a table, one
// panel per table interval so that the piecewise-linear kinks fall on panel ends.  As a sum
// over the 2 P + 1 nodes x_i = (i - P) h/2 it is a cosine sum with weights that do not
// depend on nu, and the cosine is even: k_kernel_nodes leaves, once, the P + 1 folded
// weights c_j = w_{P+j} G(j h/2) + w_{P-j} G(-j h/2) (FP64, h/6 and the Simpson factors in
// them), and k_correction sums c_j cos(2 pi nu j h/2) for each nu >= 0; -nu has the same.
//
// Bound: the FP64 pipe (2 FMA per clock and SM).  Thread t takes the nodes j = t + 128 m.  With
// d the half turns per node, cos(d j) = cos(d t) cos(128 d m) - sin(d t) sin(128 d m): the
// block's 128 d m are evaluated once, into shared memory, and a thread sums two products per
// node, every cosine as exact as if evaluated by itself.  (The absolute error matters: Ghat
// falls to 1e-6 of Ghat(0) and less at the field's edge.  A recurrence from node to node
// costs as many multiply-adds; its error grows with the square of the steps, 512 for the longest
// table: at 4e-11 of Ghat(0) 2e-6 of the value, now 8e-8.)  8193 samples at n = 512 take 17 us; by
// rotations, 4 multiply-adds per node, 29; with a block per nu, the kernel evaluated and
// three cospi taken in every panel, 1106, on every wst_plan_set_kernel_table, that is on every
// training step.
constexpr int kNodePanels = 256;   // panels per cell, analytic kernels
constexpr int kCorrThreads = 128;
constexpr int kMaxTurns = 512;     // kCorrThreads kMaxTurns > P: tables of 65536 samples, W = 16
static_assert(kCorrThreads * kMaxTurns >= 65536 && kMaxSupport * kNodePanels < 65536, "every node has a turn");

static int node_panels(const wst_plan_s *p) {
  return p->cfg.kernel == WST_KERNEL_TABLE ? p->cfg.ktable_len - 1 : kNodePanels * p->W;
}
int64_t kernel_node_count(const wst_plan_s *p) { return (int64_t)node_panels(p) + 1; }

// G(x_i) at node i of 0 .. 2 P (a table's nodes are its samples and their midpoints)
__device__ __forceinline__ double node_value(int kind, int i, int P, double half_h, double param, const float *tab,
                                             int W) {
  if (kind == WST_KERNEL_TABLE) {
    const int k = i >> 1;
    return (i & 1) ? 0.5 * ((double)tab[k] + (double)tab[k + 1]) : (double)tab[k];
  }
  const double x = (double)(i - P) * half_h;
  if (kind == WST_KERNEL_GAUSS) return exp(-(x * x) / (2.0 * param * param));
  const double z = 2.0 * x / W;
  return exp(param * (sqrt(fmax(0.0, 1.0 - z * z)) - 1.0));
}

// Ghat(0) / Ghat(nu), nu = n_img / (2 n): how much the grid correction raises the edge of the
// image's rows over their centre (host, for the analytic kernels: Simpson, 64 panels a cell)
double kernel_edge_ratio(const wst_plan_s *p) {
  const int W = p->W, P = 64 * W;
  const double h = (double)W / P, nu = 0.5 * p->n_img / p->n;
  double g0 = 0.0, g1 = 0.0;
  for (int i = 0; i <= 2 * P; ++i) {
    const double x = 0.5 * h * (i - P), z = 2.0 * x / W;
    const double g = p->cfg.kernel == WST_KERNEL_GAUSS ? exp(-(x * x) / (2.0 * p->cfg.kparam * p->cfg.kparam))
                                                       : exp(p->cfg.kparam * (sqrt(fmax(0.0, 1.0 - z * z)) - 1.0));
    const double w = (i & 1) ? 4.0 : (i == 0 || i == 2 * P) ? 1.0 : 2.0;
    g0 += w * g;
    g1 += w * g * cos(2.0 * M_PI * nu * x);
  }
  return fabs(g0 / g1);
}

__global__ void k_kernel_nodes(double *nodes, int P, int kind, int W, double param, const float *tab) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j > P) return;
  const double half_h = 0.5 * (double)W / (double)P;
  auto weight = [&](int i) { return (half_h / 3.0) * ((i & 1) ? 4.0 : (i == 0 || i == 2 * P) ? 1.0 : 2.0); };
  double c = weight(P + j) * node_value(kind, P + j, P, half_h, param, tab, W);
  if (j > 0) c += weight(P - j) * node_value(kind, P - j, P, half_h, param, tab, W);
  nodes[j] = c;
}

__global__ void __launch_bounds__(kCorrThreads) k_correction(float *corr, int n, const double *__restrict__ nodes,
                                                             int P, int W, const float *__restrict__ tab,
                                                             float *__restrict__ tab_max) {
  const int k = blockIdx.x;  // nu = k / n, 0 <= k <= n/2
  if (k > n / 2) {  // a table's last block: its largest |sample|, for the gridder's bound
    // (as integers, in which a NaN is the largest: the rows then take float sums and show it)
    __shared__ uint32_t s_max;
    if (threadIdx.x == 0) s_max = 0u;
    __syncthreads();
    uint32_t m = 0u;
    for (int i = threadIdx.x; i <= P; i += kCorrThreads) m = max(m, __float_as_uint(fabsf(__ldg(tab + i))));
    atomicMax(&s_max, m);
    __syncthreads();
    if (threadIdx.x == 0) *tab_max = __uint_as_float(s_max);
    return;
  }
  // 2 nu j h/2 in half turns: the numerator is below 2^53, so rounded once
  auto turn = [&](int j) { return (double)((long long)k * W * j) / ((double)n * (double)P); };
  __shared__ double2 s_turn[kMaxTurns];  // cos, sin of 128 d m
  for (int m = threadIdx.x; m <= P / kCorrThreads; m += kCorrThreads) {
    double s, c;
    sincospi(turn(m * kCorrThreads), &s, &c);
    s_turn[m] = make_double2(c, s);
  }
  __syncthreads();
  double ac = 0.0, as = 0.0;
  for (int j = threadIdx.x, m = 0; j <= P; j += kCorrThreads, ++m) {
    const double x = __ldg(nodes + j);
    const double2 t = s_turn[m];
    ac = fma(x, t.x, ac);
    as = fma(x, t.y, as);
  }
  double s, c;
  sincospi(turn(threadIdx.x), &s, &c);
  __shared__ double red[kCorrThreads];
  red[threadIdx.x] = ac * c - as * s;
  __syncthreads();
  for (int st = kCorrThreads / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const float r = (float)(1.0 / red[0]);
    corr[n / 2 - k] = r;
    if (k < n / 2) corr[n / 2 + k] = r;
  }
}

cudaError_t build_tables(wst_plan_s *p) {
  const int n = p->n;
  k_twiddles<<<(n + 255) / 256, 256, 0, p->stream>>>(p->tw, n);
  k_l2<<<(n + 255) / 256, 256, 0, p->stream>>>(p->l2ff, p->l2d, n, p->cfg.fov / (double)n);
  p->launches += 2;
  return cudaGetLastError();
}

cudaError_t build_correction(wst_plan_s *p) {
  const int P = node_panels(p);
  k_kernel_nodes<<<(P + 256) / 256, 256, 0, p->stream>>>(p->knodes, P, p->cfg.kernel, p->W, p->cfg.kparam, p->ktable);
  k_correction<<<p->n / 2 + 1 + (p->ktable ? 1 : 0), kCorrThreads, 0, p->stream>>>(p->corr, p->n, p->knodes, P, p->W,
                                                                                   p->ktable, p->kmax);
  p->launches += 2;
  return cudaGetLastError();
}

// Plane range per image: either the configured one, or the min/max of the finite w
// found by the sort's reduction (stored as order-preserving integers).
__device__ __forceinline__ float ordered_to_float(uint32_t o) {
  uint32_t b = (o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o;
  return __uint_as_float(b);
}

__global__ void k_plane_centres(double *wrange, float4 *wrange_ff, float2 *wcentre, double *wcentre_d, float2 *dwff,
                                const uint32_t *wminmax, int batch, int n_w, double cfg_lo,
                                double cfg_hi, int from_data) {
  const int P = blockIdx.x * blockDim.x + threadIdx.x;  // one thread per global plane
  if (P >= batch * n_w) return;
  const int img = P / n_w, k = P - img * n_w;
  double lo = cfg_lo, hi = cfg_hi;
  if (from_data) {
    uint32_t omin = wminmax[2 * img], omax = wminmax[2 * img + 1];
    if (omin == 0xFFFFFFFFu) {  // no finite w in this image
      lo = hi = 0.0;
    } else {
      lo = (double)ordered_to_float(omin);
      hi = (double)ordered_to_float(omax);
    }
  }
  double scale = (hi > lo) ? (double)n_w / (hi - lo) : 0.0;
  double dw = (hi - lo) / (double)n_w;
  const double wk = lo + ((double)k + 0.5) * dw;
  wcentre[P] = ff_split(wk);
  wcentre_d[P] = wk;
  if (k != 0) return;
  wrange[4 * img + 0] = lo;
  wrange[4 * img + 1] = scale;
  wrange[4 * img + 2] = dw;
  wrange[4 * img + 3] = hi;
  dwff[img] = ff_split(dw);
  const float2 lo_ff = ff_split(lo), sc_ff = ff_split(scale);
  wrange_ff[img] = make_float4(lo_ff.x, lo_ff.y, sc_ff.x, sc_ff.y);
}

cudaError_t build_plane_centres(wst_plan_s *p) {
  const bool from_data = p->cfg.w_min == p->cfg.w_max;
  k_plane_centres<<<(p->n_planes + 63) / 64, 64, 0, p->stream>>>(
      p->wrange, p->wrange_ff, p->wcentre, p->wcentre_d, p->dwff, p->W_.wminmax, p->batch, p->n_w, p->cfg.w_min,
      p->cfg.w_max, from_data ? 1 : 0);
  p->launches += 1;
  return cudaGetLastError();
}

}  // namespace wst
