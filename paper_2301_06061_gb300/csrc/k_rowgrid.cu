// Row-wise gridding fused with the row FFT (K-G + K-F rows), and its adjoint fused with
// degridding (K-D) or with the tabulated-kernel gradient (K-KG).
//
// Forward, per (plane, row q) work item: the visibilities whose W-row footprint covers
// row q are the contiguous buckets j0 = q - W + 1 ... q (k_sort.cu).  If there are
// none the row is zero: the item writes zeros and is done (no gridding, no FFT, no read
// of a plane).  Otherwise the row is accumulated in shared memory -- each thread takes
// visibilities, weights its W taps by G(a - W/2 + g_x) G(d - W/2 + g_y), d = q - j0,
// and adds them with shared-memory atomics (section 2, Eq. 3) -- then transformed in
// place (centring sign (-1)^(p+q) folded into the first stage) and written once.  The
// paper's gridder instead adds every tap of every visibility to the mesh in global
// memory, and the FFT reads the mesh back.
//
// Adjoint, per item: the row of the adjoint plane is transformed with the negative
// exponent (sign (-1)^(p+q) after the last stage), kept in shared memory, and every
// visibility whose footprint covers the row reads its W taps from it: degridding adds
// w G_y(d) sum_a G_x(a) row[i0 + a] to dvis; the kernel gradient scatters the tap
// products into a shared partial table.  Rows nobody reads are skipped.
//
// Rows are handed out by a device counter to the thread groups of persistent CTAs
// (GroupCfg).
//
// Fixed-point accumulation.  Shared-memory integer atomics sustain about three times
// the rate of float ones on this GPU.  The sort leaves, per row bucket and bin of 64
// columns, the sum of max(|Re|, |Im|) of the weighted values whose taps reach the bin;
// for row q, M_b = the sum of bin b over the buckets j0 = q - W + 1 ... q bounds every
// cell of bin b by M_b G^2 (G the largest |kernel value|); the sort's last pass
// (k_row_bounds) leaves max_b M_b and sum_b M_b per row.  With B = max_b M_b G^2 the
// row is accumulated in int32 units of delta = B / 2^34: each tap is rounded to a
// multiple of delta (error <= delta/2).  B is a sum of magnitudes, far above the cells
// of a dense bin (random phases add up like a square root), which is what makes the
// fine quantum usable; but a cell or a single tap can exceed 2^31 delta = B/8 (a
// dominant visibility, a coherent pile-up), so every integer atomic returns the old
// value and the kernel checks for a wrapped partial sum or a saturated conversion: if
// any occurred in the row, the row is zeroed and accumulated again with float atomics.
// Rows whose busiest bin holds fewer than 64 mean contributions take delta = B / 2^30,
// which cannot overflow (sparse rows would otherwise overflow often; their cells are
// few-term sums, for which the coarser quantum is precise enough).
// Rows whose busiest bin holds more than kFixedBinCap times the row's mean magnitude
// per visibility-row (the bins count a visibility-row once per bin it reaches,
// 1 + (W - 1)/64 bins on average) go straight to float atomics.  On the benchmark
// workload the image error against the FP64 oracle equals that of all-float
// accumulation.
//
// Rows shorter than 8192.  One quantum for a whole row takes bits from every cell far below
// its busiest bin, and rounds otherwise than float sums do.  Neither may show:
//   - wst_grid hands the cells to the caller: its rows are summed in float.
//   - In an image a cell's rounding is one term of the row's transform, which rounds by about
//     2^-25 of the row's root sum of squares, R.  The integers' roundings add up to
//     0.76 sqrt(visibilities) delta over the row (seven taps).  With m the mean magnitude, R
//     is about 0.6 m sqrt(visibilities) or more, and the steps of unit_of keep the sum below
//     the transform's rounding up to 400 contributions in the busiest bin; beyond, float sums
//     round as much themselves (their partial sums grow with the count).  A row that one
//     value dominates (R near B) leaves the range with the finest quantum and is taken
//     again with B / 2^32, about half the transform's rounding at 8192 visibilities, but no
//     coarser: then float.
//   - A strong grid correction amplifies either rounding alike at the image's edge, by
//     (Ghat(0) / Ghat(1/2))^2, and with it the difference between the two: 2e-5 of an image
//     at 1e4.  Plans above that (kFixedMaxRatio, Gaussians of 9 and 10 and unpadded
//     Kaiser-Bessel tables among them) and tables, whose transform only the device knows, take
//     float sums, and so do rows below 1024, whose float sums repeat from call to call (an
//     unpadded Kaiser-Bessel table of 8 came out 50% different at 512^2).
// What it saves (float sums are compare-and-swap loops): 4096^2 x 32 planes, 4.08M
// visibilities, 1.28 instead of 1.69 ms in this kernel, 64 images of 2048^2 x 16, 37.7M, 7.7
// instead of 12.2, 9 of 1024^2 x 5, 5.9M, 0.96 instead of 3.4.
#include "fft_core.cuh"

namespace wst {

// The row kernels' threads: a row has TPR, and the rows of a CTA are worked on by groups
// of GT threads (whole warps) that claim rows and synchronise on their own: a group with
// a dense row does not hold up the others, and empty rows cost no barrier of the CTA.  The
// groups share the CTA's twiddle tables.  Rows shorter than 512 have fewer than 32 threads;
// a group then takes GR rows in step.  CTAs of 128 threads, so that short workloads (a
// 256^2 image has 16 rows per SM) still spread over the SMs.  With 256 threads on 2 to 16 rows
// in step, an item and its offsets fetched row by row, 64 images of 2048^2 x 16 took 14.3 ms,
// now 7.7 (integer sums).
template <int N, int MINT = 128>
struct GroupCfg {
  static constexpr int EPT = RowCfg<N>::EPT, TPR = RowCfg<N>::TPR, PADL = RowCfg<N>::PADL;
  static constexpr int GT = TPR >= 32 ? TPR : 32;
  static constexpr int GR = GT / TPR;
  static constexpr int THREADS = TPR >= MINT ? TPR : MINT;
  static constexpr int GROUPS = THREADS / GT;
  static constexpr int ROWS = GROUPS * GR;  // rows in a CTA's shared memory
};

// The gridder's configuration: four rows of 4096 at once in a CTA of 1024 threads, which
// share its 33 KB of twiddle tables (two CTAs with a row each fit otherwise: 1327 instead of
// 1277 us on 32 planes of 4096^2 with 4.08M visibilities, 986 instead of 882 us on 21 planes
// with the ES kernel).  Two rows of 8192 in a CTA leave 64 registers a thread: 5.90 instead of
// 5.03 ms on 16 planes with 20M visibilities.
// The configuration of float sums, which dense rows bound (shared compare-and-swap loops): CTAs
// of 256 threads on 256 / TPR rows in step.  With the groups above, which let a few dense
// rows finish last, wst_grid took 545 instead of 364 us at 2048^2 x 12 (1.33M visibilities, ES
// of 8), four images of 1024^2 x 8 (4M, support 7) 3.60 instead of 2.23 ms, 16 of 512^2 x 8 (2M)
// 1.66 instead of 1.29.  Rows shorter than 1024 need two rounds of CTAs for that: with 4096
// rows of 512 in all the groups are ahead (623 against 660 us, 200,000 visibilities), and a
// 256^2 x 8 image has too few rows for either.  Integer sums are faster in groups.
constexpr int kStepCtas = 4;  // per SM
template <int N>
struct StepCfg {
  static constexpr int EPT = RowCfg<N>::EPT, TPR = RowCfg<N>::TPR, PADL = RowCfg<N>::PADL;
  static constexpr int THREADS = RowCfg<N>::THREADS, GT = THREADS, GR = GT / TPR, GROUPS = 1, ROWS = GR;
};
template <int N, bool STEP = false>
using GridCfg = std::conditional_t<STEP, StepCfg<N>, GroupCfg<N, N == 4096 ? 1024 : 128>>;
// whether a group writes a row out during its next row's gridding: where it is alone
template <int N>
constexpr bool kPending = N >= 8192;

// rows whose kernel copies the tap-major table to shared memory (smem_taps: if it fits)
template <int N>
constexpr bool kTapsShared = N == 8192;

// barrier of one group: the CTA, a warp, or a named barrier of the group's warps
template <int GT, int GROUPS>
struct GroupSync {
  int g;
  __device__ __forceinline__ void operator()() const {
    if constexpr (GROUPS == 1) __syncthreads();
    else if constexpr (GT == 32) __syncwarp();
    else asm volatile("barrier.cta.sync %0, %1;" ::"r"(g + 1), "n"(GT) : "memory");
  }
  // barrier with the or of a predicate over the group
  __device__ __forceinline__ bool any(bool x) const {
    if constexpr (GROUPS == 1) {
      return __syncthreads_or(x);
    } else if constexpr (GT == 32) {
      const bool r = __any_sync(0xFFFFFFFFu, x);
      __syncwarp();
      return r;
    } else {
      uint32_t r;
      asm volatile(
          "{\n .reg .pred p, q;\n setp.ne.u32 q, %1, 0;\n barrier.cta.red.or.pred p, %2, %3, q;\n"
          " selp.u32 %0, 1, 0, p;\n}\n"
          : "=r"(r)
          : "r"((uint32_t)x), "r"(g + 1), "n"(GT)
          : "memory");
      return r != 0;
    }
  }
};

// Rows are handed out in batches: the first ones to each group by its index, the others by
// a device counter, claimed ahead of time.  A batch is at most kRowBatch rows (one lane of
// the group's first warp looks at each; eight keep the end of a long row stream balanced)
// and few enough that every group gets several.
constexpr int kRowBatch = 8;
// threads per SM that the short rows' registers are limited for
constexpr int kRowThreadsPerSm = 768;

template <int N>
__device__ __forceinline__ void zero_row(float2 *srow, int jt) {
  float4 *p = reinterpret_cast<float4 *>(srow);
  for (int i = jt; i < N / 2; i += RowCfg<N>::TPR) p[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
}

// The W x-taps G(a - W/2 + g_x), a = 0 .. W-1.  For the Gaussian, three exponentials
// instead of W: with t = g_x - W/2, G(t + a + 1) / G(t + a) = R q^a, R = exp(-(2t + 1) c),
// q = exp(-2c), c = 1/(2 sigma^2); each exponential is a power of two, exp(-y c) =
// 2^(-y c log2 e), with c log2 e rounded once from FP64 (the FP32 argument carries the
// same rounding as with exp).
// taps: the tap-major table, in shared memory if SMT (else in device memory), or null.
template <int WT, bool SMT>
__device__ __forceinline__ void x_taps(const KernelParams &kp, const float *taps, float gx, float q, float (&g)[WT]) {
  static_assert(WT <= kTapRow, "taps of a row");
  if (kp.kind == WST_KERNEL_GAUSS) {
    const float t = gx - kp.half;
    float ga = exp2f(-t * t * kp.l2c);
    float ra = exp2f(-(2.0f * t + 1.0f) * kp.l2c);
#pragma unroll
    for (int a = 0; a < WT; ++a) {
      g[a] = ga;
      ga *= ra;
      ra *= q;
    }
  } else if (taps) {
    // tabulated kernel: all W taps share the sub-cell position, so the samples that bracket
    // them are two neighbouring rows of the tap-major table, four 16-byte loads.  The loads
    // bound the gridder with a table (a warp's go to 32 different lines each): rows of 8192,
    // one CTA per SM, have the memory to keep the table in shared memory
    const float pos = gx * (float)kp.per_cell;
    const int i = min((int)pos, kp.per_cell - 1);
    const float f = pos - (float)i;
    const float4 *row = reinterpret_cast<const float4 *>(taps + (size_t)i * kTapRow);
    float lo[kTapRow], hi[kTapRow];
#pragma unroll
    for (int k = 0; k < kTapRow / 4; ++k) {
      const float4 x = SMT ? row[k] : __ldg(row + k), y = SMT ? row[kTapRow / 4 + k] : __ldg(row + kTapRow / 4 + k);
      lo[4 * k] = x.x, lo[4 * k + 1] = x.y, lo[4 * k + 2] = x.z, lo[4 * k + 3] = x.w;
      hi[4 * k] = y.x, hi[4 * k + 1] = y.y, hi[4 * k + 2] = y.z, hi[4 * k + 3] = y.w;
    }
#pragma unroll
    for (int a = 0; a < WT; ++a) g[a] = fmaf(f, hi[a] - lo[a], lo[a]);
  } else {
#pragma unroll
    for (int a = 0; a < WT; ++a) g[a] = kernel_tap(kp, (float)a - kp.half + gx);
  }
}

// f(a, G(a - W/2 + g_x)) for every tap a: the unrolled x_taps where the support has an
// instance of its own (and not EVAL), else each tap evaluated
template <int WT, bool EVAL, bool SMT, class F>
__device__ __forceinline__ void for_taps(const KernelParams &kp, const float *taps, float gx, float q, const F &f) {
  if constexpr (WT > 0 && !EVAL) {
    float g[WT];
    x_taps<WT, SMT>(kp, taps, gx, q, g);
#pragma unroll
    for (int a = 0; a < WT; ++a) f(a, g[a]);
  } else {
    const int W = WT > 0 ? WT : kp.support;
#pragma unroll
    for (int a = 0; a < W; ++a) f(a, kernel_tap(kp, (float)a - kp.half + gx));
  }
}

constexpr int kFixedBinCap = 8192;
template <int N, bool FFT>
constexpr bool kFixedRows = N >= kFixedMinN || (FFT && N >= kFixedImagingMinN);

// delta / B of a row shorter than 8192, n_eff the mean contributions in its busiest bin.
// Sparse bins hold sums of a few taps: up to 64 the quantum stays below 2^-26 of the mean
// magnitude, and a cell may hold, before the row is accumulated again, the whole bin below
// 16 and half of it below 64.  From 64 on it is B / 2^34, a cell up to an eighth of the bin.
__device__ __forceinline__ float unit_of(float n_eff) {
  return n_eff < 16.0f ? 0x1p-30f : n_eff < 64.0f ? 0x1p-32f : 0x1p-34f;
}

// one tap into the planar row: float atomics, or (FIXED) the tap already in units of the
// row's quantum (the record's value was scaled by 1/delta once), converted and added as
// an integer atomic; ovf turns negative if the cell's partial sum wrapped around (the
// returned old value and the new sum have signs no in-range sum can give).  Saturated
// conversions are excluded per record (grid_row), not per tap.
template <bool FIXED>
__device__ __forceinline__ void add_tap(float *sre, float *sim, int c, float re, float im, int &ovf) {
  if constexpr (FIXED) {
    const int xr = __float2int_rn(re), xi = __float2int_rn(im);
    const int o1 = atomicAdd(reinterpret_cast<int *>(sre) + c, xr);
    const int o2 = atomicAdd(reinterpret_cast<int *>(sim) + c, xi);
    const int s1 = o1 + xr, s2 = o2 + xi;
    ovf |= ((o1 ^ s1) & (xr ^ s1)) | ((o2 ^ s2) & (xi ^ s2));
  } else {
    atomicAdd(&sre[c], re);
    atomicAdd(&sim[c], im);
  }
}

// Accumulate the visibilities of rows j0 = q - d_lo ... q into the row, stored planar
// (re[0..N), im[0..N)).  Their sub-buckets are contiguous in the sorted records, so the
// range bnd[0] .. bnd[d_lo + 1] is split evenly over the row's threads, one visibility
// per thread (two in flight); bnd[i] is where row j0 = q - d_lo + i starts.  WT > 0
// fixes the support at compile time.
__device__ __forceinline__ void cp_async16_rg(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// 4- or 8-byte asynchronous copy
template <int BYTES>
__device__ __forceinline__ void cp_async_small(uint32_t dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}

// The previous row's transformed values, written out while this row is gridded: two
// groups of four of a thread's outputs while the row's offsets load, then four per
// record it grids, the rest when its gridding ends, so that a row's 128 KB leave the SM
// spread over the next row's gridding instead of in one burst at the end of its
// transform.
template <int N>
struct PendingRow {
  static constexpr int EPT = RowCfg<N>::EPT, TPR = RowCfg<N>::TPR, CH = 4, NCH = EPT / CH;
  static constexpr int NST = num_stages(N, EPT), RL = stage_radix(N, EPT, NST - 1);
  float2 v[EPT];
  float2 *orow;
  int next;  // next group of CH outputs to write; NCH: nothing pending
  // one group, chosen by a chain of branches whose stores are separate asm statements
  // (a merged store would index v at run time and move it out of registers)
  template <int C>
  __device__ __forceinline__ void write_group(int jt) {
#pragma unroll
    for (int k = 0; k < CH; ++k) {
      const int e = C * CH + k;  // output e = b RL + r of the last stage
      float2 *a = orow + out_index<N, EPT, TPR, NST - 1>(jt, e / RL, e % RL);
      asm volatile("st.global.cs.v2.f32 [%0], {%1, %2};" ::"l"(a), "f"(v[e].x), "f"(v[e].y) : "memory");
    }
  }
  template <int C = 0>
  __device__ __forceinline__ void write_chain(int jt) {
    if constexpr (C < NCH) {
      if (next == C) write_group<C>(jt);
      else write_chain<C + 1>(jt);
    }
  }
  __device__ __forceinline__ void write_one(int jt) {
    if (next >= NCH) return;
    write_chain(jt);
    ++next;
  }
  __device__ __forceinline__ void write_all(int jt) {
#pragma unroll
    for (int c = 0; c < NCH; ++c)
      if (c >= next) {
#pragma unroll
        for (int k = 0; k < CH; ++k) {
          const int e = c * CH + k;
          __stcs(&orow[out_index<N, EPT, TPR, NST - 1>(jt, e / RL, e % RL)], v[e]);
        }
      }
    next = NCH;
  }
};
struct NoPending {
  __device__ __forceinline__ void write_one(int) {}
  __device__ __forceinline__ void write_all(int) {}
};

// With FIXED, qscale = 1/delta and gmax the largest |kernel value|: a record whose scaled
// value times gmax comes within 0.2% of 2^31 (a margin for the rounding of the taps)
// could saturate a conversion, and sends the row to float atomics like a wrapped sum.
template <int N, int WT, bool FIXED, bool STEP, class PEND>
__device__ __forceinline__ int grid_row(float *sre, float *sim, const Record *__restrict__ rec,
                                        const uint32_t *bnd, int d_lo, const KernelParams &kp, int jt,
                                        float qscale, float gmax, RecHead *stg, int stg_stride, const float *taps, PEND &pd) {
  constexpr int TPR = RowCfg<N>::TPR;
  int ovf = 0;
  const uint32_t s_end = bnd[d_lo + 1];
  if constexpr (STEP && WT == 0) {
    const int W = kp.support;
    for (uint32_t s = bnd[0] + jt; s < s_end; s += TPR) {
      int i = d_lo;
      while (s < bnd[i]) --i;
      const RecHead r = rec_head(rec, s);
      const float gy = kernel_tap(kp, (float)(d_lo - i) - kp.half + rec_gy(r));
      const float gx = rec_gx(r);
      const int i0 = rec_i0(r);
      const float vre = r.vre * gy, vim = r.vim * gy;
      for (int a = 0; a < W; ++a) {
        const float g = kernel_tap(kp, (float)a - kp.half + gx);
        add_tap<false>(sre, sim, i0 + a, vre * g, vim * g, ovf);
      }
    }
    return 0;
  }
  const float q = exp2f(-2.0f * kp.l2c);
  // this thread's record heads are copied into its own three shared slots two records
  // ahead (cp.async), so two loads are in flight while a record is gridded
  const uint32_t slot0 = (uint32_t)__cvta_generic_to_shared(stg);
  const uint32_t sstep = (uint32_t)(stg_stride * sizeof(RecHead));
  uint32_t s = bnd[0] + jt;
  if (s < s_end) cp_async16_rg(slot0, rec + s);
  asm volatile("cp.async.commit_group;" ::: "memory");
  if (s + TPR < s_end) cp_async16_rg(slot0 + sstep, rec + s + TPR);
  asm volatile("cp.async.commit_group;" ::: "memory");
  int i = 0;  // the thread's records come in increasing order, so do their buckets
  int cur = 0, nxt = 2;  // slot of this record, slot of the one two ahead
  for (; s < s_end; s += TPR) {
    if (s + 2 * TPR < s_end) cp_async16_rg(slot0 + nxt * sstep, rec + s + 2 * TPR);
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 2;" ::: "memory");
    const RecHead r = stg[cur * stg_stride];
    cur = cur == 2 ? 0 : cur + 1;
    nxt = nxt == 2 ? 0 : nxt + 1;
    while (i < d_lo && bnd[i + 1] <= s) ++i;  // the last row starting at or before the record
    // the record's row offset keeps y in [-W/2, W/2): no range test
    const float y = (float)(d_lo - i) - kp.half + rec_gy(r);
    const float gy = WT > 0 && kp.kind == WST_KERNEL_GAUSS ? exp2f(-y * y * kp.l2c) : kernel_tap(kp, y);
    const int i0 = rec_i0(r);
    const float gq = FIXED ? gy * qscale : gy;
    const float vre = r.vre * gq, vim = r.vim * gq;
    if (FIXED && fmaxf(fabsf(vre), fabsf(vim)) * gmax >= 0x1.ffp30f) ovf = -1;
    for_taps<WT, false, kTapsShared<N>>(kp, taps, rec_gx(r), q, [&](int a, float g) {
      add_tap<FIXED>(sre, sim, i0 + a, vre * g, vim * g, ovf);
    });
    pd.write_one(jt);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  return ovf;
}

// One row q of a plane: accumulate, transform (FFT) and write it (with a PendingRow, during
// the next row's gridding: pd holds the row before this one on entry and this row on
// return).  bnd[0 .. d_lo + 1]: where the rows j0 = q - d_lo ... q start, and the end; mb:
// the row's largest bin sum and the total of its bin sums.  Every thread of the row group
// calls it; it ends with the row buffer free again.
template <int N, bool FFT, int WT, bool STEP, class PEND, class SYNC>
__device__ __forceinline__ void grid_one_row(float2 *srow, const uint32_t *bnd, int d_lo, float2 mb,
                                             const Record *__restrict__ rec, int q, bool nonempty,
                                             const KernelParams &kp, float2 *__restrict__ orow, const float2 *twt,
                                             int jt, float gmax, RecHead *stg, int stg_stride, const float *taps,
                                             bool ints, PEND &pd, const SYNC &sync) {
  using C = RowCfg<N>;
  constexpr int EPT = C::EPT, TPR = C::TPR;
  constexpr int NST = num_stages(N, EPT);
  constexpr int R0 = stage_radix(N, EPT, 0);
  constexpr int RL = stage_radix(N, EPT, NST - 1);
  auto smi = [](int i) { return i + i / EPT; };
  const int W = WT > 0 ? WT : kp.support;
  float *sre = reinterpret_cast<float *>(srow), *sim = sre + N;  // planar accumulation
  // two groups of the previous row's outputs go out before the row is zeroed (more, or one
  // more after the first record heads are requested, measured slower)
  pd.write_one(jt);
  pd.write_one(jt);
  zero_row<N>(srow, jt);
  sync();
  // the same decision and quantum in every thread of the row
  const uint32_t cnt = nonempty ? bnd[d_lo + 1] - bnd[0] : 0u;
  const float mmax = mb.x, mtot = mb.y;
  const float bound = mmax * (gmax * gmax);
  // n_eff: the busiest bin's magnitude in units of the row's mean per visibility-row
  const float n_eff = mmax * (float)cnt * (1.0f + (float)(W - 1) / (float)kBinCols) / fmaxf(mtot, 0x1p-126f);
  // (a NaN in a kernel table makes the bound NaN and takes float sums, which show it)
  constexpr bool INTS = kFixedRows<N, FFT> && !STEP;
  const bool fixed = INTS && ints && nonempty && cnt < (1u << 30) && bound >= 0x1p-90f && bound <= 0x1p+100f &&
                     n_eff <= (float)kFixedBinCap;
  // a bin of fewer than ~64 mean contributions may hold a single tap above B/8: such rows
  // take delta = B / 2^30, with which no tap or partial sum can leave the int32 range
  float unit = N >= kFixedMinN ? (n_eff >= 64.0f ? 0x1p-34f : 0x1p-30f) : unit_of(n_eff);
  bool fx = fixed;
  auto in_ints = [&] {
    return grid_row<N, WT, INTS, STEP>(sre, sim, rec, bnd, d_lo, kp, jt, 1.0f / (bound * unit), gmax, stg, stg_stride,
                                       taps, pd);
  };
  auto in_float = [&] {
    grid_row<N, WT, false, STEP>(sre, sim, rec, bnd, d_lo, kp, jt, 1.0f, gmax, stg, stg_stride, taps, pd);
  };
  int ovf = 0;
  if (nonempty) {
    if (fixed) ovf = in_ints();
    else in_float();
  }
  // a tap or a partial sum left the int32 range: shorter rows once more with B / 2^32, then in
  // float.  (B / 2^30 would hold any row, but rounds by twice what the row's transform does
  // where one value dominates it.)
  bool redo = false;
  if constexpr (INTS) redo = sync.any(ovf < 0);
  else sync();
  if constexpr (INTS && N < kFixedMinN) {
    if (redo && unit < 0x1p-32f) {
      zero_row<N>(srow, jt);
      sync();
      unit = 0x1p-32f;
      redo = sync.any(in_ints() < 0);
    }
  }
  if (redo) {
    zero_row<N>(srow, jt);
    sync();
    in_float();
    fx = false;
    sync();
  }
  pd.write_all(jt);  // the previous row is out before this one's transform takes its place
  const float delta = fx ? bound * unit : 1.0f;
  const int *ire = reinterpret_cast<const int *>(sre), *iim = reinterpret_cast<const int *>(sim);
  if constexpr (FFT) {
    float2 v[EPT];
    if (fx) {
#pragma unroll
      for (int b = 0; b < EPT / R0; ++b)
#pragma unroll
        for (int r = 0; r < R0; ++r) {
          const int idx = in_index<N, EPT, TPR, 0>(jt, b, r);
          const float sg = ((idx + q) & 1) ? -delta : delta;  // centring sign and quantum
          v[b * R0 + r] = make_float2(sg * __int2float_rn(ire[idx]), sg * __int2float_rn(iim[idx]));
        }
    } else {
#pragma unroll
      for (int b = 0; b < EPT / R0; ++b)
#pragma unroll
        for (int r = 0; r < R0; ++r) {
          const int idx = in_index<N, EPT, TPR, 0>(jt, b, r);
          const float sg = ((idx + q) & 1) ? -1.0f : 1.0f;  // centring sign
          v[b * R0 + r] = make_float2(sg * sre[idx], sg * sim[idx]);
        }
    }
    sync();  // natural-order reads done before the padded writes
    const TableTw<N, EPT, TPR, 1> twp{twt, jt};
    stage_compute_f<N, EPT, TPR, 0, 1>(v, jt, twp);
    middle_stages_f<N, EPT, TPR, 1, 1>(v, jt, srow, smi, twp, sync);
    stage_compute_f<N, EPT, TPR, NST - 1, 1>(v, jt, twp);
    if constexpr (std::is_same_v<PEND, PendingRow<N>>) {
      // kept for the next row's gridding (assigned on every path, so that the old values
      // are dead after their last write)
#pragma unroll
      for (int e = 0; e < EPT; ++e) pd.v[e] = v[e];
      pd.orow = orow;
      pd.next = (orow && nonempty) ? 0 : PEND::NCH;
    } else if (orow && nonempty) {
#pragma unroll
      for (int b = 0; b < EPT / RL; ++b)
#pragma unroll
        for (int r = 0; r < RL; ++r)  // streaming stores: keep the L2 for the records
          __stcs(&orow[out_index<N, EPT, TPR, NST - 1>(jt, b, r)], v[b * RL + r]);
    }
  } else {
    if (orow) {
      if (fx)
        for (int i = jt; i < N; i += TPR)
          orow[i] = make_float2(delta * __int2float_rn(ire[i]), delta * __int2float_rn(iim[i]));
      else
        for (int i = jt; i < N; i += TPR) orow[i] = make_float2(sre[i], sim[i]);
    }
  }
  sync();  // the row buffer is reused by the next row
}

template <int N, bool FFT, int WT, bool STEP = false>
__global__ void __launch_bounds__(GridCfg<N, STEP>::THREADS,
                                  STEP ? (FFT ? kStepCtas : 1) : N >= 4096 ? 1 : kRowThreadsPerSm / GridCfg<N>::THREADS)
k_grid_rows(const Record *__restrict__ rec, const uint32_t *__restrict__ off, int p0, int np,
            KernelParams kp, float2 *__restrict__ out, uint8_t *__restrict__ occ,
            unsigned long long *__restrict__ counter, Tw tw, const float2 *__restrict__ rowbound,
            unsigned long long *__restrict__ rows_done, int batch, bool smem_taps, bool ints) {
  using C = GridCfg<N, STEP>;
  constexpr int TPR = C::TPR, GT = C::GT, GR = C::GR, GROUPS = C::GROUPS;
  extern __shared__ __align__(16) float2 sm_rows[];
  const int g = threadIdx.x / GT, gt = threadIdx.x % GT;   // group, thread of the group
  const int rl = threadIdx.x / TPR, jt = threadIdx.x % TPR;  // row of the CTA, thread of the row
  const GroupSync<GT, GROUPS> sync{g};
  float2 *srow = sm_rows + rl * C::PADL;
  float2 *twt = sm_rows + C::ROWS * C::PADL;  // twiddle tables (visible after the first barrier)
  // three record-head slots per thread after the tables
  RecHead *stg = reinterpret_cast<RecHead *>(twt + (FFT ? line_table_size<N, C::EPT, TPR>() : 0)) + threadIdx.x;
  const int stg_stride = C::THREADS;
  if constexpr (FFT) fill_line_tables<N, C::EPT, TPR>(twt, tw);
  // G^2 of the fixed-point bound (G = 1 for the Gaussian and the ES kernel, the largest
  // |sample| of a table: linear interpolation stays below it)
  const float gmax = kp.kind == WST_KERNEL_TABLE ? __ldg(kp.table_max) : 1.0f;
  const float *taps = kp.tap_table;
  if constexpr (kTapsShared<N> && WT > 0) {
    if (smem_taps) {
      float4 *t = reinterpret_cast<float4 *>(stg - threadIdx.x + 3 * C::THREADS);
      for (int i = threadIdx.x; i < (kp.per_cell + 1) * (kTapRow / 4); i += C::THREADS)
        t[i] = __ldg(reinterpret_cast<const float4 *>(kp.tap_table) + i);
      taps = reinterpret_cast<const float *>(t);
    }
  }
  __syncthreads();
  const long long total = (long long)np * N;
  const int W = WT > 0 ? WT : kp.support;
  const long long group0 = (long long)blockIdx.x * GROUPS + g, ngroups = (long long)gridDim.x * GROUPS;
  if constexpr (GR == 1) {
    // batches of rows (a power of two, so that a batch lies in one plane).  The bucket
    // offsets its rows need, q0 - W + 1 ... q0 + batch, and the rows' bounds are copied
    // (cp.async) while the batch before it is worked on; the group's first warp then lists
    // the non-empty rows (and fills occ), and the group grids and transforms only those.
    __shared__ long long s_item[GROUPS];
    __shared__ int s_list[GROUPS][kRowBatch], s_cnt[GROUPS];
    __shared__ uint32_t s_off[GROUPS][2][kRowBatch + kMaxSupport + 1];
    __shared__ __align__(8) float2 s_rb[GROUPS][2][kRowBatch];
    const uint32_t off_sm = (uint32_t)__cvta_generic_to_shared(&s_off[g][0][0]);
    const uint32_t rb_sm = (uint32_t)__cvta_generic_to_shared(&s_rb[g][0][0]);
    auto fetch = [&](long long base, int buf) {  // by the first warp
      if (base < total) {
        const int64_t b0 = (int64_t)(p0 + base / N) * N;
        const int q0 = (int)(base % N);
        const int j = q0 - (W - 1) + gt;  // entry gt: where row j starts (unused below the plane)
        if (gt < W + batch && j >= 0)
          cp_async_small<4>(off_sm + (uint32_t)(buf * (kRowBatch + kMaxSupport + 1) + gt) * 4u,
                            off + (b0 + j) * kColBlocks);
        if (kFixedRows<N, FFT> && ints && gt < batch)
          cp_async_small<8>(rb_sm + (uint32_t)(buf * kRowBatch + gt) * 8u, rowbound + b0 + q0 + gt);
      }
    };
    // the transforming path of long rows writes each row during the next row's gridding
    std::conditional_t<FFT && kPending<N>, PendingRow<N>, NoPending> pd;
    if constexpr (FFT && kPending<N>) {
      pd.next = PendingRow<N>::NCH;
      pd.orow = nullptr;
    }
    long long next = group0 * batch;  // first warp: the next batch, its data under way
    long long after = (ngroups + group0) * batch;  // lane 0: the one after it
    if (gt < 32) fetch(next, 0);
    for (int buf = 0;; buf ^= 1) {
      if (gt < 32) {
        const long long base = next;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        next = __shfl_sync(0xFFFFFFFFu, after, 0);
        if (gt == 0) after = 2 * ngroups * batch + (long long)atomicAdd(counter, (unsigned long long)batch);
        fetch(next, buf ^ 1);
        const bool valid = gt < batch && base + gt < total;
        const int skip = max(0, W - 1 - ((int)(base % N) + gt));  // rows below the plane
        const bool nonempty = valid && s_off[g][buf][gt + skip] != s_off[g][buf][gt + W];
        if (valid) occ[base + gt] = nonempty ? 1 : 0;
        // plain gridding hands the planes to the caller: it also lists the empty rows,
        // which get zeros; the column pass reads only occupied rows of transformed planes
        const bool listed = FFT ? nonempty : valid;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, listed);
        if (listed) s_list[g][__popc(m & ((1u << gt) - 1u))] = gt * 2 + (nonempty ? 1 : 0);
        if (gt == 0) {
          s_cnt[g] = __popc(m);
          s_item[g] = base;
        }
        if (rows_done) {  // the occupied rows of the batch, for the caller's statistics
          const unsigned occupied = __ballot_sync(0xFFFFFFFFu, nonempty);
          if (gt == 0 && occupied) atomicAdd(rows_done, (unsigned long long)__popc(occupied));
        }
      }
      sync();
      const long long base = s_item[g];
      if (base >= total) break;
      const int cnt = s_cnt[g];
      for (int k = 0; k < cnt; ++k) {
        const int e = s_list[g][k], r = e >> 1;
        const long long item = base + r;
        const int pl = (int)(item / N), q = (int)(item % N);
        const int d_lo = min(q, W - 1);
        const float2 mb = kFixedRows<N, FFT> && ints ? s_rb[g][buf][r] : make_float2(0.0f, 0.0f);
        grid_one_row<N, FFT, WT, STEP>(srow, &s_off[g][buf][r + W - 1 - d_lo], d_lo, mb, rec, q, e & 1, kp,
                                 out + ((int64_t)pl * N + q) * N, twt, jt, gmax, stg, stg_stride, taps, ints, pd, sync);
      }
      if (cnt == 0) sync();  // s_item, s_cnt and the list are read before they are written again
    }
    pd.write_all(jt);  // the group's last row
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else {
    __shared__ uint32_t s_bnd[C::ROWS][kMaxSupport + 2];
    static_assert(!kFixedRows<N, FFT> || STEP, "float sums");
    long long next = group0 * GR;
    while (true) {
      long long base;
      if constexpr (GT == 32) {  // a group is one warp, its next rows claimed ahead of time
        base = __shfl_sync(0xFFFFFFFFu, next, 0);
        if (gt == 0) next = ngroups * GR + (long long)atomicAdd(counter, (unsigned long long)GR);
      } else {
        __shared__ long long s_item;
        if (gt == 0) s_item = (long long)atomicAdd(counter, (unsigned long long)GR);
        sync();
        base = s_item;
        sync();
      }
      if (base >= total) break;
      const long long item = base + rl % GR;
      const bool valid = item < total;
      const int pl = valid ? (int)(item / N) : 0;
      const int q = valid ? (int)(item % N) : 0;
      const int64_t b0 = (int64_t)(p0 + pl) * N;
      const int d_lo = min(q, W - 1);
      for (int i = jt; i <= d_lo + 1; i += TPR) s_bnd[rl][i] = off[(b0 + q - d_lo + i) * kColBlocks];
      sync();
      const bool empty = !valid || s_bnd[rl][0] == s_bnd[rl][d_lo + 1];
      if (valid && jt == 0) occ[item] = empty ? 0 : 1;
      if (rows_done && valid && jt == 0 && !empty) atomicAdd(rows_done, 1ull);
      if (!FFT || sync.any(!empty)) {
        float2 *orow = valid && (!FFT || !empty) ? out + ((int64_t)pl * N + q) * N : nullptr;
        NoPending none;
        grid_one_row<N, FFT, WT, STEP>(srow, s_bnd[rl], d_lo, make_float2(0.0f, 0.0f), rec, q, !empty, kp, orow, twt, jt,
                                       gmax, stg, stg_stride, taps, false, none, sync);
      }
      sync();
    }
  }
}

// -------------------------------------------------------------------------------------
// adjoint: row FFT^H of the adjoint plane + degridding / kernel gradient
// -------------------------------------------------------------------------------------
// x[t] added to at[t][offset] for every t with at[t] set (shared memory).  A shared float
// atomic is a compare-and-swap loop of its own, and a run of them a serial chain of round
// trips; with `together` the first attempts of all T go out at once and only what lost a race
// (another lane or an equal address in the same run) is added the usual way.  That pays
// where the lanes of a warp seldom share a sample: at kTogether samples per cell and more,
// less than one pair of 32 (8193 samples, a 512^2 training step: 132 -> 107 us; 92 with rows
// claimed when a group is free).
constexpr float kTogether = 512.0f;
template <int T>
__device__ __forceinline__ void add_all(float *const (&at)[T], const float (&x)[T], int offset, bool together) {
  if (!together) {
#pragma unroll
    for (int t = 0; t < T; ++t)
      if (at[t]) atomicAdd(at[t] + offset, x[t]);
    return;
  }
  uint32_t old[T], got[T];
#pragma unroll
  for (int t = 0; t < T; ++t)
    if (at[t]) old[t] = __float_as_uint(*(volatile float *)(at[t] + offset));
#pragma unroll
  for (int t = 0; t < T; ++t)
    if (at[t])
      got[t] = atomicCAS(reinterpret_cast<uint32_t *>(at[t] + offset), old[t],
                         __float_as_uint(__uint_as_float(old[t]) + x[t]));
#pragma unroll
  for (int t = 0; t < T; ++t)
    if (at[t] && got[t] != old[t]) atomicAdd(at[t] + offset, x[t]);
}

// Rows are handed out to groups by the counter, when a group is free for one.  Degridding adds
// a record's row sum to the caller's element, one 8-byte vector reduction.
//
// Order of the sums.  The W row sums of a visibility alternate in sign where the image's
// edges dominate it (a strong grid correction), and cancel: added from the first tap row to
// the last their partial sums stay as small as the sums themselves, in another order they
// do not, and the result carries their rounding.  Rows are therefore claimed one by one, in
// order and no earlier than they are worked on, and a row's records are walked from the
// last bucket (its visibilities' first tap row) to the first: bucket by bucket up to 128
// threads to a row (kByBucket), where the buckets' time keeps the rows of sparse images in
// order too, in one even split from 256 on, where buckets are long enough for that.  With
// two to eight rows to a batch, claimed ahead, and the records walked forward, an unpadded
// Kaiser-Bessel table of 8 gave visibilities of a 2048^2 image 5.7e-5 off those in order, now
// 8e-6, as two runs in order differ, and of an 8192^2 one 3.5e-5, now 1.9e-5 (in order 7e-6;
// bucket by bucket 1.5e-5).  10M visibilities on 16 planes of 8192^2 took 6.62 ms then, now
// 6.75, 2.56 of it here (bucket by bucket 7.41), 400,000 on 16 of 1024^2 191 us, now 185 (165
// evenly split).
//
// Sums kept in sorted order, where a warp's reductions fall on whole sectors, and handed back
// by a pass of their own took as long (the whole call 6.69 against 6.66 ms at 10M visibilities
// on 16 planes of 8192^2, 17.2 against 16.9 at 20M on 8 of 16384^2) and 8 bytes of workspace
// per visibility.  Bound by the latency of a row's load, transform and records in turn with
// two rows per SM; the taps stay evaluated one by one (the recurrence of the forward gridder
// saves 0.13 ms here, but see below).
template <int TPR, bool KGRAD>
constexpr bool kByBucket = !KGRAD && TPR <= 128;
template <int N, int WT, bool KGRAD>
__global__ void __launch_bounds__(GroupCfg<N, KGRAD ? 256 : 128>::THREADS,
                                  N >= 16384 || (KGRAD && N == 8192) ? 1 : KGRAD || N == 8192 ? 2 : N == 4096 ? 3
                                  : 1024 / GroupCfg<N>::THREADS)
k_rows_adjoint(const float2 *__restrict__ planes, const Record *__restrict__ rec,
               const uint32_t *__restrict__ off, int p0, int np, KernelParams kp,
               float2 *__restrict__ dvis, float *__restrict__ dtab,
               unsigned long long *__restrict__ counter, Tw tw, int batch) {
  using C = GroupCfg<N, KGRAD ? 256 : 128>;
  constexpr int EPT = C::EPT, TPR = C::TPR, GT = C::GT, GR = C::GR, GROUPS = C::GROUPS;
  constexpr int NST = num_stages(N, EPT);
  constexpr int R0 = stage_radix(N, EPT, 0);
  constexpr int RL = stage_radix(N, EPT, NST - 1);
  extern __shared__ __align__(16) float2 sm_rows[];
  // (the table gradient keeps nothing else in static shared memory: its partial table takes
  // what the rows leave, 6972 samples at 16384)
  __shared__ long long s_item[GROUPS];
  float2 *twt = sm_rows + C::ROWS * C::PADL;  // twiddle tables (visible after the first barrier)
  fill_line_tables<N, C::EPT, TPR>(twt, tw);
  float *ptab = reinterpret_cast<float *>(twt + line_table_size<N, C::EPT, C::TPR>());  // KGRAD partial table
  const int g = threadIdx.x / GT, gt = threadIdx.x % GT;
  const int rl = threadIdx.x / TPR, jt = threadIdx.x % TPR;
  const GroupSync<GT, GROUPS> sync{g};
  float2 *srow = sm_rows + rl * C::PADL;
  auto smi = [](int i) { return i + i / EPT; };
  const long long total = (long long)np * N;
  const int W = WT > 0 ? WT : kp.support;
  if (KGRAD) {
    for (int i = threadIdx.x; i < kp.table_len; i += blockDim.x) ptab[i] = 0.0f;
  }
  __syncthreads();
  auto row_empty = [&](long long item) {
    const int64_t b0 = (int64_t)(p0 + item / N) * N;
    const int q = (int)(item % N);
    return off[(b0 + max(0, q - W + 1)) * kColBlocks] == off[(b0 + q + 1) * kColBlocks];
  };
  auto do_row = [&](long long item, bool nonempty) {
    const int pl = (int)(item / N), q = (int)(item % N);
    const int64_t b0 = (int64_t)(p0 + pl) * N;
    const int d_lo = min(q, W - 1);
    const float2 *grow = planes + ((int64_t)pl * N + q) * N;
    float2 v[EPT];
#pragma unroll
    for (int b = 0; b < EPT / R0; ++b)
#pragma unroll
      for (int r = 0; r < R0; ++r)
        v[b * R0 + r] = nonempty ? __ldcs(grow + in_index<N, EPT, TPR, 0>(jt, b, r)) : make_float2(0.0f, 0.0f);
    // where the rows j0 = q - d_lo ... q start, and the end (nothing if the row is empty)
    static_assert(kColBlocks == 1, "a row's offsets are neighbours");
    const uint32_t *bnd = off + (b0 + q - d_lo);
    if constexpr (!KGRAD) {  // from shared memory: one latency for all of them, under the transform
      __shared__ uint32_t s_bnd[C::ROWS][kMaxSupport + 2];
      for (int i = jt; i <= d_lo + 1; i += TPR) s_bnd[rl][i] = nonempty ? bnd[i] : 0u;
      bnd = s_bnd[rl];
    }
    const TableTw<N, EPT, TPR, -1> twp{twt, jt};
    stage_compute_f<N, EPT, TPR, 0, -1>(v, jt, twp);
    middle_stages_f<N, EPT, TPR, 1, -1>(v, jt, srow, smi, twp, sync);
    stage_compute_f<N, EPT, TPR, NST - 1, -1>(v, jt, twp);
    sync();  // every padded read done before the natural-order writes
#pragma unroll
    for (int b = 0; b < EPT / RL; ++b)
#pragma unroll
      for (int r = 0; r < RL; ++r) {
        const int idx = out_index<N, EPT, TPR, NST - 1>(jt, b, r);
        float2 x = v[b * RL + r];
        if ((idx + q) & 1) x = make_float2(-x.x, -x.y);
        srow[idx] = x;
      }
    sync();
    // a record of bucket i (row j0 = q - d_lo + i), which bnd[i] .. bnd[i + 1] hold
    auto take = [&](int i, uint32_t s, const RecHead &rc) {
      const float targ_y = (float)(d_lo - i) - kp.half + rec_gy(rc);
      const float gy = kernel_tap(kp, targ_y);
      const float gx0 = rec_gx(rc);
      const float2 *cell = srow + rec_i0(rc);
      if constexpr (!KGRAD) {
        float are = 0.0f, aim = 0.0f;
        // the taps one by one, as the table gradient takes them: the image's corners enter with
        // the grid correction's 1e3 to 1e5 and cancel here, which magnifies any other rounding
        for_taps<WT, true, false>(kp, nullptr, gx0, 0.0f, [&](int a, float gx) {
          const float2 c = cell[a];
          are = fmaf(gx, c.x, are);
          aim = fmaf(gx, c.y, aim);
        });
        const uint2 tail = __ldg(reinterpret_cast<const uint2 *>(rec + s) + 2);  // index, weight
        const float wt = __uint_as_float(tail.y) * gy;
        float2 *at = dvis + tail.x;
        if (reinterpret_cast<uintptr_t>(dvis) & 7u) {  // a caller's array on 4 bytes
          atomicAdd(&at->x, wt * are);
          atomicAdd(&at->y, wt * aim);
        } else {
          asm volatile("red.relaxed.gpu.global.add.v2.f32 [%0], {%1, %2};" ::"l"(at), "f"(wt * are), "f"(wt * aim)
                       : "memory");
        }
      } else {
        // c_a = Re(conj(gh[q, i0 + a]) (w V)); x-profile tap a gets c_a G_y(d), the
        // y-profile tap d gets sum_a c_a G_x(a); each is split over the two table
        // samples bracketing the tap's argument
        float sum_cx = 0.0f;
        constexpr int T = WT > 0 ? WT : 4;  // taps at a time
        const bool together = kp.table_scale >= kTogether;
        auto split = [&](float targ, float x, float *&at, float &lo, float &hi) {
          const float pos = (targ + kp.half) * kp.table_scale;
          int k = (int)floorf(pos);
          k = max(0, min(k, kp.table_len - 2));
          const float f = pos - (float)k;
          at = ptab + k;
          lo = x * (1.0f - f);
          hi = x * f;
          return fmaf(f, __ldg(kp.table + k + 1) - __ldg(kp.table + k), __ldg(kp.table + k));  // G(targ)
        };
        for (int a0 = 0; a0 < W; a0 += T) {
          float *at[T];
          float lo[T], hi[T];
#pragma unroll
          for (int t = 0; t < T; ++t) {
            const int a = a0 + t;
            if (WT > 0 || a < W) {
              const float2 c = cell[a];
              const float cr = c.x * rc.vre + c.y * rc.vim;
              sum_cx = fmaf(cr, split((float)a - kp.half + gx0, cr * gy, at[t], lo[t], hi[t]), sum_cx);
            } else {
              at[t] = nullptr;
            }
          }
          add_all<T>(at, lo, 0, together);
          add_all<T>(at, hi, 1, together);
        }
        float *at[1];
        float lo[1], hi[1];
        split(targ_y, sum_cx, at[0], lo[0], hi[0]);
        add_all<1>(at, lo, 0, false);
        add_all<1>(at, hi, 1, false);
      }
    };
    // from the last bucket to the first (the visibilities' first tap rows first): bucket by
    // bucket, or all of the row's records split evenly over its threads, one head in flight
    if constexpr (kByBucket<TPR, KGRAD>) {
      for (int i = d_lo; i >= 0; --i)
        for (uint32_t s = bnd[i] + jt; s < bnd[i + 1]; s += TPR) take(i, s, rec_head(rec, s));
    } else {
      const uint32_t last = bnd[d_lo + 1] - 1u, n_rec = nonempty ? bnd[d_lo + 1] - bnd[0] : 0u;
      RecHead nxt{};
      if (jt < n_rec) nxt = rec_head(rec, last - jt);
      int i = d_lo;
      for (uint32_t k = jt; k < n_rec; k += TPR) {
        const uint32_t s = last - k;
        const RecHead rc = nxt;
        if (k + TPR < n_rec) nxt = rec_head(rec, s - TPR);
        while (bnd[i] > s) --i;  // the last row starting at or before the record
        take(i, s, rc);
      }
    }
    sync();  // the row buffer is reused by the next row
  };
  if constexpr (GR == 1) {
    while (true) {
      if (gt == 0) s_item[g] = (long long)atomicAdd(counter, (unsigned long long)batch);
      sync();
      const long long base = s_item[g];
      if (base >= total) break;
      sync();  // s_item is read before it is written again
      for (long long item = base; item < base + batch && item < total; ++item)
        if (!row_empty(item)) do_row(item, true);  // (others nobody reads)
    }
  } else {
    while (true) {
      long long base = 0;
      if (gt == 0) base = (long long)atomicAdd(counter, (unsigned long long)GR);
      base = __shfl_sync(0xFFFFFFFFu, base, 0);  // a group is one warp here
      if (base >= total) break;
      const long long item = base + rl % GR;
      const bool nonempty = item < total && !row_empty(item);
      if (__any_sync(0xFFFFFFFFu, nonempty)) do_row(item < total ? item : base, nonempty);
    }
  }
  if (KGRAD) {
    __syncthreads();
    for (int i = threadIdx.x; i < kp.table_len; i += blockDim.x)
      if (ptab[i] != 0.0f) atomicAdd(&dtab[i], ptab[i]);
  }
}

// -------------------------------------------------------------------------------------
// host side
// -------------------------------------------------------------------------------------
static Tw tw_half(const wst_plan_s *p) {
  Tw t;
  t.t = p->tw;
  t.hmask = (p->n >> 1) - 1;
  t.hbit = p->n >> 1;
  return t;
}

// the grid of a persistent row kernel: every resident CTA, no more than there are rows for;
// and the rows of a batch, so that each group gets 32 batches or more of a long stream (dense
// rows come in runs: with eight batches the gridder of 1M visibilities at 2048^2 x 16 ended on
// a few groups, 245 us, now 152; rows one by one cost 4096^2 x 32 1428 instead of 1277 us)
template <class C, class K>
static cudaError_t persistent_grid(wst_plan_s *p, K kern, size_t smem, int64_t rows, int &grid, int &batch) {
  // always raised to the request: the 48 KB default counts the kernel's static shared
  // memory too, so a dynamic request just under 48 KB can already exceed it
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0, sms = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, C::THREADS, smem);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->device);
  if (e != cudaSuccess) return e;
  const int64_t resident = (int64_t)(per_sm > 0 ? per_sm : 1) * sms, need = (rows + C::ROWS - 1) / C::ROWS;
  grid = (int)(resident < need ? resident : need);
  const int64_t b = rows / ((int64_t)grid * C::GROUPS * 32);
  // short rows have few threads for a dense row: eight at a time, 26.6M visibilities on eight
  // 2048^2 images (W = 8) took 15.5 ms, two 8.6 (64 sparser images 7.3 and 7.7)
  const int most = C::TPR <= 128 ? 2 : kRowBatch;
  for (batch = 1; 2 * batch <= b && 2 * batch <= most;) batch *= 2;
  return cudaSuccess;
}

template <int N, bool FFT, bool STEP>
static cudaError_t launch_grid_rows_as(wst_plan_s *p, int p0, int np, float2 *out) {
  using C = GridCfg<N, STEP>;
  // the imaging path has the common supports unrolled
  auto kern = k_grid_rows<N, FFT, 0, STEP>;
  const bool own = FFT && (p->cfg.support == 7 || p->cfg.support == 8);
  if constexpr (FFT) {
    if (p->cfg.support == 7) kern = k_grid_rows<N, FFT, 7, STEP>;
    else if (p->cfg.support == 8) kern = k_grid_rows<N, FFT, 8, STEP>;
  }
  size_t smem = sizeof(float2) * (C::ROWS * C::PADL + (FFT ? line_table_size<N, C::EPT, C::TPR>() : 0)) +
                (STEP && !own ? 0 : 3 * C::THREADS * sizeof(RecHead));
  bool smem_taps = false;
  if (FFT && kTapsShared<N> && p->ktap) {
    int most = 0;
    const cudaError_t e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, p->device);
    if (e != cudaSuccess) return e;
    const size_t tab = sizeof(float) * kTapRow * (kernel_params(p).per_cell + 1);
    smem_taps = smem + tab + 1024 <= (size_t)most;  // 1 KB: the kernel's static shared memory
    if (smem_taps) smem += tab;
  }
  int grid = 0, batch = 0;
  cudaError_t e = persistent_grid<C>(p, kern, smem, (int64_t)np * N, grid, batch);
  if (e != cudaSuccess) return e;
  unsigned long long *counter = p->W_.counters + CNT_WORK;  // cleared by the caller
  kern<<<grid, C::THREADS, smem, p->stream>>>(p->W_.records, p->W_.offsets, p0, np, kernel_params(p), out,
                                             p->W_.occ, counter, tw_half(p), p->W_.rowbound,
                                             FFT ? p->W_.counters + CNT_ROWS : nullptr, batch, smem_taps,
                                             p->fixed_rows);
  return cudaGetLastError();
}

template <int N, bool FFT>
static cudaError_t launch_grid_rows(wst_plan_s *p, int p0, int np, float2 *out) {
  if constexpr (N <= 2048) {  // float sums on rows in step (StepCfg) where two rounds of their CTAs fill the SMs
    int sms = 0;
    const cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->device);
    if (e != cudaSuccess) return e;
    const int64_t ctas = (int64_t)np * N / StepCfg<N>::ROWS;
    if (!(FFT && p->fixed_rows) && (N >= 1024 || ctas >= (int64_t)2 * kStepCtas * sms))
      return launch_grid_rows_as<N, FFT, true>(p, p0, np, out);
  }
  return launch_grid_rows_as<N, FFT, false>(p, p0, np, out);
}

template <int N, bool KGRAD>
static cudaError_t launch_rows_adjoint(wst_plan_s *p, int p0, int np, const float2 *planes, float2 *dvis, float *dtab) {
  using C = GroupCfg<N, KGRAD ? 256 : 128>;
  auto kern = k_rows_adjoint<N, 0, KGRAD>;
  if (p->cfg.support == 8) kern = k_rows_adjoint<N, 8, KGRAD>;
  if constexpr (!KGRAD)
    if (p->cfg.support == 7) kern = k_rows_adjoint<N, 7, KGRAD>;
  const size_t smem = sizeof(float2) * (C::ROWS * C::PADL + line_table_size<N, C::EPT, C::TPR>()) +
                      (KGRAD ? sizeof(float) * p->cfg.ktable_len : 0);
  int grid = 0, batch = 0;
  cudaError_t e = persistent_grid<C>(p, kern, smem, (int64_t)np * N, grid, batch);
  if (e != cudaSuccess) return e;
  if (!KGRAD) batch = 1;  // in order (k_rows_adjoint)
  unsigned long long *counter = p->W_.counters + CNT_WORK;  // cleared by row_occupancy
  kern<<<grid, C::THREADS, smem, p->stream>>>(planes, p->W_.records, p->W_.offsets, p0, np, kernel_params(p),
                                             dvis, dtab, counter, tw_half(p), batch);
  return cudaGetLastError();
}

#define WST_N_SWITCH(n, CALL)         \
  switch (n) {                        \
    case 64: return CALL(64);         \
    case 128: return CALL(128);       \
    case 256: return CALL(256);       \
    case 512: return CALL(512);       \
    case 1024: return CALL(1024);     \
    case 2048: return CALL(2048);     \
    case 4096: return CALL(4096);     \
    case 8192: return CALL(8192);     \
    case 16384: return CALL(16384);   \
  }                                   \
  return cudaErrorInvalidValue;

cudaError_t grid_rows(wst_plan_s *p, int p0, int p1, float2 *out, bool fft) {
  const int np = p1 - p0;
  if (np <= 0) return cudaSuccess;
  p->launches += 1;
  if (fft) {
#define CALL_F(n) launch_grid_rows<n, true>(p, p0, np, out)
    WST_N_SWITCH(p->n, CALL_F)
#undef CALL_F
  } else {
#define CALL_G(n) launch_grid_rows<n, false>(p, p0, np, out)
    WST_N_SWITCH(p->n, CALL_G)
#undef CALL_G
  }
}

cudaError_t rows_adjoint(wst_plan_s *p, int p0, int p1, const float2 *planes, float2 *dvis, float *dtab) {
  const int np = p1 - p0;
  if (np <= 0) return cudaSuccess;
  p->launches += 1;
  if (dtab) {
#define CALL_K(n) launch_rows_adjoint<n, true>(p, p0, np, planes, nullptr, dtab)
    WST_N_SWITCH(p->n, CALL_K)
#undef CALL_K
  } else {
#define CALL_D(n) launch_rows_adjoint<n, false>(p, p0, np, planes, dvis, nullptr)
    WST_N_SWITCH(p->n, CALL_D)
#undef CALL_D
  }
}

// occ of a chunk's rows, as k_grid_rows leaves it, for the adjoint column pass; the work
// counter of the row pass after it is cleared on the way
__global__ void k_row_occ(const uint32_t *__restrict__ off, int64_t b0, int64_t rows, int n, int W,
                          uint8_t *__restrict__ occ, unsigned long long *__restrict__ work) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *work = 0ull;
  if (i >= rows) return;
  const int64_t b = b0 + i;
  occ[i] = off[(b - min((int)(i % n), W - 1)) * kColBlocks] != off[(b + 1) * kColBlocks];
}

cudaError_t row_occupancy(wst_plan_s *p, int p0, int p1) {
  const int64_t rows = (int64_t)(p1 - p0) * p->n;
  if (rows <= 0) return cudaSuccess;
  k_row_occ<<<(unsigned)((rows + 255) / 256), 256, 0, p->stream>>>(p->W_.offsets, (int64_t)p0 * p->n, rows, p->n, p->W,
                                                                   p->W_.occ, p->W_.counters + CNT_WORK);
  p->launches += 1;
  return cudaGetLastError();
}

}  // namespace wst
