// Fused persistent kernel: per cluster, FP32 and FP64 rows -> counter-RNG
// minimal sets -> FP32 solve with error bound (refined when ill-conditioned:
// 3D with residuals in pairs of FP32, 2D in FP64) -> FP32 scoring pass
// (upper-bound counts; in stages that drop trials the lead's residuals rule
// out) -> exact counts, best bound first, of the trials that can still win
// (FP64 only inside the error band) -> lowest-index argmax -> FP64 inlier mask
// and normal-equation refine -> heading.  Sec. III-A (Alg. 1, Eq. 4) and Sec. III-B (Eq. LSQ_eq,
// Eq. eq:LSQPerCluster, Alg. 2) of arXiv 2012.12618.
//
// Parallel mapping (GB300-first, not the paper's thread-per-trial): clusters
// are work items taken by persistent CTAs from an LPT-ordered list; inside a
// cluster, trials map to warps/lanes and points to lanes, with the cluster's
// FP32 rows staged in shared memory (what exceeds it in global scratch) and its
// FP64 rows in L1/L2-resident global scratch.
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

#include "rvh_device.cuh"
#include "rvh_kernels.h"
#include "rvh_scoring.cuh"

namespace rvh {

__device__ __forceinline__ unsigned long long best_key(int count, int h) {
  return ((unsigned long long)(uint32_t)(count + 1) << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)h);
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block reductions.  Each warp reduces with one redux instruction per 32-bit
// word, its lane 0 leaves the result in red, and after one barrier every
// thread combines the kWarps results.  There is no barrier in front: red has
// to be an array that no thread can still be reading from an earlier use,
// i.e. at least one other barrier lies between two uses of it.
__device__ __forceinline__ unsigned long long block_best(int count, int h, unsigned long long* red) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = __reduce_max_sync(0xffffffffu, count);
  const int hm = __reduce_min_sync(0xffffffffu, count == c ? h : 0x7fffffff);
  if (lane == 0) red[warp] = c >= 0 ? best_key(c, hm) : 0ull;
  __syncthreads();
  unsigned long long r = red[0];
#pragma unroll
  for (int w = 1; w < kWarps; ++w) r = max(r, red[w]);
  return r;
}

// sums of a and b (each below 2^31 over the block), a in the low word
__device__ __forceinline__ unsigned long long block_sum2(unsigned a, unsigned b, unsigned long long* red) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  a = __reduce_add_sync(0xffffffffu, a);
  b = __reduce_add_sync(0xffffffffu, b);
  if (lane == 0) red[warp] = (unsigned long long)b << 32 | a;
  __syncthreads();
  unsigned long long r = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) r += red[w];
  return r;
}

// maximum of non-negative floats (their bit patterns order like integers)
__device__ __forceinline__ float block_max_float(float v, int* red) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m = __reduce_max_sync(0xffffffffu, __float_as_int(v));
  if (lane == 0) red[warp] = m;
  __syncthreads();
  int r = red[0];
#pragma unroll
  for (int w = 1; w < kWarps; ++w) r = max(r, red[w]);
  return __int_as_float(r);
}

// ---- a4: upper-bound counts U_h = #{|r32| <= thi_h} of every trial (the hot loop) --
// Lane l handles trial sub-group l / pw and point quads l % pw, l % pw + pw,
// ...: pw = 32 is warp-per-trial-group with lanes over points, pw = 1 lanes
// over trials with broadcast rows.  Four trials per lane whatever
// hyps_per_lane asks: eight packed trials (pairs of registers per
// coordinate) do not fit in the 64 registers a thread has at four CTAs per SM.
template <int DIM, typename RV>
__device__ void phase_a_dispatch(int pw, const RV rows, int N, const Smem& S, int nh) {
  if (pw == 1) {
    phase_a_tiles<DIM, 1, 4>(rows, N, S, nh);
  } else if (pw == 8) {
    phase_a_tiles<DIM, 8, 4>(rows, N, S, nh);
  } else {
    phase_a_tiles<DIM, 32, 4>(rows, N, S, nh);
  }
}

// FP64 rows (a0, a1, a2, w) of a cluster's points.  The 3D model keeps them
// in global scratch, written once when the cluster is loaded, with the low
// parts of the FP32 row (pack_low) in place of w: every 3D trial refines its
// solve with those, the winner's inliers and band points need the rest.  The
// 2D model computes its rows when asked (only the winner's inliers, band
// points and rare refinements need them).
template <int DIM>
struct Rows64 {
  const FrameDesc* a;
  int64_t o;
  double4_32a* pre;
  __device__ __forceinline__ double4_32a at(int j) const { return with_w(j, a->dop[o + j]); }
  // The same row when the point's FP32 cosine-model row, which carries the
  // Doppler, is at hand.
  __device__ __forceinline__ double4_32a at(int j, float4 row) const { return with_w(j, DIM == 3 ? row.w : row.z); }
  __device__ __forceinline__ double4_32a with_w(int j, float w) const {
    if (DIM == 3) {
      double4_32a s = pre[j];
      s.w = (double)w;
      return s;
    }
    double t[3];
    row_f64<2>(a->trig, a->az[o + j], 0.0f, t);
    return make_double4_32a(t[0], t[1], 0.0, (double)w);
  }
};

// FP64 rows computed from the frame's inputs in both models: the source of
// the finishing pass, which runs after the CTA's row slot has moved on to
// later clusters.
template <int DIM>
struct Rows64Inputs {
  const FrameDesc* a;
  int64_t o;
  __device__ __forceinline__ double4_32a at(int j) const {
    double t[3];
    row_f64<DIM>(a->trig, a->az[o + j], DIM == 3 ? a->el[o + j] : 0.0f, t);
    return make_double4_32a(t[0], t[1], t[2], (double)a->dop[o + j]);
  }
};

// FP64 velocity of trial h in the oracle's exact rounding sequence.  Returns
// false if rejected.
template <int DIM, typename RS>
__device__ bool hyp_f64(const FrameDesc& a, const RS& R, int ci, int h, int N, double v[3]) {
  int q[3];
  draw_minimal_set<DIM>(a.key, a.cluster_base + ci, h, N, q);
  const double4_32a s0 = R.at(q[0]), s1 = R.at(q[1]), s2 = R.at(DIM == 3 ? q[2] : q[0]);
  const double r0[3] = {s0.x, s0.y, s0.z}, r1[3] = {s1.x, s1.y, s1.z}, r2[3] = {s2.x, s2.y, s2.z};
  const double w[3] = {s0.w, s1.w, DIM == 3 ? s2.w : 0.0};
  return solve_f64<DIM>(r0, r1, r2, w, a.eps, v, nullptr);
}

// ---- what the lead's residuals say about every other trial --------------------------
// The lead L (a trial with a high exact count) has a residual
// r_L(j) = w_j - a_j.v_L at every point, and trial h's is r_L(j) - a_j.d with
// d = v_h - v_L.  So h can only hold
//   - points with |r_L| <= tau + max|a.d|, of those the lead does not hold, and
//   - points with |a.d| <= tau + |r_L| <= 2 tau, of those it does: with
//     t = a1 / a0 (the tangent of the azimuth) that is an interval of t,
//     |d0 + d1 t + a2 d2 / a0| <= 2 tau / a0.  In 3D a2 d2 varies with the
//     elevation, and d2 is large (elevations span little, so trials differ
//     most in their vertical velocity): the lower and the upper half of a2's
//     range have an interval each.
// Histograms over the points still to be scored -- the excess |r_L| -
// thi of the points outside the lead, a quarter octave per bin, and t of the
// points inside, evenly over the cluster's range, per half of a2 -- turn both into counts
// per trial, which replace "every point still to come" in the pruning test.
// Everything is rounded so that the counts only err upwards: bins are taken
// by the same monotone FP32 expressions on both sides, and the band
// half-widths of both trials (which bound the FP32 residuals' and
// velocities' errors) are added to the thresholds.
constexpr int kExcessBins = 64, kTanBins = 32;
template <int DIM>
constexpr int kHalves = DIM == 3 ? 2 : 1;
constexpr int kExcessBase = 119 << 2;  // bin 0: an excess below 2^-8 m/s

__device__ __forceinline__ int excess_bin(float x) {
  return min(max((__float_as_int(x) >> 21) - kExcessBase, 0), kExcessBins - 1);
}

// The cluster's directions a: range of t = a1 / a0, 1 / min a0, max|a2|, and
// the least a2 and a quarter of its range (a half's centre and half-width);
// tan_ok = 0 (some a0 not safely positive) leaves the interval test out.
// The line model's rows (x, 1, y) have residuals of the same form with a =
// (1, x): t = x in [0, 1], a0 = 1, and the components of d change places.
struct DirRange {
  float t0, tinv, tabs, a0inv, zmax, z0, zq;
  int tan_ok;
};

__device__ __forceinline__ int tan_bin(const DirRange& g, float t) {
  return min(max(__float2int_rd((t - g.t0) * g.tinv), 0), kTanBins - 1);
}

template <typename Row>
__device__ __forceinline__ float row_tan(const Row& p, bool line) {
  return line ? p.x : p.y * rcp_approx(p.x);
}

// floats as integers of the same order, and back
__device__ __forceinline__ int float_order(float f) {
  const int i = __float_as_int(f);
  return i ^ (i >> 31 & 0x7fffffff);
}
__device__ __forceinline__ float order_float(int i) { return __int_as_float(i ^ (i >> 31 & 0x7fffffff)); }

__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Upper bound of a normal record's band half-width.
__device__ __forceinline__ float record_band(float4 hy, float tau_hi, bool line) {
  return line ? 0.50001f * (hy.w - hy.z) : fmaxf(hy.w - tau_hi, 0.0f) + 0x1p-20f * hy.w;
}

// The certain-inlier threshold of a record: |r32| <= tlo is an inlier.  The
// upper threshold thi is tau + b rounded up, so thi - tau bounds the band
// half-width b; a line's record, which has no third component, carries tlo there.
__device__ __forceinline__ float record_tlo(float4 hy, TauPair tau, bool line) {
  return line ? hy.z : __fsub_rd(tau.lo, __fsub_ru(hy.w, tau.hi));
}

// Where a trial's points can lie, as bins: excess bins 0 .. out of the points
// outside the lead, t bins lo .. hi - 1 of those inside, per half of a2.
// Packed in one word, six bits each.
struct HoldRange {
  uint32_t v;
  __device__ __forceinline__ int out() const { return (int)(v & 63u); }
  __device__ __forceinline__ int lo(int c) const { return (int)(v >> (6 + 12 * c) & 63u); }
  __device__ __forceinline__ int hi(int c) const { return (int)(v >> (12 + 12 * c) & 63u); }
};

template <int DIM>
__device__ __forceinline__ HoldRange hold_range(const DirRange& g, float4 lead, float lead_band, bool line, float4 hy) {
  // thi_h covers tau and the velocity error of h; 2 lead_band covers the
  // lead's velocity and residuals
  const float d0 = hy.x - lead.x, d1 = hy.y - lead.y, dz = DIM == 3 ? hy.z - lead.z : 0.0f;
  const float dx = line ? d1 : d0, dy = line ? d0 : d1;
  const float ax = fabsf(dx), ay = fabsf(dy), az = DIM == 3 ? g.zmax * fabsf(dz) : 0.0f;
  const float slack = 2.0f * lead_band + 4e-6f * (ax + ay + fabsf(dz));
  // max|a.d|: unit directions, or the ends of x's range for the line model
  const float reach = line ? fmaxf(ax, fabsf(dx + dy)) : sqrt_approx(fmaf(dx, dx, dy * dy)) + az;
  HoldRange h;
  h.v = (uint32_t)excess_bin((hy.w + reach + slack) * 1.0001f - lead.w);
  const float r = rcp_approx(dy);  // dy = 0: ends at +-inf, all of t or none of it
#pragma unroll
  for (int c = 0; c < kHalves<DIM>; ++c) {
    uint32_t lo = 0u, hi = kTanBins;
    if (g.tan_ok) {
      float u, v;
      if (DIM == 2) {
        const float K = (hy.w + lead.w + slack) * g.a0inv * 1.0001f + 1e-5f * (ax + ay * g.tabs);
        u = (-dx - K) * r;
        v = (K - dx) * r;
      } else {
        // a0 (d0 + d1 t) within K0 of -a2 dz, a0 in [min a0, 1]
        const float mid = (g.z0 + (float)(2 * c + 1) * g.zq) * dz;
        const float K0 = (hy.w + lead.w + slack + g.zq * fabsf(dz)) * 1.0001f;
        const float s = 1e-5f * (ax + ay * g.tabs + az + K0);
        const float A = -K0 - mid - s, B = K0 - mid + s;
        u = ((A < 0.0f ? A * g.a0inv * 1.0001f : A) - s - dx) * r;
        v = ((B > 0.0f ? B * g.a0inv * 1.0001f : B) + s - dx) * r;
      }
      lo = (uint32_t)min(max(__float2int_rd((fminf(u, v) - g.t0) * g.tinv), 0), kTanBins);
      hi = (uint32_t)max(min(__float2int_rd((fmaxf(u, v) - g.t0) * g.tinv), kTanBins - 1) + 1, (int)lo);
    }
    h.v |= lo << (6 + 12 * c) | hi << (12 + 12 * c);
  }
  return h;
}

// The red_ arrays carry values between warps.  Between the reads of one use
// and the writes of the next lies a barrier, each time:
//   red_i  medians (write, barrier, read, barrier); the staged pass's tops
//          (then the lead pass's barriers); prune_list (a barrier at its end);
//          the mask pass's inlier counts (a barrier at its end)
//   red_c  the staged pass's counts of the lead, while warps may still read the
//          tops in red_i (a barrier after them); the mask pass's changed
//          entries (a barrier at its end)
//   red_u  block_best: count_trial's barriers before the next, or the one after the loop
//   red_v  block_sum2: a barrier between its two uses in a count, and at count_trial's end
//   red_f  block_max_float, once per cluster
//   red_d  the line model's ranges (write, barrier, read, barrier), then the direction
//          range, read by thread 0 before the trials' barrier
//   red_t  the mask pass's sums, read after its last barrier and written after
//          the first one of the next pass
struct ClusterShared {
  unsigned long long best;
  float4 win;      // winner's FP32 record
  int red_i[kWarps];
  int red_f[kWarps];
  double red_t[9];            // the normal-equation sums of the winner's inliers
  unsigned long long ctr[2];  // exact counts, band points
  unsigned long long wctr[3][kWarps];  // per warp: fp64 trials, refined trials, (trial, point) pairs scored
  unsigned long long clk[6];  // cycles per stage (thread 0's view of the CTA)
  unsigned long long red_u[kWarps];  // block_best
  unsigned long long red_v[kWarps];  // block_sum2
  double cv64[3];             // FP64 velocity of the trial being counted (when it has band points)
  double win_v64[3];          // FP64 velocity of the current winner (valid if win_has_v64)
  int win_has_v64;
  int red_c[kWarps];
  double lo_v[3];             // least-squares velocity of the current inlier set
  float4 lo_hy;               // its FP32 record (-X, -Y, -Z, thi) and lower threshold
  float lo_tlo;
  int lo_ok;
  int stop;                   // adaptive trial count: enough trials have run
  double ln_T;                // line model (Alg. 1): the cluster's MAD threshold
  int sel_digit, sel_k;       // medians: digit or bin and rank inside it,
  int sel_hi, sel_n;          // the upper middle's bin, listed keys
  unsigned long long sel_key[2];  // and the middle keys
  double ln_min[2], ln_scale[2];  // line model: normalisation of azimuth and Doppler
  unsigned long long runs[2];  // trials run, pairs scored
  int nref;                   // 2D trials queued for refinement in the current chunk
  DirRange dir;               // the cluster's directions (staged pass)
  int red_d[5][kWarps];
  // Points still to be scored when the lead was taken, by its residual:
  // inside it, those below each bin of t per half of a2; outside it, those up
  // to each bin of the excess.  From stage 0 / 1 on and, in the second half of
  // the array, from 2 / 3 on, as 16-bit halves.
  unsigned lead_in[2 * 2 * (kTanBins + 1)];
  unsigned lead_out[2 * kExcessBins];
  unsigned lead_cnt;          // the lead's certain points and band points
};

// Adaptive trial count: with `best` the best (count + 1, -index) key so far,
// n points, k = DIM and m trials run, true once (1 - eps^k)^m <= 1 - p for
// eps = count / n: the standard RANSAC bound on the chance that every trial
// so far drew an outlier.  The power is taken by binary exponentiation in
// the same order as the oracle's, one IEEE rounding per operation, so both
// decide alike.  One thread; kept out of line.
__device__ __noinline__ int adaptive_stop(unsigned long long best, int n, int k, int m, double p) {
  const int count = (int)(best >> 32) - 1;
  if (count < 0) return 0;
  const double eps = (double)count / (double)n;
  const double ek = k == 2 ? eps * eps : (eps * eps) * eps;
  double r = 1.0, b = 1.0 - ek;
  for (int e = m; e > 0; e >>= 1) {
    if (e & 1) r = r * b;
    b = b * b;
  }
  return r <= 1.0 - p ? 1 : 0;
}

// FP32 record of an FP64 velocity v for the re-threshold of a local
// optimisation round: X = fl32(v), e >= |X - v|, the band of band_f32 around
// tau outside which FP32 residuals decide like FP64 ones.
template <int DIM>
__device__ __forceinline__ void velocity_record(const double v[3], float wmax, TauPair tau, float4* hy, float* tlo) {
  float X[3], e[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    X[k] = __double2float_rn(v[k]);
    e[k] = __double2float_ru(fabs((double)X[k] - v[k]));
  }
  float b = band_f32<DIM>(wmax, X, e);
  if (!(b < 1e30f) || !(fabsf(X[0]) < 1e30f) || !(fabsf(X[1]) < 1e30f) || !(fabsf(X[2]) < 1e30f)) {
    *hy = make_float4(-X[0], -X[1], -X[2], __int_as_float(0x7f800000));  // every point decided in FP64
    *tlo = -1.0f;
    return;
  }
  b = fmaxf(b, kBandFloor);
  *hy = make_float4(-X[0], -X[1], -X[2], __fadd_ru(tau.hi, b));
  *tlo = __fsub_rd(tau.lo, b);
}

// ---- Alg. 1 as printed (line model, 2D): normalised (azimuth, Doppler) points,
// line fits through two seed points, perpendicular-distance test against the
// cluster's median absolute deviation.  The FP64 values of each point are
// kept in its FP64 row slot (x, y, -, -), which the 2D cosine
// model does not use.

// Alg. 1 point-to-line test in FP64, evaluated as printed: aa = -m, bb = 1,
// cc = -c, distn = aa x + bb y + cc, distd = sqrt(aa^2 + bb^2) (passed in),
// dist = |distn / distd| <= thresh.
__device__ __forceinline__ bool line_in64(double m, double c, double distd, double x, double y, double thresh) {
  const double distn = (-m) * x + y + (-c);
  return fabs(distn / distd) <= thresh;
}

// FP64 line (m, c, distd) through two normalised points; false when they
// share x (no slope).
__device__ __forceinline__ bool line_seeds64(const double4_32a& p0, const double4_32a& p1, double v[3]) {
  const double dx = p1.x - p0.x;
  if (dx == 0.0) return false;
  const double m = (p1.y - p0.y) / dx;
  v[0] = m;
  v[1] = p0.y - m * p0.x;
  v[2] = sqrt(m * m + 1.0);
  return true;
}

// The same of trial h, through its two seed points.
__device__ __forceinline__ bool line_hyp64(const FrameDesc& a, const double4_32a* pre, int ci, int h, int N, double v[3]) {
  int q[3];
  draw_minimal_set<2>(a.key, a.cluster_base + ci, h, N, q);
  return line_seeds64(pre[q[0]], pre[q[1]], v);
}

// FP32 scoring record of an FP64 line: (-m32, -c32, 0, thi) and tlo, such
// that with rows (x32, 1, y32) the FP32 residual r32 = fmaf(-m32, x32,
// fmaf(-c32, 1, y32)) satisfies |r32| <= tlo => inlier and |r32| > thi =>
// outlier under line_in64.  With |x|, |y| <= 1 (normalised), rounding the
// inputs and the arithmetic to FP32 moves the residual by at most
// u (2.01 (1 + |c| + |m|) + 1.0001 |r|), the FP64 residual carries
// 3 * 2^-53 (1 + |c| + |m|), and the FP64 quotient test is certain outside
// T distd (1 -+ 2^-50); b below covers both sides with margin.
__device__ __forceinline__ Hyp32 line_record(const double v[3], double T) {
  Hyp32 h;
  h.refined = 0;
  h.nx = -__double2float_rn(v[0]);
  h.ny = -__double2float_rn(v[1]);
  const double td = T * v[2];
  const double am = fabs(v[0]), ac = fabs(v[1]);
  const double b = (0x1p-22 * (1.0 + ac + am + td) + 0x1p-50 * (1.0 + ac + am)) * (1.0 + 0x1p-20);
  const double hi = td * (1.0 + 0x1p-50) + b, lo = td * (1.0 - 0x1p-50) - b;
  h.kind = kHypNormal;
  h.thi = __double2float_ru(hi);
  h.nz = h.tlo = lo >= 0.0 ? __double2float_rd(lo) : -1.0f;
  if (!(hi < 1e30) || !(am < 0x1p60) || !(ac < 0x1p60)) {  // residuals below 2^62: finite squares
    h.kind = kHypExactOnly;
    h.thi = __int_as_float(0x7f800000);
    h.nz = h.tlo = -1.0f;
  }
  return h;
}

// The same record from the FP32 rows p, q of the two seed points, for seeds
// at least kLineDx apart in x (kHypUndecided otherwise): FP64 there cost the
// trial stage a quarter of the line model's time.  With u = 2^-24 the
// coordinates are within u / 2 of the FP64 ones and the differences dx, dy
// within u + u|d| <= 2u, so the slope is within dm = 2u (1 + |m|) / |dx| + 4u |m|
// of the FP64 line's (rcp_approx and one rounding: below 4u).  Against the
// line through the seeds, r32 carries the points' rounding u (1 + |m|), dm
// times |x - x0| <= 1, the roundings of c and of two FMAs u (1 + 2|c| + |r|);
// FP64's own share is 2^-50 (1 + |c| + |m|) as above; distd moves by at most
// dm and its FP32 evaluation by 2^-21 of it.
constexpr float kLineDx = 0x1p-12f;
__device__ __forceinline__ Hyp32 line_record_f32(float4 p, float4 q, TauPair T) {
  Hyp32 h;
  h.refined = 0;
  const float dx = q.x - p.x, dy = q.z - p.z;
  const float r = rcp_approx(dx);
  const float m = dy * r, c = fmaf(-m, p.x, p.z);
  const float am = fabsf(m), ac = fabsf(c);
  const float dm = kU * (2.01f * (1.0f + am) * fabsf(r) + 4.01f * am);
  const float sd = sqrt_approx(fmaf(m, m, 1.0f));
  const float th = T.hi * (sd * (1.0f + 0x1p-20f) + dm) * (1.0f + 0x1p-20f);
  const float tl = T.lo * (sd * (1.0f - 0x1p-20f) - dm) * (1.0f - 0x1p-20f);
  const float b = (kU * (2.0f + am + 2.0f * ac + th) + dm) * (1.0f + 0x1p-10f);
  h.nx = -m;
  h.ny = -c;
  h.thi = __fadd_ru(th, b);
  const float lo = __fsub_rd(tl, b);
  h.nz = h.tlo = lo >= 0.0f ? lo : -1.0f;
  h.kind = kHypNormal;
  if (!(fabsf(dx) >= kLineDx) || !(h.thi < 1e30f)) h.kind = kHypUndecided;
  return h;
}

// k-th smallest (0-based, k < N) of N keys: key(j) as 64-bit patterns of
// non-negative doubles (monotone as integers; NaN sorts last), by radix digits
// of 8 bits from the top.  hist: 256 ints of shared memory.  Exact: returns
// the key.
template <typename Key>
__device__ __noinline__ unsigned long long block_select(Key key, int N, int k, int* hist, ClusterShared& cs) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned long long prefix = 0ull, hmask = 0ull;
  for (int shift = 56; shift >= 0; shift -= 8) {
    hist[tid] = 0;  // kThreads == 256 bins
    __syncthreads();
    for (int j = tid; j < N; j += kThreads) {
      const unsigned long long kb = key(j);
      if ((kb & hmask) == prefix) atomicAdd(&hist[(int)((kb >> shift) & 255ull)], 1);
    }
    __syncthreads();
    if (warp == 0) {
      int c[8], tot = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        c[i] = hist[8 * lane + i];
        tot += c[i];
      }
      int incl = tot;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
      }
      const int excl = incl - tot;
      if (excl <= k && k < incl) {
        int kk = k - excl, d = 0;
        while (d < 7 && kk >= c[d]) kk -= c[d++];
        cs.sel_digit = 8 * lane + d;
        cs.sel_k = kk;
      }
    }
    __syncthreads();
    prefix |= (unsigned long long)cs.sel_digit << shift;
    hmask |= 0xFFull << shift;
    k = cs.sel_k;
  }
  return prefix;
}

// Bin 0 .. kMedianBins - 1 of a key, monotone in it: the double truncated to
// FP32 (its high bits; below 2^-126: 0) times the number of bins, NaN and
// anything from 1 on in the last.
constexpr int kMedianBins = 1024;
constexpr int kMedianList = 512;
__device__ __forceinline__ int median_bin(unsigned long long key) {
  const int hi = (int)(key >> 32);
  if (hi < 0x38100000) return 0;
  if (hi >= 0x3ff00000) return kMedianBins - 1;
  const float f = __int_as_float(((hi - 0x38000000) << 3) | (int)((unsigned)key >> 29));
  return (int)(f * (float)kMedianBins);
}

// Median of N keys (even N: 0.5 * (lower + upper middle)), exact: a histogram
// of kMedianBins even bins over [0, 1] finds the bins of the two middle
// ranks, whose few keys are ranked against each other; more than kMedianList
// keys in them (few distinct values) go to the radix select.  Two passes over
// the keys instead of eight per middle: the radix selects over global memory
// took 44% of the line model's time (dense2d 0.69 -> 0.47 ms).  hist:
// kMedianBins ints, list: kMedianList keys of shared memory.
template <typename Key>
__device__ __forceinline__ double block_median(Key key, int N, int* hist, unsigned long long* list,
                                               ClusterShared& cs) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k1 = N >> 1, k0 = (N & 1) ? k1 : k1 - 1;
  constexpr int kPer = kMedianBins / kThreads;
#pragma unroll
  for (int i = 0; i < kPer; ++i) hist[tid + i * kThreads] = 0;
  if (tid == 0) cs.sel_n = 0;
  __syncthreads();
  for (int j = tid; j < N; j += kThreads) atomicAdd(&hist[median_bin(key(j))], 1);
  __syncthreads();
  int c[kPer], tot = 0;
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    c[i] = hist[kPer * tid + i];
    tot += c[i];
  }
  int incl = tot;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
  if (lane == 31) cs.red_i[warp] = incl;
  __syncthreads();
  int below = incl - tot;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) below += w < warp ? cs.red_i[w] : 0;
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    if (below <= k0 && k0 < below + c[i]) {
      cs.sel_digit = kPer * tid + i;
      cs.sel_k = k0 - below;  // rank of the lower middle among the listed keys
    }
    if (below <= k1 && k1 < below + c[i]) cs.sel_hi = kPer * tid + i;
    below += c[i];
  }
  __syncthreads();
  const int b0 = cs.sel_digit, b1 = cs.sel_hi;  // no key lies in a bin between them
  for (int j = tid; j < N; j += kThreads) {
    const unsigned long long kb = key(j);
    const int b = median_bin(kb);
    if (b == b0 || b == b1) {
      const int pos = atomicAdd(&cs.sel_n, 1);
      if (pos < kMedianList) list[pos] = kb;
    }
  }
  __syncthreads();
  const int m = cs.sel_n, r0 = cs.sel_k;
  if (m > kMedianList) {
    const double hi = __longlong_as_double((long long)block_select(key, N, k1, hist, cs));
    if (N & 1) return hi;
    const double lo = __longlong_as_double((long long)block_select(key, N, k0, hist, cs));
    return 0.5 * (lo + hi);
  }
  for (int i = tid; i < m; i += kThreads) {
    const unsigned long long ki = list[i];
    int rank = 0;
    for (int t = 0; t < m; ++t) rank += list[t] < ki || (list[t] == ki && t < i) ? 1 : 0;
    if (rank == r0) cs.sel_key[0] = ki;
    if (rank == r0 + (k1 - k0)) cs.sel_key[1] = ki;
  }
  __syncthreads();
  const double lo = __longlong_as_double((long long)cs.sel_key[0]);
  const double hi = __longlong_as_double((long long)cs.sel_key[1]);
  return (N & 1) ? hi : 0.5 * (lo + hi);
}

// Bytes of the trial area of shared memory: hchunk trials, and at least the
// final reduction (up to 9 sums per thread).
__host__ __device__ constexpr size_t trial_area_bytes(int hchunk) {
  const size_t trials = (size_t)hchunk * (sizeof(float4) + sizeof(float) + sizeof(int) + sizeof(uint16_t)) +
                        (((size_t)hchunk + 15) & ~(size_t)15);
  const size_t reduction = (size_t)9 * kThreads * sizeof(double);
  return trials > reduction ? trials : reduction;
}

// The line model's rows stage: min / max of azimuth and Doppler, normalised
// FP64 points into the FP64 slots and FP32 rows (x, 1, y) into the scoring
// rows, then the MAD threshold into cs.ln_T.  Normalisation (the paper's
// normalize(), undefined there): min-max scaling, x = (t - t_min) *
// (1 / (t_max - t_min)), 0 when the range is empty.  The trial area of shared
// memory is free at this point: it holds the medians' histogram and list, and
// the FP64 Dopplers of as many points as fit the rest (2432 with the default
// sizes; larger clusters read them back from their slots).  Out of line:
// runs once per cluster.
template <typename RV>
__device__ __noinline__ void line_rows_and_threshold(const FrameDesc& a, const RV rows, double4_32a* pre, int64_t o,
                                                     int N, const Smem& S, int hchunk, ClusterShared& cs) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float inf = __int_as_float(0x7f800000);
  float m4[4] = {inf, inf, inf, inf};  // min t, -max t, min v, -max v
  for (int j = tid; j < N; j += kThreads) {
    const float t = a.az[o + j], v = a.dop[o + j];
    m4[0] = fminf(m4[0], t);
    m4[1] = fminf(m4[1], -t);
    m4[2] = fminf(m4[2], v);
    m4[3] = fminf(m4[3], -v);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = __reduce_min_sync(0xffffffffu, float_order(m4[i]));
    if (lane == 0) cs.red_d[i][warp] = r;
  }
  __syncthreads();
  if (tid < 2) {  // azimuth, Doppler
    int lo = cs.red_d[2 * tid][0], hi = cs.red_d[2 * tid + 1][0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) {
      lo = min(lo, cs.red_d[2 * tid][w]);
      hi = min(hi, cs.red_d[2 * tid + 1][w]);
    }
    const double l = (double)order_float(lo), h = -(double)order_float(hi);
    cs.ln_min[tid] = l;
    cs.ln_scale[tid] = h > l ? 1.0 / (h - l) : 0.0;
  }
  __syncthreads();
  const double tmin = cs.ln_min[0], vmin = cs.ln_min[1], rt = cs.ln_scale[0], rv = cs.ln_scale[1];
  int* hist = reinterpret_cast<int*>(S.hyp);
  unsigned long long* list = reinterpret_cast<unsigned long long*>(hist + kMedianBins);
  double* sy = reinterpret_cast<double*>(list + kMedianList);
  const bool in_smem =
      N <= (int)((trial_area_bytes(hchunk) - kMedianBins * sizeof(int)) / sizeof(double)) - kMedianList;
  for (int j = tid; j < N; j += kThreads) {
    const float az = a.az[o + j];
    const double x = ((double)az - tmin) * rt;
    const double y = ((double)a.dop[o + j] - vmin) * rv;
    pre[j] = make_double4_32a(x, y, 0.0, 0.0);
    rows.put(j, make_float4(__double2float_rn(x), 1.0f, __double2float_rn(y), az));
    if (in_smem) sy[j] = y;
  }
  // Eq. eq:MAD read as the median absolute deviation of the normalised
  // Doppler; each thread reads the keys it wrote
  auto y_at = [&](int j) { return in_smem ? sy[j] : pre[j].y; };
  auto bits = [](double d) { return (unsigned long long)__double_as_longlong(fabs(d)); };
  const double med = block_median([&](int j) { return bits(y_at(j)); }, N, hist, list, cs);
  const double T = block_median([&](int j) { return bits(y_at(j) - med); }, N, hist, list, cs);
  if (tid == 0) cs.ln_T = T;
  __syncthreads();
}

// Exact count of one trial by the whole CTA: FP32 certainties, then an FP64
// re-decision of the points inside the trial's error band.  When there are
// band points the trial's FP64 velocity is left in cs.cv64 and *band > 0.
template <int DIM, typename RV, bool EXT>
__device__ int exact_count_block(const FrameDesc& a, const RV rows, const Rows64<DIM>& R,
                                 int ci, int h, int N, float4 hy, float tlo, ClusterShared& cs, int* band) {
  const int tid = threadIdx.x;
  unsigned in = 0, near = 0;
  for (int j = tid; j < N; j += kThreads) {
    const float r = fabsf(resid_f32<DIM>(rows.at(j), hy.x, hy.y, hy.z));
    if (r <= tlo) ++in;
    else if (!(r > hy.w)) ++near;
  }
  const unsigned long long lb = block_sum2(in, near, cs.red_v);
  const int L = (int)(lb & 0xFFFFFFFFull), B = (int)(lb >> 32);
  *band = B;
  if (B == 0) return L;
  __syncthreads();
  if (tid == 0) {
    double v[3] = {0.0, 0.0, 0.0};
    if constexpr (EXT && DIM == 2) {
      if (a.line_model) line_hyp64(a, R.pre, ci, h, N, v);
      else hyp_f64<DIM>(a, R, ci, h, N, v);
    } else {
      hyp_f64<DIM>(a, R, ci, h, N, v);
    }
    cs.cv64[0] = v[0];
    cs.cv64[1] = v[1];
    cs.cv64[2] = v[2];
    cs.ctr[1] += (unsigned long long)B;
  }
  __syncthreads();
  const double v[3] = {cs.cv64[0], cs.cv64[1], cs.cv64[2]};
  unsigned lbin = 0;
  auto cosine_band = [&]() {
    for (int j = tid; j < N; j += kThreads) {
      const float4 row = rows.at(j);
      const float r = fabsf(resid_f32<DIM>(row, hy.x, hy.y, hy.z));
      if (!(r <= tlo) && !(r > hy.w)) {
        const double4_32a s = R.at(j, row);
        const double a64[3] = {s.x, s.y, s.z};
        if (fabs(residual_f64<DIM>(a64, s.w, v)) <= a.tau) ++lbin;
      }
    }
  };
  if constexpr (EXT && DIM == 2) {
    if (a.line_model) {
      for (int j = tid; j < N; j += kThreads) {
        const float r = fabsf(resid_f32<DIM>(rows.at(j), hy.x, hy.y, hy.z));
        if (!(r <= tlo) && !(r > hy.w)) {
          const double4_32a p = R.pre[j];
          if (line_in64(v[0], v[1], v[2], p.x, p.y, cs.ln_T)) ++lbin;
        }
      }
    } else {
      cosine_band();
    }
  } else {
    cosine_band();
  }
  return L + (int)block_sum2(lbin, 0u, cs.red_v);
}

template <int DIM>
__device__ void write_invalid(const FrameDesc& a, int ci, int st) {
  a.vx[ci] = __longlong_as_double(0x7ff8000000000000LL);
  a.vy[ci] = __longlong_as_double(0x7ff8000000000000LL);
  if (a.vz) a.vz[ci] = __longlong_as_double(0x7ff8000000000000LL);
  a.heading[ci] = __longlong_as_double(0x7ff8000000000000LL);
  a.inlier_count[ci] = 0;
  a.best[ci] = -1;
  a.status[ci] = st;
}

// a8: normal equations G v = g over the inliers (sums t: 2D Scc, Scs, Sss,
// Scv, Ssv; 3D the six entries of G then g), solved by Cramer's rule when
// there are at least k inliers and |det G| > 1e-12 trace^k.  Returns false
// (v untouched) otherwise.  The local-optimisation rounds and the final
// solve both use this, so a set accepted by a round solves identically.
template <int DIM>
__device__ __forceinline__ bool normal_solvable(const double* t, int n_in) {
  if (DIM == 2) {
    const double tr = t[0] + t[2];
    return n_in >= 2 && fabs(det2_f64(t[0], t[1], t[1], t[2])) > 1e-12 * (tr * tr);
  }
  const double tr = t[0] + t[3] + t[5];
  const double G0[3] = {t[0], t[1], t[2]}, G1[3] = {t[1], t[3], t[4]}, G2[3] = {t[2], t[4], t[5]};
  return n_in >= 3 && fabs(det3_f64(G0, G1, G2)) > 1e-12 * (tr * tr * tr);
}

template <int DIM>
__device__ __forceinline__ bool solve_normal(const double* t, int n_in, double v[3]) {
  if (!normal_solvable<DIM>(t, n_in)) return false;
  if (DIM == 2) {
    const double G0[3] = {t[0], t[1], 0.0}, G1[3] = {t[1], t[2], 0.0}, g[3] = {t[3], t[4], 0.0};
    double vs[3];
    solve_f64<2>(G0, G1, nullptr, g, 0.0, vs, nullptr);
    v[0] = vs[0];
    v[1] = vs[1];
    v[2] = 0.0;
    return true;
  } else {
    const double G0[3] = {t[0], t[1], t[2]}, G1[3] = {t[1], t[3], t[4]}, G2[3] = {t[2], t[4], t[5]};
    const double g[3] = {t[6], t[7], t[8]};
    double vs[3];
    solve_f64<3>(G0, G1, G2, g, 0.0, vs, nullptr);
    v[0] = vs[0];
    v[1] = vs[1];
    v[2] = vs[2];
    return true;
  }
}

// Final solve of a cluster: the normal equations, with a fallback to the
// winning minimal-set velocity (whose heading is formed here too).  One thread.
template <int DIM, bool EXT>
__device__ __noinline__ void finish_cluster(const FrameDesc& a, const Rows64Inputs<DIM>& R, int ci, int N, int hstar, int n_in,
                               const double* t, const double* v64, bool has_v64) {
  double vout[3] = {v64[0], v64[1], v64[2]};
  int st = 0;
  const bool ok = solve_normal<DIM>(t, n_in, vout);
  if (!ok) {
    st |= RVH_STATUS_LSQ_FALLBACK;
    if constexpr (EXT && DIM == 2) {
      if (a.line_model) {  // a line has no velocity to fall back to
        vout[0] = vout[1] = vout[2] = __longlong_as_double(0x7ff8000000000000LL);
      } else if (!has_v64) {
        hyp_f64<DIM>(a, R, ci, hstar, N, vout);
      }
    } else {
      if (!has_v64) hyp_f64<DIM>(a, R, ci, hstar, N, vout);
    }
    a.heading[ci] = atan2(vout[1], vout[0]);
  }
  a.vx[ci] = vout[0];
  a.vy[ci] = vout[1];
  if (a.vz) a.vz[ci] = DIM == 3 ? vout[2] : 0.0;
  a.inlier_count[ci] = n_in;
  a.best[ci] = hstar;
  a.status[ci] = st;
}

// Heading of a cluster whose normal equations are solvable (else
// finish_cluster forms it): atan2 of Cramer's numerators, so that it does not
// wait for the velocity's divisions.  One thread, in another warp than
// finish_cluster's.  A frame of few clusters ends with these two, one cluster
// per CTA: one thread doing both, with the library's atan2, took 2.8 us of it;
// 64 clusters 20.6 -> 19.5 us.
template <int DIM>
__device__ __noinline__ void finish_heading(const FrameDesc& a, int ci, int n_in, const double* t) {
  if (!normal_solvable<DIM>(t, n_in)) return;
  double det, x, y;
  if (DIM == 2) {
    det = det2_f64(t[0], t[1], t[1], t[2]);
    x = det2_f64(t[3], t[1], t[4], t[2]);
    y = det2_f64(t[0], t[3], t[1], t[4]);
  } else {
    const double G0[3] = {t[0], t[1], t[2]}, G1[3] = {t[1], t[3], t[4]}, G2[3] = {t[2], t[4], t[5]};
    const double A0[3] = {t[6], t[1], t[2]}, A1[3] = {t[7], t[3], t[4]}, A2[3] = {t[8], t[4], t[5]};
    const double B0[3] = {t[0], t[6], t[2]}, B1[3] = {t[1], t[7], t[4]}, B2[3] = {t[2], t[8], t[5]};
    det = det3_f64(G0, G1, G2);
    x = det3_f64(A0, A1, A2);
    y = det3_f64(B0, B1, B2);
  }
  if (det < 0.0) {
    x = -x;
    y = -y;
  }
  a.heading[ci] = atan2_table(a.trig, y, x);
}

// A cluster waiting for its final solve and heading: the
// CTA queues up to kFinishBatch of them in shared memory and finishes them
// together, one lane each.  Serial FP64 on one lane costs as much pipe time
// per instruction as a full warp, so a lone thread finishing each cluster
// kept the other 255 threads at the next barrier for microseconds.
constexpr int kFinishBatch = 16;
struct FinishRec {
  double t[9];
  double v64[3];
  int64_t o;
  int n_in, hstar, ci, frame, N, has_v64;
};

// Accumulates the normal-equation sums of one inlier row (a0, a1, a2, w).
template <int DIM>
__device__ __forceinline__ void accumulate_row(double* sums, const double4_32a& s) {
  if (DIM == 2) {
    sums[0] = fma(s.x, s.x, sums[0]);
    sums[1] = fma(s.x, s.y, sums[1]);
    sums[2] = fma(s.y, s.y, sums[2]);
    sums[3] = fma(s.x, s.w, sums[3]);
    sums[4] = fma(s.y, s.w, sums[4]);
  } else {
    sums[0] = fma(s.x, s.x, sums[0]);
    sums[1] = fma(s.x, s.y, sums[1]);
    sums[2] = fma(s.x, s.z, sums[2]);
    sums[3] = fma(s.y, s.y, sums[3]);
    sums[4] = fma(s.y, s.z, sums[4]);
    sums[5] = fma(s.z, s.z, sums[5]);
    sums[6] = fma(s.x, s.w, sums[6]);
    sums[7] = fma(s.y, s.w, sums[7]);
    sums[8] = fma(s.z, s.w, sums[8]);
  }
}

// a7 + a8: decides every point of the cluster against one velocity (FP32
// certainties from the record hy / tlo, FP64 re-decisions with v64 inside
// the band), writes the mask, and reduces the normal-equation sums of the
// inliers into cs.red_t.  Returns the inlier count; with later (a pass after
// the cluster's first), *changed receives the number of mask entries that
// differ from what the mask held before.  The trial area of shared memory is free at this point
// and holds the reduction.
template <int DIM, typename RV, bool EXT>
__device__ __forceinline__ int mask_and_sums(const FrameDesc& a, const RV rows, const Rows64<DIM>& R, int64_t o, int N,
                                             float4 hy, float tlo, const double v64[3], const Smem& S,
                                             ClusterShared& cs, bool later, int* changed) {
  const int tid = threadIdx.x;
  constexpr int NS = DIM == 2 ? 5 : 9;
  // 2D rows of the local-optimisation rounds: the first pass over a cluster
  // (later = false, the mask not written yet) leaves each inlier's
  // (cos, sin) in the cluster's FP64 row slot, which the 2D model does not
  // use otherwise; later passes read it back where the mask says that the
  // point was an inlier before, 16 bytes from L2 in place of the 12 FP64
  // instructions (of 17 per inlier) that bound this pass: two rounds on 4096
  // clusters of 8..2048 points 0.411 -> 0.334 ms.
  double2* const kept = EXT && DIM == 2 && a.lo_iters > 0 ? reinterpret_cast<double2*>(R.pre) : nullptr;
  double sums[NS];
#pragma unroll
  for (int i = 0; i < NS; ++i) sums[i] = 0.0;
  int nin = 0, nch = 0;
  auto cosine_pass = [&]() {
    for (int j = tid; j < N; j += kThreads) {
      const float4 row = rows.at(j);
      const float r = fabsf(resid_f32<DIM>(row, hy.x, hy.y, hy.z));
      bool in = r <= tlo;
      const bool band = !in && !(r > hy.w);
      const uint8_t was = EXT && later ? a.mask[o + j] : 0;
      if (in || band) {
        double4_32a s;
        if (EXT && DIM == 2 && was) {
          const double2 cs2 = kept[j];
          s = make_double4_32a(cs2.x, cs2.y, 0.0, (double)row.z);
        } else {
          s = R.at(j, row);
          if (EXT && DIM == 2 && kept) kept[j] = make_double2(s.x, s.y);
        }
        if (band) {
          const double a64[3] = {s.x, s.y, s.z};
          in = fabs(residual_f64<DIM>(a64, s.w, v64)) <= a.tau;
        }
        if (in) {
          ++nin;
          accumulate_row<DIM>(sums, s);
        }
      }
      if (EXT && later) nch += (was != (in ? 1 : 0));
      a.mask[o + j] = in ? 1 : 0;
    }
  };
  if constexpr (EXT && DIM == 2) {
    if (a.line_model) {
      // the line model decides its band points by Alg. 1's distance test
      for (int j = tid; j < N; j += kThreads) {
        const float r = fabsf(resid_f32<DIM>(rows.at(j), hy.x, hy.y, hy.z));
        bool in = r <= tlo;
        if (!in && !(r > hy.w)) {
          const double4_32a p = R.pre[j];
          in = line_in64(v64[0], v64[1], v64[2], p.x, p.y, cs.ln_T);
        }
        if (in) {
          ++nin;
          accumulate_row<DIM>(sums, R.at(j));
        }
        a.mask[o + j] = in ? 1 : 0;
      }
    } else {
      cosine_pass();
    }
  } else {
    cosine_pass();
  }
  // Reduce the per-thread sums through shared memory: warp i sums sum i,
  // each lane a strided share of the threads that held points, then a
  // shuffle tree; 12 dependent FP64 adds per sum.
  const int warp = tid >> 5, lane = tid & 31;
  nin = warp_sum(nin);
  if (EXT && later) nch = warp_sum(nch);
  const int nact = min(N, kThreads);
  double* red = reinterpret_cast<double*>(S.hyp);  // NS x kThreads
  if (tid < nact) {
#pragma unroll
    for (int i = 0; i < NS; ++i) red[i * kThreads + tid] = sums[i];
  }
  if (lane == 0) {
    cs.red_i[warp] = nin;
    cs.red_c[warp] = nch;
  }
  __syncthreads();
  for (int i = warp; i < NS; i += kWarps) {
    double acc = 0.0;
    for (int k = lane; k < nact; k += 32) acc += red[i * kThreads + k];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) cs.red_t[i] = acc;
  }
  int n_in = 0, n_ch = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    n_in += cs.red_i[w];
    n_ch += cs.red_c[w];
  }
  __syncthreads();
  if (changed) *changed = n_ch;
  return n_in;
}

// Local-optimisation rounds (refine_iterations > 0): solve the current set,
// re-threshold every point against that velocity, keep the new set if its
// normal equations are solvable (else restore the previous set by
// re-deciding with the record and velocity that produced it), stop when
// nothing changes.  Starts from the winner's set (its sums in cs.red_t) and
// returns the final set's inlier count, its sums left in cs.red_t.  Kept out
// of line so that the default path's register allocation does not carry it.
template <int DIM, typename RV>
__device__ __noinline__ int local_opt_rounds(const FrameDesc& a, const RV rows, const Rows64<DIM>& R, int64_t o, int N,
                                             float4 gen_hy, float gen_tlo, const double* v64, float wmax, int n_in,
                                             const Smem& S, ClusterShared& cs) {
  const int tid = threadIdx.x;
  double gen_v[3] = {v64[0], v64[1], v64[2]};  // the FP64 velocity that produced the current set
  for (int it = 0; it < a.lo_iters; ++it) {
    if (tid == 0) {
      double v[3] = {0.0, 0.0, 0.0};
      cs.lo_ok = solve_normal<DIM>(cs.red_t, n_in, v) ? 1 : 0;
      if (cs.lo_ok) {
        cs.lo_v[0] = v[0];
        cs.lo_v[1] = v[1];
        cs.lo_v[2] = v[2];
        velocity_record<DIM>(v, wmax, a.tau32, &cs.lo_hy, &cs.lo_tlo);
      }
    }
    __syncthreads();
    if (!cs.lo_ok) break;
    const float4 nhy = cs.lo_hy;
    const float ntlo = cs.lo_tlo;
    const double nv[3] = {cs.lo_v[0], cs.lo_v[1], cs.lo_v[2]};
    int changed = 0;
    const int n2 = mask_and_sums<DIM, RV, true>(a, rows, R, o, N, nhy, ntlo, nv, S, cs, true, &changed);
    if (changed == 0) break;  // same set, same sums
    // the next round solves it, if there is one
    if (tid == 0) cs.lo_ok = normal_solvable<DIM>(cs.red_t, n2) ? 1 : 0;
    __syncthreads();
    if (!cs.lo_ok) {
      n_in = mask_and_sums<DIM, RV, true>(a, rows, R, o, N, gen_hy, gen_tlo, gen_v, S, cs, true, nullptr);
      break;
    }
    gen_hy = nhy;
    gen_tlo = ntlo;
    gen_v[0] = nv[0];
    gen_v[1] = nv[1];
    gen_v[2] = nv[2];
    n_in = n2;
  }
  return n_in;
}

// Keeps, in order, the trials at positions 0 .. n - 1 of the staged pass's
// list (list_trial) for which keep(h) holds, writing them to S.list[0 ..);
// returns how many.  Entries are read before any is written (compaction in
// place).  red: kWarps ints of shared memory.
template <bool LISTED, typename Keep>
__device__ __forceinline__ int prune_list(const Smem& S, int n, Keep keep, int* red) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int out = 0;
  for (int r0 = 0; r0 < n; r0 += 4 * kThreads) {
    int hv[4], c = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      int h = list_trial<LISTED>(S, n, r0 + 4 * tid + k);
      if (h >= 0 && !keep(h)) h = -1;
      hv[k] = h;
      c += h >= 0 ? 1 : 0;
    }
    int incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += t;
    }
    if (lane == 31) red[warp] = incl;
    __syncthreads();
    int pos = out + incl - c, tot = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const int v = red[w];
      tot += v;
      pos += w < warp ? v : 0;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (hv[k] >= 0) S.list[pos++] = (uint16_t)hv[k];
    out += tot;
    __syncthreads();
  }
  return out;
}

// ---- the staged scoring pass (a4 with exact pruning) ---------------------------------
// Quads (4 points) of the first stage and of the next one; the third stage is
// twice the second, the fourth twice the third, and a fifth takes all other
// points (a last stage of less than half the one before is joined to that).
// Clusters of fewer than kStageMinPoints points are scored in one pass.  What bounds the pass is the FP32 scoring of the
// pairs that stay (8.6e12 pairs/s inside the kernel, 9.15e12 in isolation),
// then the lead pass, the histograms' scans and the first pruning test,
// together about 40 points' worth of scoring 1024 trials.  Measured, ms per
// frame (dense2d / stress2d / dense3d): without the pass 0.292 / 0.846 /
// 1.93; pruning by "every point still to come" instead of the lead's
// residuals (72% / 100% / 66% of the pairs) 0.261 / 0.845 / 1.688; this pass
// (42% / 59% / 38%) 0.221 / 0.787 / 1.480.  2D: first stage of 64 / 96 / 128
// points 0.229 / 0.224 / 0.221 (a longer one finds a better lead), threshold
// of 192 instead of 256 points 0.223 / 0.802; a new lead after every early
// stage evaluates fewer pairs (29%) but took 0.305 ms.  3D with an interval
// per half of a2 (27% of the pairs): 1.372 -> 1.229 ms, and with its tighter
// first test a first stage of 96 / 64 points 1.218 / 1.220, threshold 192 /
// 128 points at 64 1.210 / 1.209.
template <int DIM>
constexpr int kStage0Quads = DIM == 2 ? 32 : 16;
constexpr int kStage1Quads = 32;
template <int DIM>
constexpr int kStageMinPoints = DIM == 2 ? 256 : 128;
constexpr int kStageMaxPoints = 32767;  // points are counted in 16-bit halves

// The cluster's direction range (DirRange) from this thread's own rows: each
// warp's part into cs.red_d; the caller's next barrier is followed by
// direction_range_finish.
template <int DIM, typename RV>
__device__ __forceinline__ void direction_range(const RV rows, int N, bool line, ClusterShared& cs) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float inf = __int_as_float(0x7f800000);
  float a0 = inf, t0 = inf, t1 = -inf, z0 = inf, z1 = -inf;
  for (int j = tid; j < N; j += kThreads) {
    const float4 p = rows.at(j);
    const float t = row_tan(p, line);
    a0 = fminf(a0, line ? p.y : p.x);
    t0 = fminf(t0, t);
    t1 = fmaxf(t1, t);
    if (DIM == 3) {
      z0 = fminf(z0, p.z);
      z1 = fmaxf(z1, p.z);
    }
  }
  const int r0 = __reduce_min_sync(0xffffffffu, float_order(a0)), r1 = __reduce_min_sync(0xffffffffu, float_order(t0)),
            r2 = __reduce_max_sync(0xffffffffu, float_order(t1)),
            r3 = DIM == 3 ? __reduce_min_sync(0xffffffffu, float_order(z0)) : 0,
            r4 = DIM == 3 ? __reduce_max_sync(0xffffffffu, float_order(z1)) : 0;
  if (lane == 0) {
    cs.red_d[0][warp] = r0;
    cs.red_d[1][warp] = r1;
    cs.red_d[2][warp] = r2;
    cs.red_d[3][warp] = r3;
    cs.red_d[4][warp] = r4;
  }
}

template <int DIM>
__device__ __forceinline__ void direction_range_finish(ClusterShared& cs) {
  if (threadIdx.x != 0) return;
  int r[5];
#pragma unroll
  for (int i = 0; i < (DIM == 3 ? 5 : 3); ++i) {
    r[i] = cs.red_d[i][0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w)
      r[i] = i == 2 || i == 4 ? max(r[i], cs.red_d[i][w]) : min(r[i], cs.red_d[i][w]);
  }
  const float a0 = order_float(r[0]), t0 = order_float(r[1]), t1 = order_float(r[2]);
  const float inv = __fdividef(kTanBins - 0.01f, t1 - t0);
  cs.dir.t0 = t0;
  cs.dir.tinv = t1 > t0 && inv < 1e30f ? inv : 0.0f;  // else one bin holds them all
  cs.dir.tabs = fmaxf(fabsf(t0), fabsf(t1));
  cs.dir.a0inv = rcp_approx(a0) * kRcpUp;
  cs.dir.tan_ok = a0 > 1e-3f && a0 < 2.0f;
  if (DIM == 3) {
    const float z0 = order_float(r[3]), z1 = order_float(r[4]);
    cs.dir.zmax = fmaxf(fabsf(z0), fabsf(z1));
    cs.dir.z0 = z0;
    // a little wide: centre +- zq holds its half whatever the rounding
    cs.dir.zq = 0.25f * (z1 - z0) + 1e-6f;
  } else {
    cs.dir.zmax = cs.dir.z0 = cs.dir.zq = 0.0f;
  }
}

// Scores the chunk's normal trials in stages.  After the first stage the
// trial with the highest partial count becomes the lead (a later chunk
// starts from the lead it finds); one pass over the points counts the lead
// and takes the histograms of its residuals over the points still to be
// scored.  A trial whose partial count plus the points still to come that it
// can hold (lead_bound, its counts per stage) cannot beat the lead's key
// leaves the list, U = -1.  That sum is no less than the trial's exact
// count, and the lead is ranked by the points it certainly holds, so a trial
// dropped this way cannot win: the winner is the one that scoring every
// trial over every point gives, found by the best-first counts among the
// trials that stayed.  Returns the (trial, point) pairs scored by this warp.
template <int DIM, bool EXT, typename RV>
__device__ __forceinline__ unsigned long long staged_pass(const FrameDesc& a, const RV rows, const Smem& S,
                                                          ClusterShared& cs, int hc0, int nh, int N,
                                                          unsigned long long* n_cand) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool line = EXT && DIM == 2 && a.line_model;
  const int nq = (N + 3) >> 2;
  unsigned long long scored = 0;
  unsigned top = 0;
  // pieces of (trial group, quad) units of quads [qa, qb), split evenly over the warps
  auto score = [&](auto listed, int A, int qa, int qb) {
    constexpr int G = 32 * kStagedHpl<decltype(listed)::value>;
    const int span = qb - qa, total = ((A + G - 1) / G) * span;
    const int per = (total + kWarps - 1) / kWarps;
    for (int u = warp * per, e = min(total, u + per); u < e;) {
      const int g = u / span, a0 = qa + u % span, a1 = min(qb, a0 + (e - u));
      scored += score_segment<DIM, decltype(listed)::value>(rows, N, S, A, g, a0, a1, &top);
      u += a1 - a0;
    }
  };
  constexpr int NH = kHalves<DIM>, kIn = NH * (kTanBins + 1);
  if (tid < 2 * kIn) cs.lead_in[tid] = 0u;
  if (tid < 2 * kExcessBins) cs.lead_out[tid] = 0u;
  unsigned long long lim = cs.best;  // the key to beat
  int q0 = 0, lead = -1;
  float4 lw = cs.win;
  if (lim == 0ull || !(lw.w < 1e30f)) {  // no lead with an FP32 record yet
    score(std::false_type{}, nh, 0, kStage0Quads<DIM>);
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) cs.red_i[warp] = (int)top;
    __syncthreads();
    top = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) top = max(top, (unsigned)cs.red_i[w]);
    if (top == 0u) return scored;  // no normal trial
    q0 = kStage0Quads<DIM>;
    lead = 0xFFFF - (int)(top & 0xFFFFu);
    lw = S.hyp[lead];
  } else {
    __syncthreads();
  }
  const int e1 = q0 + kStage1Quads, e2 = e1 + 2 * kStage1Quads, e3 = e2 + 4 * kStage1Quads;
  const DirRange dir = cs.dir;
  const float ltlo = record_tlo(lw, a.tau32, line);
  {
    // the lead's count and the histograms
    unsigned cnt = 0;  // certain and band points in 16-bit halves
    for (int j = tid; j < N; j += kThreads) {
      const float4 p = rows.at(j);
      const float r = fabsf(resid_f32<DIM>(p, lw.x, lw.y, lw.z));
      if (r <= ltlo) cnt += 1u;
      else if (!(r > lw.w)) cnt += 1u << 16;
      const int q = j >> 2;
      if (q >= q0) {
        const unsigned one = (q < e1 || (q >= e2 && q < e3)) ? 1u : 1u << 16;
        if (r <= lw.w)
          atomicAdd(&cs.lead_in[(q < e2 ? 0 : kIn) +
                                (DIM == 3 && p.z >= dir.z0 + 2.0f * dir.zq ? kTanBins + 1 : 0) +
                                tan_bin(dir, row_tan(p, line))],
                    one);
        else if (r > lw.w)  // NaN: held by no trial
          atomicAdd(&cs.lead_out[(q < e2 ? 0 : kExcessBins) + excess_bin(r - lw.w)], one);
      }
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) cs.red_c[warp] = (int)cnt;  // not red_i: a warp may still be reading the tops there
    __syncthreads();
    if (warp < 1 + NH) {  // warp 1: outside, the others: inside, a half of a2 each
      unsigned* h = warp == 1 ? cs.lead_out : cs.lead_in + (warp >> 1) * (kTanBins + 1);
      const int stride = warp == 1 ? kExcessBins : kIn;
      const int b = warp == 1 ? 2 * lane : lane;
      uint2 c0 = make_uint2(h[b], h[stride + b]), c1 = make_uint2(0u, 0u);
      if (warp == 1) c1 = make_uint2(h[b + 1], h[stride + b + 1]);
      uint2 incl = make_uint2(c0.x + c1.x, c0.y + c1.y);
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const unsigned tx = __shfl_up_sync(0xffffffffu, incl.x, d), ty = __shfl_up_sync(0xffffffffu, incl.y, d);
        if (lane >= d) {
          incl.x += tx;
          incl.y += ty;
        }
      }
      auto put = [&](int bin, unsigned x, unsigned y) {
        y += y >> 16;              // stages 2 and 3, 3
        x += (y & 0xFFFFu) << 16;  // 1 on
        x += x >> 16;              // 0 on
        h[bin] = x;
        h[stride + bin] = y;
      };
      if (warp == 1) {
        put(b, incl.x - c1.x, incl.y - c1.y);
        put(b + 1, incl.x, incl.y);
      } else {
        put(lane, incl.x - c0.x, incl.y - c0.y);
        if (lane == 31) put(kTanBins, incl.x, incl.y);
      }
    } else if (warp == 3) {
      const unsigned v = __reduce_add_sync(0xffffffffu, lane < kWarps ? (unsigned)cs.red_c[lane] : 0u);
      if (lane == 0) cs.lead_cnt = v;
    }
    __syncthreads();
  }
  if (lead >= 0) {
    const int certain = (int)(cs.lead_cnt & 0xFFFFu), near = (int)(cs.lead_cnt >> 16);
    const unsigned long long key = best_key(certain, hc0 + lead);
    if (tid == 0) {
      if (near == 0) {  // counted exactly: it leaves the pool
        S.U[lead] = -1;
        if (key > lim) {
          cs.best = key;
          cs.win = lw;
          cs.win_has_v64 = 0;
        }
        ++*n_cand;
      } else {
        S.U[lead] = certain + near;
      }
    }
    lim = max(lim, key);
  }
  const float lead_band = record_band(lw, a.tau32.hi, line);
  // the pruning test before stage s: the points from it on that trial h can hold
  auto keep = [&](int h, HoldRange r, int s) {
    const int sh = (s & 1) << 4;
    const unsigned* in = cs.lead_in + (s >> 1) * kIn;
    int n = (int)(cs.lead_out[(s >> 1) * kExcessBins + r.out()] >> sh & 0xFFFFu);
#pragma unroll
    for (int c = 0; c < NH; ++c)
      n += (int)(in[c * (kTanBins + 1) + r.hi(c)] >> sh & 0xFFFFu) -
           (int)(in[c * (kTanBins + 1) + r.lo(c)] >> sh & 0xFFFFu);
    const bool k = best_key(S.U[h] + n, hc0 + h) > lim;
    if (!k) S.U[h] = -1;
    return k;
  };
  int A = prune_list<false>(
      S, nh,
      [&](int h) {
        if (h == lead) return false;  // its count is already known
        const HoldRange r = hold_range<DIM>(dir, lw, lead_band, line, S.hyp[h]);
        S.tlo[h] = __uint_as_float(r.v);
        return keep(h, r, 0);
      },
      cs.red_i);
  for (int s = 1; A > 0 && q0 < nq; ++s) {
    const int q1 = s == 1 ? e1 : (s == 2 ? e2 : (s == 3 ? e3 : nq));
    const bool last = s == 4 || q1 + (q1 - q0) / 2 >= nq;  // no short last stage
    score(std::true_type{}, A, q0, last ? nq : q1);
    if (last) break;
    __syncthreads();
    q0 = q1;
    A = prune_list<true>(
        S, A, [&](int h) { return keep(h, HoldRange{__float_as_uint(S.tlo[h])}, s); }, cs.red_i);
  }
  return scored;
}

// a2 + a3 for trials hc0 .. hc0 + nh - 1 of cluster ci under the cosine
// model: draw, FP32 solve (refined when ill-conditioned), bound, records
// into S.  Trials with a wide band refine their velocity.  3D minimal sets
// are often ill-conditioned and refine on the spot above kRefineBand.  2D
// ones have |det| = |sin(t1 - t0)| and mostly narrow bands, whose few band
// points cost less than refining; those above tau / 32 are queued, and when
// they are at least an eighth of the chunk (a cluster of narrow azimuth
// extent, such as a far object, where nearly every seed pair is
// ill-conditioned) a second pass refines them, one per lane.  Elsewhere the
// pass's latency would cost more than the band points it saves; either way
// the decisions are exact.
template <int DIM, typename RV>
__device__ __forceinline__ void cosine_trial_chunk(const FrameDesc& a, const RV rows, const Rows64<DIM>& R,
                                                     const Smem& S, ClusterShared& cs, int ci, int N, int hc0,
                                                     int nh, float wmax, unsigned* fp64_count,
                                                     unsigned* refined_count) {
  const int tid = threadIdx.x;
  const float refine_band = DIM == 3 ? kRefineBand : a.tau32.hi * 0x1p-5f;
  unsigned n_fp64 = 0, n_ref = 0;
  for (int hl = tid; hl < nh; hl += kThreads) {
    int q[3];
    draw_minimal_set<DIM>(a.key, a.cluster_base + ci, hc0 + hl, N, q);
    const int q2 = DIM == 3 ? q[2] : q[0];
    const float4 p0 = rows.at(q[0]), p1 = rows.at(q[1]), p2 = rows.at(q2);
    const int qs[3] = {q[0], q[1], q2};
    auto seed64 = [&]() {
      if constexpr (DIM == 3) return LowSeeds{R.pre, {qs[0], qs[1], qs[2]}};
      else return [&](int i) { return R.at(qs[i]); };
    }();
    const float rb = DIM == 3 ? refine_band : __int_as_float(0x7f800000);
    Hyp32 hy = hyp_f32<DIM>(p0, p1, p2, seed64, rb, wmax, a.acc, a.rej, a.tau32);
    if (hy.kind == kHypUndecided) {
      ++n_fp64;
      double v[3];
      if (hyp_f64<DIM>(a, R, ci, hc0 + hl, N, v)) {
        hy = hyp_f32<DIM>(p0, p1, p2, seed64, rb, wmax, 0.0f, 0.0f, a.tau32);
        if (hy.kind != kHypNormal) {
          hy.kind = kHypExactOnly;
          hy.thi = __int_as_float(0x7f800000);
          hy.tlo = -1.0f;
        }
      } else {
        hy.kind = kHypRejected;
      }
    }
    if (hy.kind == kHypExactOnly) ++n_fp64;
    n_ref += hy.refined;
    S.hyp[hl] = make_float4(hy.nx, hy.ny, hy.nz, hy.kind == kHypRejected ? __int_as_float(0x7fc00000) : hy.thi);
    S.kind[hl] = (int8_t)hy.kind;
    if constexpr (DIM == 2) {
      // the queue lives in U until the second pass has read it
      if (hy.kind == kHypNormal && hy.thi - a.tau32.hi > refine_band) S.U[atomicAdd(&cs.nref, 1)] = hl;
    } else {
      S.U[hl] = hy.kind == kHypRejected ? -1 : (hy.kind == kHypExactOnly ? N : 0);
    }
  }
  if constexpr (DIM == 2) {
    __syncthreads();
    const int nr = 8 * cs.nref >= nh ? cs.nref : 0;
    for (int i = tid; i < nr; i += kThreads) {
      const int hl = S.U[i];
      int q[3];
      draw_minimal_set<DIM>(a.key, a.cluster_base + ci, hc0 + hl, N, q);
      const int qs[3] = {q[0], q[1], q[0]};
      // seed rows from the frame's arrays: keeping the loaded FP32 rows
      // alive across the solve instead measured slower on trials that refine
      auto seed64 = [&](int k) { return R.at(qs[k]); };
      // the trial was accepted in the first pass: no conditioning test
      Hyp32 hy = hyp_f32<DIM>(rows.at(q[0]), rows.at(q[1]), rows.at(q[0]), seed64, refine_band, wmax, 0.0f,
                              0.0f, a.tau32);
      if (hy.kind != kHypNormal) {
        hy.kind = kHypExactOnly;
        hy.thi = __int_as_float(0x7f800000);
        hy.tlo = -1.0f;
        ++n_fp64;
      }
      n_ref += hy.refined;
      S.hyp[hl] = make_float4(hy.nx, hy.ny, hy.nz, hy.thi);
        S.kind[hl] = (int8_t)hy.kind;
    }
    __syncthreads();
    for (int hl = tid; hl < nh; hl += kThreads) {
      const int k = S.kind[hl];
      S.U[hl] = k == kHypRejected ? -1 : (k == kHypExactOnly ? N : 0);
    }
    if (tid == 0) cs.nref = 0;
  }
  *fp64_count += n_fp64;
  *refined_count += n_ref;
}

template <int DIM, bool SMEM_ROWS, bool EXT>
__device__ void process_cluster(const FrameDesc& a, const Smem& S, ClusterShared& cs, int ci, int hchunk,
                                int pw, int prune, int frame, FinishRec* fq, int* fq_n,
                                double4_32a* cta_pre, int row_cap) {
  const int tid = threadIdx.x;
  const int64_t o = a.offsets[ci];
  const int64_t e = a.offsets[ci + 1];
  if (o < 0 || e < o || e > a.n_points || (e - o) > 0x7fffffff) {
    if (tid == 0) write_invalid<DIM>(a, ci, RVH_STATUS_BAD_OFFSETS);
    return;
  }
  const int N = (int)(e - o);
  if (N < DIM) {
    for (int j = tid; j < N; j += kThreads) a.mask[o + j] = 0;
    if (tid == 0) write_invalid<DIM>(a, ci, RVH_STATUS_TOO_FEW_POINTS);
    return;
  }
  using RV = typename std::conditional<SMEM_ROWS, TileRowsOf<DIM>, HybridRowsOf<DIM>>::type;
  RV rows;
  if constexpr (SMEM_ROWS) {
    rows.f = S.rows;
  } else {
    // the tail's tiles start at the cluster's own float4 [N] region, whose
    // cap unused entries leave room for rounding its end up
    constexpr int NC = DIM == 2 ? 3 : 4;
    rows.s.f = S.rows;
    rows.cap = row_cap;
    rows.g.f = reinterpret_cast<float*>(a.rows_g + o) - (size_t)row_cap * NC;
  }
  // FP64 rows: the CTA's own slot when the cluster fits it (the slot is
  // reused cluster after cluster and stays in L2), else the frame's
  // per-point scratch
  const Rows64<DIM> R = {&a, o, (SMEM_ROWS && cta_pre) ? cta_pre : a.rows64_g + o};
  long long t_stage = clock64();
  auto stage_done = [&](int k) {
    if (tid == 0) {
      const long long t = clock64();
      cs.clk[k] += (unsigned long long)(t - t_stage);
      t_stage = t;
    }
  };

  // a1: FP32 rows in shared memory (sincosf), FP64 rows in global scratch;
  // the line model of Alg. 1 normalises its points and computes its MAD
  // threshold instead
  float wm = 0.0f;
  auto cosine_rows = [&]() {
    for (int j = tid; j < N; j += kThreads) {
      const float w = a.dop[o + j];
      const float az = a.az[o + j];
      const float el = DIM == 3 ? a.el[o + j] : 0.0f;
      const float4 row = row_f32<DIM>(az, el, w);
      rows.put(j, row);
      if (DIM == 3) {
        double a64[3];
        row_f64<DIM>(a.trig, az, el, a64);
        R.pre[j] = make_double4_32a(
            a64[0], a64[1], a64[2],
            pack_low(low_part(a64[0], row.x), low_part(a64[1], row.y), low_part(a64[2], row.z)));
      }
      wm = fmaxf(wm, fabsf(w));
    }
  };
  if constexpr (EXT && DIM == 2) {
    if (a.line_model) {
      line_rows_and_threshold<RV>(a, rows, R.pre, o, N, S, hchunk, cs);
      if (tid == 0 && a.threshold) a.threshold[ci] = cs.ln_T;  // the API wrote NaN before
    } else {
      cosine_rows();
    }
  } else {
    cosine_rows();
  }
  // pad the last quad of the scoring pass: NaN Dopplers never count
  if (tid < ((N + 3) & ~3) - N) {
    const float nan = __int_as_float(0x7fc00000);
    rows.put(N + tid, make_float4(0.0f, 0.0f, nan, nan));
  }
  if (tid == 0) {
    cs.best = 0ull;
    cs.nref = 0;
  }
  const bool may_stage = prune && pw == 1 && N >= kStageMinPoints<DIM> && N <= kStageMaxPoints;
  const bool line = EXT && DIM == 2 && a.line_model;
  if (may_stage) direction_range<DIM>(rows, N, line, cs);
  const float wmax = block_max_float(wm, cs.red_f);  // its barrier also orders the row writes
  if (may_stage) direction_range_finish<DIM>(cs);
  unsigned n_fp64 = 0, n_ref = 0;
  unsigned long long n_cand = 0, n_scored = 0;
  stage_done(0);

  // trials run in chunks of hchunk, or in the adaptive blocks of trial_block
  const int chunk = (EXT && a.trial_block > 0) ? a.trial_block : hchunk;
  [[maybe_unused]] int trials_run = a.H;  // all of them, unless the adaptive count stops early
  for (int hc0 = 0; hc0 < a.H; hc0 += chunk) {
    const int nh = min(chunk, a.H - hc0);
    // a2 + a3: draw, FP32 solve (refined when ill-conditioned), bound
    auto cosine_trials = [&]() {
      cosine_trial_chunk<DIM, RV>(a, rows, R, S, cs, ci, N, hc0, nh, wmax, &n_fp64, &n_ref);
    };
    if constexpr (EXT && DIM == 2) {
      if (a.line_model) {
        const TauPair T = {__double2float_rd(cs.ln_T), __double2float_ru(cs.ln_T)};
        for (int hl = tid; hl < nh; hl += kThreads) {
          // Alg. 1: the line through the two normalised seed points
          int q[3];
          draw_minimal_set<2>(a.key, a.cluster_base + ci, hc0 + hl, N, q);
          Hyp32 hy = line_record_f32(rows.at(q[0]), rows.at(q[1]), T);
          if (hy.kind == kHypUndecided) {
            double v[3];
            if (line_seeds64(R.pre[q[0]], R.pre[q[1]], v)) {
              hy = line_record(v, cs.ln_T);
            } else {
              hy.kind = kHypRejected;
              hy.nx = hy.ny = hy.nz = 0.0f;
            }
          }
          if (hy.kind == kHypExactOnly) ++n_fp64;
          S.hyp[hl] = make_float4(hy.nx, hy.ny, hy.nz, hy.kind == kHypRejected ? __int_as_float(0x7fc00000) : hy.thi);
          S.kind[hl] = (int8_t)hy.kind;
          S.U[hl] = hy.kind == kHypRejected ? -1 : (hy.kind == kHypExactOnly ? N : 0);
        }
      } else {
        cosine_trials();
      }
    } else {
      cosine_trials();
    }
    __syncthreads();
    stage_done(1);

    // a5 + a6 (used by the staged pass and by the best-first counts below):
    // exact count of trial hc0 + c, which leaves the pool (U = -1) and
    // becomes the lead if its key beats it
    auto count_trial = [&](int c) {
      const float4 hy = S.hyp[c];
      const float htlo = record_tlo(hy, a.tau32, line);
      int B = 0;
      const int C = exact_count_block<DIM, RV, EXT>(a, rows, R, ci, hc0 + c, N, hy, htlo, cs, &B);
      ++n_cand;
      if (tid == 0) {
        S.U[c] = -1;
        const unsigned long long k = best_key(C, hc0 + c);
        if (k > cs.best) {
          cs.best = k;
          cs.win = hy;
          cs.win_has_v64 = B > 0;
          cs.win_v64[0] = cs.cv64[0];
          cs.win_v64[1] = cs.cv64[1];
          cs.win_v64[2] = cs.cv64[2];
        }
      }
      __syncthreads();
    };

    // a4: scoring pass (the hot loop)
    if (may_stage) {
      const unsigned long long scored = staged_pass<DIM, EXT>(a, rows, S, cs, hc0, nh, N, &n_cand);
      if ((tid & 31) == 0) n_scored += scored;
    } else {
      phase_a_dispatch<DIM>(pw, rows, N, S, nh);
      if (tid == 0) n_scored += (unsigned long long)nh * (unsigned long long)N;
    }
    __syncthreads();
    stage_done(2);

    // a5 + a6: exact counts of the trials whose upper bound can still win,
    // best first: the trial with the highest key (U, then lowest index) is
    // counted next, until no remaining key beats the lead.  C_h <= U_h, so a
    // trial whose key (U_h, h) does not beat the lead cannot win with its
    // exact count either, and the winner -- the highest exact count, the
    // lowest index among equals -- is the one counting every trial would
    // give.  Trials of earlier chunks have lower indices; the lead's key
    // already ranks them.  A counted trial leaves the pool (U = -1).
    for (;;) {
      int um = -1, hm = 0x7fffffff;
      for (int hl = tid; hl < nh; hl += kThreads) {
        const int u = S.U[hl];
        if (u > um) {
          um = u;
          hm = hc0 + hl;
        }
      }
      const unsigned long long km = block_best(um, hm, cs.red_u);
      if (km <= cs.best) break;  // also km == 0: no trial left
      count_trial((int)(0xFFFFFFFFu - (uint32_t)(km & 0xFFFFFFFFull)) - hc0);
    }
    __syncthreads();
    stage_done(3);
    if constexpr (EXT) {
      // adaptive trial count: stop once the bound says enough trials have run
      if (a.confidence > 0.0 && hc0 + nh < a.H) {
        if (tid == 0) cs.stop = adaptive_stop(cs.best, N, DIM, hc0 + nh, a.confidence);
        __syncthreads();
        if (cs.stop) {
          trials_run = hc0 + nh;
          break;
        }
      }
    }
  }

  if (tid == 0) cs.ctr[0] += n_cand;
  {
    // Counters of this warp, without atomics: a 64-bit shared-memory atomic is
    // a compare-and-swap loop, and in 3D, where every thread refines trials,
    // 256 of them on one word took longer than the mask pass of a small
    // cluster: dense3d 1.205 -> 1.083 ms; dense2d, with fewer spills, 0.2203 ->
    // 0.2177.
    const unsigned fp64s = __reduce_add_sync(0xffffffffu, n_fp64), refs = __reduce_add_sync(0xffffffffu, n_ref);
    if ((tid & 31) == 0) {
      cs.wctr[0][tid >> 5] += fp64s;
      cs.wctr[1][tid >> 5] += refs;
      cs.wctr[2][tid >> 5] += n_scored;  // counted by lane 0
    }
  }
  if constexpr (EXT) {
    if (tid == 0) {
      cs.runs[0] += (unsigned long long)trials_run;
      cs.runs[1] += (unsigned long long)trials_run * (unsigned long long)N;
    }
  }

  const unsigned long long key = cs.best;
  if (key == 0ull) {
    for (int j = tid; j < N; j += kThreads) a.mask[o + j] = 0;
    if (tid == 0) write_invalid<DIM>(a, ci, RVH_STATUS_ALL_DEGENERATE);
    __syncthreads();
    return;
  }
  const int hstar = (int)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFull));

  // a7 + a8: the winner's mask (FP32 certainties; FP64 for its band points,
  // whose FP64 velocity was computed when it was counted) and the normal
  // equations over its inliers.
  const float4 win = cs.win;
  const float wtlo = record_tlo(win, a.tau32, line);
  const double v64[3] = {cs.win_v64[0], cs.win_v64[1], cs.win_v64[2]};
  constexpr int NS = DIM == 2 ? 5 : 9;
  int n_in = mask_and_sums<DIM, RV, EXT>(a, rows, R, o, N, win, wtlo, v64, S, cs, false, nullptr);

  if constexpr (EXT) {
    if (a.lo_iters > 0) n_in = local_opt_rounds<DIM, RV>(a, rows, R, o, N, win, wtlo, v64, wmax, n_in, S, cs);
  }
  if (tid == 0) {
    FinishRec& q = fq[*fq_n];
#pragma unroll
    for (int i = 0; i < NS; ++i) q.t[i] = cs.red_t[i];
    q.v64[0] = v64[0];
    q.v64[1] = v64[1];
    q.v64[2] = v64[2];
    q.o = o;
    q.n_in = n_in;
    q.hstar = hstar;
    q.ci = ci;
    q.frame = frame;
    q.N = N;
    q.has_v64 = cs.win_has_v64;
    *fq_n += 1;
  }
  __syncthreads();
  stage_done(4);
}

// Clusters beyond the shared-memory rows under an extension.  Out of line:
// beside the inlined copy for the others, the 2D kernel's path for those
// spilled 416 bytes (96 so).  Dense 2D frame, us per pass: adaptive count 157
// -> 152, local optimisation 358 -> 350, line model 352 -> 334.
template <int DIM, bool EXT>
__device__ __noinline__ void process_large(const FrameDesc& a, const Smem& S, ClusterShared& cs, int ci, int hchunk,
                                           int pw, int prune, int frame, FinishRec* fq, int* fq_n, int row_cap) {
  process_cluster<DIM, false, EXT>(a, S, cs, ci, hchunk, pw, prune, frame, fq, fq_n, nullptr, row_cap);
}

// EXT = true: the instantiation with the extensions of the method (the
// local-optimisation rounds and the adaptive trial count), launched only for
// batches that ask for one of them; the default instantiation carries no
// trace of them.
template <int DIM, bool EXT>
__global__ void __launch_bounds__(kThreads, RVH_MIN_BLOCKS) fused_kernel(const __grid_constant__ FusedArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ ClusterShared cs;
  __shared__ int s_item;
  __shared__ FinishRec fq[kFinishBatch];
  __shared__ int fq_n;
  Smem S;
  unsigned char* p = smem_raw;
  S.rows = reinterpret_cast<float*>(p);
  p += (size_t)((a.nmax_smem + 31) & ~31) * sizeof(float4);
  S.hyp = reinterpret_cast<float4*>(p);
  p += (size_t)a.hchunk * sizeof(float4);
  S.tlo = reinterpret_cast<float*>(p);
  p += (size_t)a.hchunk * sizeof(float);
  S.U = reinterpret_cast<int*>(p);
  p += (size_t)a.hchunk * sizeof(int);
  S.kind = reinterpret_cast<int8_t*>(p);
  p += ((size_t)a.hchunk * sizeof(int8_t) + 15) & ~(size_t)15;
  S.list = reinterpret_cast<uint16_t*>(p);

  if (blockIdx.x == 0 && a.stats_next && threadIdx.x < kStatsWords) a.stats_next[threadIdx.x] = 0ull;
  if (threadIdx.x < 2) cs.ctr[threadIdx.x] = 0ull;
  if (threadIdx.x < 3 * kWarps) (&cs.wctr[0][0])[threadIdx.x] = 0ull;
  if constexpr (EXT) {
    if (threadIdx.x < 2) cs.runs[threadIdx.x] = 0ull;
  }
  if (threadIdx.x < 6) cs.clk[threadIdx.x] = 0ull;
  if (threadIdx.x == 0) fq_n = 0;
  // the queued clusters' solves (warp 0) and headings (warp 1), one lane each
  auto flush = [&]() {
    const int n = fq_n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < 2 && lane < n) {
      const FinishRec& q = fq[lane];
      const FrameDesc& F = a.f[q.frame];
      if (warp == 0) {
        // the CTA's row slot has moved on to later clusters: rows are
        // recomputed for the (rare) fallback solve
        const Rows64Inputs<DIM> R = {&F, q.o};
        finish_cluster<DIM, EXT>(F, R, q.ci, q.N, q.hstar, q.n_in, q.t, q.v64, q.has_v64 != 0);
      } else {
        finish_heading<DIM>(F, q.ci, q.n_in, q.t);
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) fq_n = 0;
    __syncthreads();
  };
  const long long t_kernel = clock64();
  for (int round = 0;; ++round) {
    __syncthreads();
    // The first a.wave CTAs, one per SM, start with the most expensive items;
    // all else is taken from the list in order as CTAs come free.  Taken in
    // order from the start, the most expensive items went to the CTAs that
    // came first, four to an SM, and a frame of little more than one cluster
    // per CTA waited for those few SMs: 1025 clusters of 8..2048 points, 2D at
    // 256 trials 0.091 -> 0.066 ms, 3D at 2048 trials 0.38 -> 0.263 ms; frames
    // of many items per CTA are unchanged within 3%.
    if (threadIdx.x == 0) {
      int item = a.n_items;
      if (round == 0 && (int)blockIdx.x < a.wave) item = (int)blockIdx.x;
      else if (!a.direct) item = a.wave + atomicAdd(a.work_counter, 1);
      s_item = item;
    }
    __syncthreads();
    const int item = s_item;
    if (item >= a.n_items) break;
    int2 fc;
    if (a.direct) {
      // as many CTAs as items: frame-major order needs no work list
      int f = 0, rem = item;
      while (rem >= a.f[f].n_clusters) rem -= a.f[f++].n_clusters;
      fc = make_int2(f, rem);
    } else {
      fc = a.worklist[item];
    }
    const FrameDesc& F = a.f[fc.x];
    const int ci = fc.y;
    const int64_t o = F.offsets[ci], e = F.offsets[ci + 1];
    double4_32a* cta_pre =
        a.cta_rows64 ? a.cta_rows64 + (size_t)blockIdx.x * cta_slot_stride(DIM, a.nmax_smem) : nullptr;
    const int cap = smem_row_capacity(DIM, a.nmax_smem);
    if (e - o <= (int64_t)cap || e < o) {
      process_cluster<DIM, true, EXT>(F, S, cs, ci, a.hchunk, a.pw, a.prune, fc.x, fq, &fq_n, cta_pre, cap);
    } else if constexpr (EXT) {
      process_large<DIM, EXT>(F, S, cs, ci, a.hchunk, a.pw, a.prune, fc.x, fq, &fq_n, cap & ~31);
    } else {
      process_cluster<DIM, false, EXT>(F, S, cs, ci, a.hchunk, a.pw, a.prune, fc.x, fq, &fq_n, cta_pre, cap & ~31);
    }
    __syncthreads();
    if (fq_n == kFinishBatch) flush();
  }
  __syncthreads();
  flush();
  if (threadIdx.x == 0) {
    unsigned long long staged = 0;
    for (int k = 0; k < 5; ++k) staged += cs.clk[k];
    const unsigned long long total = (unsigned long long)(clock64() - t_kernel);
    cs.clk[5] = total > staged ? total - staged : 0ull;
  }
  __syncthreads();
  if (threadIdx.x < 5 && a.stats) {
    // exact counts, band points, fp64 trials, refined trials; pairs scored
    unsigned long long v = 0;
    if (threadIdx.x < 2) {
      v = cs.ctr[threadIdx.x];
    } else {
      for (int w = 0; w < kWarps; ++w) v += cs.wctr[threadIdx.x - 2][w];
    }
    if (v) atomicAdd(&a.stats[threadIdx.x < 4 ? threadIdx.x : 12], v);
  }
  if (threadIdx.x < 6 && a.stats) atomicAdd(&a.stats[4 + threadIdx.x], cs.clk[threadIdx.x]);
  if constexpr (EXT) {
    if (threadIdx.x < 2 && a.stats) atomicAdd(&a.stats[10 + threadIdx.x], cs.runs[threadIdx.x]);
  }
}

// Orders the batch's (frame, cluster) items by decreasing cost N * H (H: the
// trial_block of adaptive frames, which mostly stop after one block),
// longest-processing-time first, in buckets of an eighth of an octave (the
// floor of log2 of the cost and its next three bits), and resets the work
// counter.  One CTA.
constexpr int kCostBuckets = 512;
__device__ __forceinline__ int item_bucket(const FrameDesc& F, int ci) {
  const int64_t n = (int64_t)F.offsets[ci + 1] - F.offsets[ci];
  const int64_t cost = n > 0 ? n * (int64_t)(F.trial_block > 0 ? min(F.trial_block, F.H) : F.H) : 1;
  const int lg = 63 - __clzll(cost);
  const int sub = (int)((lg >= 3 ? cost >> (lg - 3) : cost << (3 - lg)) & 7);
  return kCostBuckets - 1 - min((lg << 3) | sub, kCostBuckets - 1);  // 0 = most expensive
}

// Items are numbered frame-major; each thread keeps the buckets of its first
// kItemsKept items in registers between the two passes.
constexpr int kItemsKept = 8;
__global__ void worklist_kernel(const __grid_constant__ FusedArgs a) {
  __shared__ int hist[kCostBuckets];
  for (int b = threadIdx.x; b < kCostBuckets; b += blockDim.x) hist[b] = 0;
  __syncthreads();
  int kept[kItemsKept];
  {
    int f = 0, base = 0, k = 0;
    for (int it = threadIdx.x; it < a.n_items; it += blockDim.x, ++k) {
      while (it - base >= a.f[f].n_clusters) base += a.f[f++].n_clusters;
      const int b = item_bucket(a.f[f], it - base);
      if (k < kItemsKept) kept[k] = b;
      atomicAdd(&hist[b], 1);
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {  // exclusive scan of the histogram, 16 buckets per lane
    constexpr int kPer = kCostBuckets / 32;
    const int lane = threadIdx.x;
    int c[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      c[k] = hist[lane * kPer + k];
      sum += c[k];
    }
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += t;
    }
    int run = incl - sum;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      hist[lane * kPer + k] = run;
      run += c[k];
    }
    if (lane == 0) *a.work_counter = 0;
  }
  __syncthreads();
  {
    int f = 0, base = 0, k = 0;
    for (int it = threadIdx.x; it < a.n_items; it += blockDim.x, ++k) {
      while (it - base >= a.f[f].n_clusters) base += a.f[f++].n_clusters;
      const int b = k < kItemsKept ? kept[k] : item_bucket(a.f[f], it - base);
      a.worklist[atomicAdd(&hist[b], 1)] = make_int2(f, it - base);
    }
  }
}

size_t fused_smem_bytes(int nmax_smem, int hchunk) {
  return (size_t)((nmax_smem + 31) & ~31) * sizeof(float4) + trial_area_bytes(hchunk);
}

cudaError_t launch_worklist(const FusedArgs& a, cudaStream_t s) {
  worklist_kernel<<<1, kWorklistThreads, 0, s>>>(a);
  return cudaGetLastError();
}

bool fused_ext(const FusedArgs& a) {
  bool ext = false;
  for (int f = 0; f < a.n_frames; ++f)
    ext = ext || a.f[f].lo_iters > 0 || a.f[f].confidence > 0.0 || a.f[f].line_model != 0;
  return ext;
}

const void* fused_kernel_fn(int dim, bool ext) {
  if (dim == 2) return ext ? (const void*)fused_kernel<2, true> : (const void*)fused_kernel<2, false>;
  return ext ? (const void*)fused_kernel<3, true> : (const void*)fused_kernel<3, false>;
}

const void* worklist_kernel_fn() { return (const void*)worklist_kernel; }

int fused_threads() { return kThreads; }

cudaError_t fused_configure_max(int dim, int device) {
  int optin = 0;
  cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  for (int ext = 0; ext < 2 && e == cudaSuccess; ++ext) {
    const void* fn = fused_kernel_fn(dim, ext != 0);
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, fn);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
  }
  return e;
}

cudaError_t fused_occupancy(int dim, size_t smem, int* blocks_per_sm) {
  if (dim == 2)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fused_kernel<2, false>, kThreads, smem);
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fused_kernel<3, false>, kThreads, smem);
}

cudaError_t launch_fused(int dim, const FusedArgs& a, int grid, size_t smem, cudaStream_t s) {
  const bool ext = fused_ext(a);
  if (dim == 2) {
    if (ext) fused_kernel<2, true><<<grid, kThreads, smem, s>>>(a);
    else fused_kernel<2, false><<<grid, kThreads, smem, s>>>(a);
  } else {
    if (ext) fused_kernel<3, true><<<grid, kThreads, smem, s>>>(a);
    else fused_kernel<3, false><<<grid, kThreads, smem, s>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace rvh
