// Robust noise measurement and clipping (SoFiA 2, Sect. 4.1 and 4.2).
//
// sigma = 1.4826 * median(|S - median(S)|) over the finite voxels, with both
// medians exact order statistics of the float32 values (mean of the two
// middle ones for an even count), then mask |= |S| > t * sigma.
//
// Data flow for one measurement over an array S of n values:
//   k_hist      (or the smoothing kernel's epilogue): histogram of S over
//               bins of the float bits (monotone in the value).
//   k_plan      a cluster of eight blocks: ranks of the middle order
//               statistics -> the bins holding the median; from the bin counts
//               alone, thresholds T1 < MAD < T2 and the value windows that can
//               hold the MAD's elements; bounds on t*sigma for the clip;
//               capacity checks; the candidate pass's class table. It clears
//               the histogram for the next measurement of the run.
//   k_pass2     one read of S: collects median candidates (values in the
//               median bins), MAD candidates (values not surely inside or
//               outside the MAD band), counts values surely inside the band,
//               sets the mask bits that are certain whatever sigma is inside
//               its bounds, and lists the few voxels whose clip is not yet
//               decided.
//   k_select    (sc_select.cu) exact selection of the wanted order statistics
//               inside the candidate lists, then of |s - m|.
//   k_clip_full decides the listed voxels with the exact sigma.
// When a candidate set would exceed its buffer, the plan switches that part
// to full passes over S (k_sel_*: radix selection of 11 + 11 + 10 bits on the
// whole array; k_clip_full); results are identical, only slower.
#include <cooperative_groups.h>

#include <atomic>
#include <cfloat>
#include <cstdio>

#include "sc_device.cuh"
#include "sc_internal.h"

namespace sc {

// ---------------------------------------------------------------------------
// Histogram (and max |x|) of the finite values of an array.
__global__ void __launch_bounds__(512) k_hist(const float* __restrict__ x, long long n, DevState* st,
                                              unsigned long long* __restrict__ hist, int win, int want_maxabs) {
  extern __shared__ unsigned int sh[];
  for (int i = threadIdx.x; i < kNumBins; i += blockDim.x) sh[i] = 0u;
  __syncthreads();
  const BinCfg cfg = win ? st->win : kFullRange;
  unsigned int mx = 0u;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const bool vec = ((reinterpret_cast<uintptr_t>(x) & 15u) == 0);
  if (vec) {
    const long long n4 = n >> 2;
    const float4* x4 = reinterpret_cast<const float4*>(x);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
      float4 v = __ldg(x4 + i);
      float a[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (isfinite(a[c])) {
          atomicAdd(&sh[bin_of(a[c], cfg)], 1u);
          mx = max(mx, __float_as_uint(fabsf(a[c])));
        }
      }
    }
    for (long long i = (n4 << 2) + (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
      float a = __ldg(x + i);
      if (isfinite(a)) {
        atomicAdd(&sh[bin_of(a, cfg)], 1u);
        mx = max(mx, __float_as_uint(fabsf(a)));
      }
    }
  } else {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
      float a = __ldg(x + i);
      if (isfinite(a)) {
        atomicAdd(&sh[bin_of(a, cfg)], 1u);
        mx = max(mx, __float_as_uint(fabsf(a)));
      }
    }
  }
  if (want_maxabs) {
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0 && mx) atomicMax(&st->maxabs_bits, mx);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kNumBins; i += blockDim.x)
    if (sh[i]) atomicAdd(hist + i, (unsigned long long)sh[i]);
}

cudaError_t launch_hist(const float* x, long long n, DevState* st, unsigned long long* hist, int win,
                        int want_maxabs, int sms, cudaStream_t s) {
  const size_t smem = kNumBins * sizeof(unsigned int);
  long long want = (n / 4 + 511) / 512;
  int grid = (int)(want < 1 ? 1 : (want > 4LL * sms ? 4LL * sms : want));
  k_hist<<<grid, 512, smem, s>>>(x, n, st, hist, win, want_maxabs);
  return cudaGetLastError();
}

// The same histogram (and max |value|) of a 16-bit cube, whose planes hold a
// multiple of 8 values: a thread takes 8 values (16 bytes) at a time and
// decodes them with their plane's scale (the plane followed along the
// grid-stride loop). With out != null the decoded float32 values are written
// there as well (the cube for the passes that read it as float32).
__global__ void __launch_bounds__(512) k_hist16(Half16 h, long long plane, long long n, DevState* st,
                                                unsigned long long* __restrict__ hist, int win, int want_maxabs,
                                                float* __restrict__ out) {
  extern __shared__ unsigned int sh[];
  for (int i = threadIdx.x; i < kNumBins; i += blockDim.x) sh[i] = 0u;
  __syncthreads();
  const BinCfg cfg = win ? st->win : kFullRange;
  unsigned int mx = 0u;
  const long long ng = n / 8, pg = plane / 8;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long dz = stride / pg, doff = stride - dz * pg;
  long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  long long z = g / pg, off = g - z * pg;
  const uint4* b4 = reinterpret_cast<const uint4*>(h.bits);
  for (; g < ng; g += stride) {
    const uint4 q = __ldg(b4 + g);
    const float cs = __ldg(h.scale + z);
    const unsigned w[4] = {q.x, q.y, q.z, q.w};
    float v[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[2 * k] = half16_value((unsigned short)(w[k] & 0xffffu), h.fmt, cs);
      v[2 * k + 1] = half16_value((unsigned short)(w[k] >> 16), h.fmt, cs);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (isfinite(v[i])) {
        atomicAdd(&sh[bin_of(v[i], cfg)], 1u);
        mx = max(mx, __float_as_uint(fabsf(v[i])));
      }
    }
    if (out) {
      float4* o4 = reinterpret_cast<float4*>(out) + 2 * g;
      o4[0] = make_float4(v[0], v[1], v[2], v[3]);
      o4[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
    z += dz;
    off += doff;
    if (off >= pg) {
      off -= pg;
      ++z;
    }
  }
  if (want_maxabs) {
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0 && mx) atomicMax(&st->maxabs_bits, mx);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kNumBins; i += blockDim.x)
    if (sh[i]) atomicAdd(hist + i, (unsigned long long)sh[i]);
}

cudaError_t launch_hist16(const Half16& h, long long plane, long long n, DevState* st, unsigned long long* hist,
                          int win, int want_maxabs, float* out, int sms, cudaStream_t s) {
  if (plane % 8 != 0 || (reinterpret_cast<uintptr_t>(h.bits) & 15u) != 0 ||
      (out && (reinterpret_cast<uintptr_t>(out) & 15u) != 0))
    return cudaErrorInvalidValue;  // the caller takes the 16-bit path only for such cubes
  const size_t smem = kNumBins * sizeof(unsigned int);
  long long want = (n / 8 + 511) / 512;
  int grid = (int)(want < 1 ? 1 : (want > 4LL * sms ? 4LL * sms : want));
  k_hist16<<<grid, 512, smem, s>>>(h, plane, n, st, hist, win, want_maxabs, out);
  return cudaGetLastError();
}

// Max |x| over finite values only (for sc_smooth's fixed-point scale).
__global__ void k_maxabs(const float* __restrict__ x, long long n, DevState* st) {
  unsigned int mx = 0u;
  const auto take = [&](float a) {
    if (isfinite(a)) mx = max(mx, __float_as_uint(fabsf(a)));
  };
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
  // (HBM-bound: 512 x 512 x 256 values took 49 us with 4-byte loads, 43 with
  // 16-byte ones, four in flight)
  const long long nq = (reinterpret_cast<uintptr_t>(x) & 15u) == 0u ? n / 4 : 0;
  long long q = t;
  for (; q + 3 * nt < nq; q += 4 * nt) {
    float4 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __ldg(reinterpret_cast<const float4*>(x) + q + k * nt);
#pragma unroll
    for (int k = 0; k < 4; ++k) take(v[k].x), take(v[k].y), take(v[k].z), take(v[k].w);
  }
  for (; q < nq; q += nt) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(x) + q);
    take(v.x), take(v.y), take(v.z), take(v.w);
  }
  for (long long i = 4 * nq + t; i < n; i += nt) take(__ldg(x + i));
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(&st->maxabs_bits, mx);
}

cudaError_t launch_maxabs(const float* x, long long n, DevState* st, int sms, cudaStream_t s) {
  long long want = (n + 255) / 256;
  int grid = (int)(want < 1 ? 1 : (want > 8LL * sms ? 8LL * sms : want));
  k_maxabs<<<grid, 256, 0, s>>>(x, n, st);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Plan: what its searches read of the scanned histogram.
struct PlanCtx {
  const unsigned long long* cum;  // exclusive prefix counts, kNumBins + 1 entries
  BinCfg cfg;
  double m_min, m_max;
};

__device__ __forceinline__ unsigned long long cum_range(const PlanCtx& P, int b1, int b2) {
  // count of values in bins b1..b2 inclusive (0 if empty range)
  if (b2 < b1) return 0ull;
  return P.cum[b2 + 1] - P.cum[b1];
}
__device__ __forceinline__ float f_down(double v) { return nextafterf(__double2float_rd(v), -INFINITY); }
__device__ __forceinline__ float f_up(double v) { return nextafterf(__double2float_ru(v), INFINITY); }

// Number of values that can possibly lie within T of some m in [m_min, m_max],
// or (sure) that surely lie within T of every one (whole bins strictly inside
// [m_max - T, m_min + T]).
__device__ __noinline__ unsigned long long within(const PlanCtx& P, float T, bool sure) {
  // one float up for a sure count's lower end and a possible count's upper
  // end, one down for the others
  const double x = P.m_max + (sure ? -(double)T : (double)T), y = P.m_min + (sure ? (double)T : -(double)T);
  const float up = f_up(x), down = f_down(y);
  const float lo = sure ? up : down, hi = sure ? down : up;
  if (sure && !(lo <= hi)) return 0ull;
  const int e = sure ? 1 : 0;
  return cum_range(P, bin_of(lo, P.cfg) + e, bin_of(hi, P.cfg) - e);
}

// Class of a 16-bit cell of the float encoding (sign, 8 exponent bits, top
// 7 mantissa bits). Every histogram bin is a union of whole cells (bins
// resolve at most 7 mantissa bits), so the median and MAD classes are exact
// functions of the cell. CLS_SURE marks cells wholly above thr_hi in |s| (all
// their values are detected whatever sigma is); CLS_AMB marks cells that
// overlap (thr_lo, thr_hi] and is refined per value by the candidate pass.
constexpr int kClsCells = (int)kClassTableBytes;
enum : unsigned int { CLS_MED = 1u, CLS_MAD = 2u, CLS_AMB = 4u, CLS_SURE = 8u };

__device__ __forceinline__ unsigned int cell_class(unsigned int cell, const NoisePlan& p, BinCfg cfg, bool med,
                                                   bool mad, bool amb) {
  const unsigned int u = cell << 16;
  if (((u >> 23) & 0xffu) == 0xffu) return 0u;  // Inf and NaN are never candidates
  const int b = bin_of_bits(u, cfg);
  unsigned int k = 0u;
  if (med && b >= p.b_med_lo && b <= p.b_med_hi) k |= CLS_MED;
  if (mad && b >= p.bA_lo && b <= p.bA_hi && !(b >= p.bB_lo && b <= p.bB_hi)) k |= CLS_MAD;
  if (amb) {
    const float lo = fabsf(__uint_as_float(u)), hi = fabsf(__uint_as_float(u | 0xffffu));
    if (hi > p.thr_lo && lo <= p.thr_hi) k |= CLS_AMB;
    if (lo > p.thr_hi) k |= CLS_SURE;
  }
  return k;
}

// Thread t of nt writes its share of the 64 KiB class table (one byte per cell).
__device__ void fill_class_table(const NoisePlan& p, BinCfg cfg, unsigned char* cls, int t, int nt) {
  if (p.flags & (PLAN_EMPTY | PLAN_STD)) return;  // the candidate pass returns before it reads the table
  const bool med = !(p.flags & PLAN_MED_FULL);
  const bool mad = !(p.flags & PLAN_MAD_FULL);
  const bool amb = (p.flags & PLAN_CLIP) && !(p.flags & PLAN_CLIP_FULL);
  // (four cells a step: every launch fetches this code once, and unrolled
  // further it costs more to fetch than to run)
#pragma unroll 1
  for (int i = t; i < kClsCells / 4; i += nt) {
    unsigned int x = 0u;
#pragma unroll
    for (int b = 0; b < 4; ++b) x |= cell_class((unsigned)(i * 4 + b), p, cfg, med, mad, amb) << (8 * b);
    reinterpret_cast<unsigned int*>(cls)[i] = x;
  }
}

// The plan proper (one thread): the median bins and the float bits of the
// MAD's bracket (0xffffffff: no such bound) are given. Returns the plan it
// stored in st->plan.
__device__ __noinline__ NoisePlan plan_of(DevState* st, const unsigned long long* cum, BinCfg cfg, int b_med_lo,
                                          int b_med_hi, unsigned int T1_bits, unsigned int T2_bits, const float* src,
                                          long long n_total, Lists L, float threshold, int clip, int std_mode,
                                          unsigned int force_flags) {
  NoisePlan p;
  p.cfg = cfg;
  p.flags = (int)force_flags;
  p.threshold = threshold;
  p.has_B = 0;
  p.B_lo = 1.0f;
  p.B_hi = 0.0f;
  p.A_lo = -INFINITY;
  p.A_hi = INFINITY;
  p.thr_lo = 0.0f;
  p.thr_hi = INFINITY;
  p.T1 = 0.0f;
  p.T2 = INFINITY;
  p.bound_med = p.bound_mad = p.bound_amb = 0ull;
  p.bA_lo = 0;
  p.bA_hi = kNumBins - 1;
  p.bB_lo = 1;
  p.bB_hi = 0;
  p.n_B = 0ull;
  const unsigned long long n = cum[kNumBins];
  p.n = n;
  st->n_cand_med = st->n_cand_mad = st->n_amb = st->n_below = 0ull;
  st->sum = st->sum2 = 0.0;
  st->std_blocks = 0u;
  st->std_again = 0;
  st->count = 0ull;
  if (clip) p.flags |= PLAN_CLIP;
  if (std_mode) p.flags |= PLAN_STD | PLAN_CLIP_FULL;
  SelJob* J[2] = {&st->sel_med, &st->sel_mad};
  for (int w = 0; w < 2; ++w) {
    J[w]->c_le = 0ull;
    J[w]->min_gt = 0xffffffffu;
    J[w]->key_lo = 0u;
    J[w]->done = 0u;
    J[w]->count_fixed = 0ull;
    J[w]->count_ptr = nullptr;
    J[w]->list = src;
    J[w]->rank_lo = J[w]->rank_hi = 0ull;
  }
  if (n == 0ull) {
    p.flags |= PLAN_EMPTY;
    st->status |= SC_ST_ALLNAN;
    st->plan = p;
    return p;
  }
  p.k_lo = (n - 1ull) / 2ull;
  p.k_hi = n / 2ull;
  p.b_med_lo = b_med_lo;
  p.b_med_hi = b_med_hi;
  p.below_med = cum[p.b_med_lo];
  p.bound_med = cum[p.b_med_hi + 1] - cum[p.b_med_lo];
  if (p.bound_med > L.cap.med) p.flags |= PLAN_MED_FULL;

  if (std_mode) {
    // K and 2^e: the lowest and the highest bin with values bound them all
    int first = 0, last = kNumBins - 1;
    for (int hi = last; first < hi;) {
      const int mid = (first + hi) >> 1;
      if (cum[mid + 1] > 0ull) hi = mid; else first = mid + 1;
    }
    for (int lo = 0; lo < last;) {
      const int mid = (lo + last + 1) >> 1;
      if (cum[mid] < n) lo = mid; else last = mid - 1;
    }
    double top = fmax(fabs(bin_lo_value(first, cfg)), fabs(bin_hi_value(last, cfg)));
    if (!isfinite(top)) top = 2.0 * (double)fmaxf(__uint_as_float(st->maxabs_bits), st->repl);  // (0: not measured)
    // no scale for magnitudes up to 2^40 (and some above 2^-20): n squares stay
    // below 2^128, and what underflows (2^-150 a value) is 2^-77 of their sum
    int e = 128;
    if (top > 0.0 && isfinite(top)) frexp(top, &e);  // top < 2^e
    e = e > -20 && e <= 40 ? 0 : (e > 128 ? 128 : (e < -126 ? -126 : e));
    st->std_scale = ldexpf(1.0f, -e);
    // no shift where 0 lies well within the spread (a quarter of the values
    // beyond 8 times the median's magnitude, on either side of it)
    const double lo = bin_lo_value(p.b_med_lo, cfg), hi = bin_hi_value(p.b_med_lo, cfg);
    const double m = isfinite(lo) ? (isfinite(hi) ? 0.5 * (lo + hi) : lo) : (isfinite(hi) ? hi : 0.0);
    const float far = __double2float_ru(8.0 * fmax(fabs(lo), fabs(hi)));
    const bool near0 = isfinite(far) && 4ull * cum[bin_of(-far, cfg)] >= n &&
                       4ull * (n - cum[bin_of(far, cfg) + 1]) >= n;
    st->std_shift = near0 ? 0.0f : __double2float_rn(m);
  }
  if (!std_mode) {
    const PlanCtx P{cum, cfg, bin_lo_value(p.b_med_lo, cfg), bin_hi_value(p.b_med_hi, cfg)};
    if (!(isfinite(P.m_min) && isfinite(P.m_max))) {
      p.flags |= PLAN_MAD_FULL | PLAN_CLIP_FULL;
    } else {
      if (T1_bits != 0xffffffffu) {
        p.T1 = __uint_as_float(T1_bits);
        p.has_B = 1;
        p.B_lo = f_up(P.m_max - (double)p.T1);
        p.B_hi = f_down(P.m_min + (double)p.T1);
        // B as whole bins strictly inside [B_lo, B_hi]: its count is exact
        // from the histogram, so the candidate pass need not count it.
        if (p.B_lo <= p.B_hi) {
          p.bB_lo = bin_of(p.B_lo, cfg) + 1;
          p.bB_hi = bin_of(p.B_hi, cfg) - 1;
        }
      }
      if (T2_bits != 0xffffffffu) {
        p.T2 = __uint_as_float(T2_bits);
        p.A_lo = f_down(P.m_min - (double)p.T2);
        p.A_hi = f_up(P.m_max + (double)p.T2);
      }
      // bound on the MAD candidates: values neither surely inside nor outside
      p.bA_lo = bin_of(p.A_lo, cfg);
      p.bA_hi = bin_of(p.A_hi, cfg);
      p.n_B = cum_range(P, p.bB_lo, p.bB_hi);  // B lies inside A: its values are within T1 < T2
      p.bound_mad = cum_range(P, p.bA_lo, p.bA_hi) - p.n_B;
      if (p.bound_mad > L.cap.mad) p.flags |= PLAN_MAD_FULL;
      if (clip) {
        if (!p.has_B || !(p.T1 > 0.0f) || !isfinite(p.T2)) {
          p.flags |= PLAN_CLIP_FULL;
        } else {
          const float s_lo = sigma_of_mad((double)p.T1), s_hi = sigma_of_mad((double)p.T2);
          p.thr_lo = __fmul_rn(threshold, s_lo);
          p.thr_hi = __fmul_rn(threshold, s_hi);
          p.bound_amb = cum_range(P, bin_of(-p.thr_hi, cfg), bin_of(-p.thr_lo, cfg)) +
                        cum_range(P, bin_of(p.thr_lo, cfg), bin_of(p.thr_hi, cfg));
          if (p.bound_amb > L.cap.amb) p.flags |= PLAN_CLIP_FULL;
        }
      }
    }
  }
  // selection jobs
  const bool med_full = (p.flags & PLAN_MED_FULL) != 0, mad_full = (p.flags & PLAN_MAD_FULL) != 0;
  st->sel_med.list = med_full ? src : L.med;
  st->sel_med.count_fixed = med_full ? (unsigned long long)n_total : L.cap.med;
  st->sel_med.count_ptr = med_full ? nullptr : &st->n_cand_med;
  st->sel_med.mode = SEL_VALUE;
  st->sel_med.rank_lo = med_full ? p.k_lo : p.k_lo - p.below_med;
  st->sel_med.rank_hi = st->sel_med.rank_lo + (p.k_hi - p.k_lo);
  st->sel_mad.list = mad_full ? src : L.mad;
  st->sel_mad.count_fixed = mad_full ? (unsigned long long)n_total : L.cap.mad;
  st->sel_mad.count_ptr = mad_full ? nullptr : &st->n_cand_mad;
  st->sel_mad.mode = SEL_ABSDEV;
  st->sel_mad.rank_lo = p.k_lo;  // minus n_below unless full
  st->sel_mad.rank_hi = p.k_hi;
  st->n_below = mad_full ? 0ull : p.n_B;
  st->plan = p;
  return p;
}

// Largest float-bit pattern a in [lo, hi) with pred(a), for a predicate that
// holds at lo, fails at hi and changes once in between: a warp tests 32
// patterns at a time (7 rounds over the 2^31 patterns of the non-negative
// floats). All 32 lanes call it.
template <class Pred>
__device__ __forceinline__ unsigned int last_true(unsigned int lo, unsigned int hi, Pred pred) {
  const unsigned int lane = threadIdx.x & 31u;
  while (hi - lo > 1u) {
    const unsigned int step = (hi - lo + 32u) / 33u;
    const unsigned int off = step * (lane + 1u);
    const bool in = off < hi - lo;
    const unsigned int t = __ballot_sync(0xffffffffu, in && pred(lo + off));
    const unsigned int k = (unsigned int)__popc(t);  // the first k patterns pass
    hi = k < 32u ? min(hi, lo + step * (k + 1u)) : hi;
    lo += step * k;
  }
  return lo;
}

// One cluster of kPlanCluster blocks. The first block scans the histogram (and
// clears it for the next measurement), finds the median bins and the bracket
// of the MAD and writes the plan; then all blocks write their share of the
// class table (and clear the histograms of full selection passes, where those
// will run).
//
// Latency-bound: one block with the plan proper on one thread took 40 us a
// measurement whatever the cube's size (two bisections of 31 dependent steps
// in float64, and 64 table cells a thread); with the bisections as 33-ary
// searches by two warps and the table spread over eight SMs it takes 14 us.
constexpr int kPlanCluster = 8;
constexpr int kPlanThreads = 1024;
__global__ void __cluster_dims__(kPlanCluster, 1, 1) __launch_bounds__(kPlanThreads)
    k_plan(DevState* st, unsigned long long* __restrict__ hist, int win, const float* src, long long n_total, Lists L,
           float threshold, int clip, int std_mode, unsigned int force_flags) {
  namespace cg = cooperative_groups;
  extern __shared__ unsigned long long cum[];  // kNumBins + 1
  __shared__ unsigned long long wsum[32];
  __shared__ NoisePlan s_plan;
  __shared__ int s_bins[2];
  __shared__ unsigned int s_T[2];
  chain_begin();
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int tid = threadIdx.x, warp = tid >> 5;
  const BinCfg cfg = win ? st->win : kFullRange;
  if (rank == 0) {
    constexpr int kLoads = (kNumBins + kPlanThreads - 1) / kPlanThreads;
    unsigned long long h[kLoads];  // all in flight together
#pragma unroll
    for (int j = 0; j < kLoads; ++j) h[j] = j * kPlanThreads + tid < kNumBins ? hist[j * kPlanThreads + tid] : 0ull;
#pragma unroll
    for (int j = 0; j < kLoads; ++j) {
      const int b = j * kPlanThreads + tid;
      if (b < kNumBins) {
        cum[b] = h[j];
        hist[b] = 0ull;
      }
    }
    if (tid == 0) {
      s_bins[0] = s_bins[1] = 0;
      s_T[0] = s_T[1] = 0xffffffffu;
    }
    __syncthreads();
    constexpr int kPer = (kNumBins + kPlanThreads - 1) / kPlanThreads;
    unsigned long long loc[kPer];
    unsigned long long s = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int b = tid * kPer + j;
      loc[j] = b < kNumBins ? cum[b] : 0ull;
      s += loc[j];
    }
    // block exclusive scan of s
    unsigned long long incl = s;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long t = __shfl_up_sync(0xffffffffu, incl, o);
      if ((tid & 31) >= o) incl += t;
    }
    if ((tid & 31) == 31) wsum[warp] = incl;
    __syncthreads();
    if (tid < 32) {
      const unsigned long long w = wsum[tid];
      unsigned long long wi = w;
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(0xffffffffu, wi, o);
        if (tid >= o) wi += t;
      }
      wsum[tid] = wi - w;
      if (tid == 31) cum[kNumBins] = wi;
    }
    __syncthreads();
    const unsigned long long n = cum[kNumBins];
    const unsigned long long k_lo = n ? (n - 1ull) / 2ull : 0ull, k_hi = n / 2ull;
    unsigned long long run = wsum[warp] + incl - s;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int b = tid * kPer + j;
      if (b < kNumBins) {
        cum[b] = run;
        // bins of the two middle order statistics
        if (k_lo >= run && k_lo < run + loc[j]) s_bins[0] = b;
        if (k_hi >= run && k_hi < run + loc[j]) s_bins[1] = b;
      }
      run += loc[j];
    }
    __syncthreads();
    if (warp < 2 && n > 0ull && !std_mode) {
      // MAD bracket: warp 0 T1, warp 1 T2 (0xffffffff: none)
      const PlanCtx P{cum, cfg, bin_lo_value(s_bins[0], cfg), bin_hi_value(s_bins[1], cfg)};
      if (isfinite(P.m_min) && isfinite(P.m_max)) {
        // T1 (warp 0): the largest T with possibly-within count <= k_lo (then
        // MAD > T1); T2 (warp 1): the smallest with surely-within count >=
        // k_hi + 1 (then MAD < T2), one above the largest without
        const bool t2 = warp == 1;
        const unsigned int top = t2 ? 0x7f7fffffu : 0x7f800000u;
        const auto under = [&](unsigned int b) {
          return within(P, __uint_as_float(b), t2) <= (t2 ? k_hi : k_lo);
        };
        unsigned int T = 0xffffffffu;
        if (t2 ? !under(top) : under(0u)) T = last_true(0u, top, under) + (t2 ? 1u : 0u);
        if ((tid & 31) == 0) s_T[warp] = T;
      }
    }
    __syncthreads();
    if (tid == 0)
      s_plan = plan_of(st, cum, cfg, s_bins[0], s_bins[1], s_T[0], s_T[1], src, n_total, L, threshold, clip, std_mode,
                       force_flags);
  }
  cl.sync();
  static_assert(sizeof(NoisePlan) % 4 == 0 && sizeof(NoisePlan) / 4 <= kPlanThreads, "a word per thread");
  if (rank != 0 && tid < (int)(sizeof(NoisePlan) / 4))
    reinterpret_cast<unsigned int*>(&s_plan)[tid] = reinterpret_cast<unsigned int*>(cl.map_shared_rank(&s_plan, 0))[tid];
  cl.sync();  // every copy is taken (a block's shared memory stays until its readers are done)
  const int t = rank * kPlanThreads + tid, nt = kPlanCluster * kPlanThreads;
  if (s_plan.flags & (PLAN_MED_FULL | PLAN_MAD_FULL)) {
    for (int i = t; i < 3 * kSelBins; i += nt) {
      (&st->sel_med.hist[0][0])[i] = 0ull;
      (&st->sel_mad.hist[0][0])[i] = 0ull;
    }
  }
  if (L.cls != nullptr) fill_class_table(s_plan, cfg, L.cls, t, nt);
}

cudaError_t launch_plan(DevState* st, unsigned long long* hist, int win, const float* src, long long n_total,
                        Lists L, float threshold, int clip, int std_mode, unsigned int force_flags,
                        cudaStream_t s) {
  const size_t smem = (kNumBins + 1) * sizeof(unsigned long long);
  return launch_chained(k_plan, kPlanCluster, kPlanThreads, smem, 0, s, st, hist, win, src, n_total, L, threshold, clip,
                        std_mode, force_flags);
}

// ---------------------------------------------------------------------------
// Candidate pass. A warp takes chunks of 128 consecutive values; lane l reads
// values l, l + 32, l + 64 and l + 96 of a chunk, so one ballot per read is
// exactly one word of the bit mask. Each value costs a class-table lookup
// (shared memory). A MAD candidate (0.7 % of the values) goes to its lane's own
// column of shared memory, without a vote; one vote per chunk finds the rare
// other classes (the SURE bit feeds the mask ballot; median candidates and
// undecided voxels are staged per warp) and full columns. Columns and stages
// are flushed with one atomic each.
//
// What bounds it: the shared-memory pipe (63 % busy, half of its wavefronts bank
// conflicts of the lookups) and issue (64 %, 19.5 instructions a value). With a
// vote per 32 values and the 20 % of the groups that hold a MAD candidate in the
// listing path it was issue (72 %, 22.4): 1200 x 1200 x 1024 values took
// 1.10 ms, now 1.06; the read alone is 0.88 at the measured HBM rate. More loads
// in flight (a cp.async ring in shared memory) cost that pipe more than they
// gave: 1.27. The columns take what two blocks an SM leave: 8 values a lane
// instead of 11 were flushed more often and cost 0.06 ms a pair where the noise
// varies by 30 % from channel to channel (more candidates).
constexpr int kP2Threads = 512;
constexpr int kP2Warps = kP2Threads / 32;
constexpr int kP2Unroll = 2;                 // chunks a warp classifies per iteration (the next ones load meanwhile)
constexpr int kP2Col = 11;                   // a lane's MAD candidates; a chunk adds at most 4
constexpr int kP2FlushAt = 8;                // flush a list holding more than this after a chunk
constexpr int kP2Stage = kP2FlushAt + 128;   // one chunk adds at most 128 entries per list
constexpr size_t kP2Smem = kClsCells + sizeof(float) * kP2Col * kP2Threads +
                           (size_t)kP2Warps * kP2Stage * (sizeof(float) + sizeof(unsigned long long));

// The lanes' columns (n values each, kP2Threads apart from `mine` on) to the list.
__device__ __forceinline__ void column_flush(const float* mine, int& n, float* glob, unsigned long long* gcount,
                                             unsigned long long cap, unsigned int* status) {
  const int lane = threadIdx.x & 31;
  int x = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  unsigned long long base = 0ull;
  if (lane == 31 && x > 0) {
    base = atomicAdd(gcount, (unsigned long long)x);
    if (base + (unsigned long long)x > cap) atomicOr(status, (unsigned int)SC_ST_OVERFLOW);
  }
  base = __shfl_sync(0xffffffffu, base, 31) + (unsigned long long)(x - n);
  for (int i = 0; i < n; ++i)
    if (base + i < cap) glob[base + i] = mine[i * kP2Threads];
  n = 0;
}

template <typename T>
__device__ __forceinline__ void stage_flush(T* stage, int& cnt, T* glob, unsigned long long* gcount,
                                            unsigned long long cap, unsigned int* status) {
  __syncwarp();
  const int lane = threadIdx.x & 31;
  unsigned long long base = 0;
  if (lane == 0 && cnt > 0) base = atomicAdd(gcount, (unsigned long long)cnt);
  base = __shfl_sync(0xffffffffu, base, 0);
  if (base + (unsigned long long)cnt > cap) {
    if (lane == 0) atomicOr(status, (unsigned int)SC_ST_OVERFLOW);
  } else {
    for (int i = lane; i < cnt; i += 32) glob[base + i] = stage[i];
  }
  __syncwarp();
  cnt = 0;
}

// Appends val from the lanes whose bit is set in b (the warp's ballot of pred).
template <typename T>
__device__ __forceinline__ void stage_push(unsigned int b, bool pred, unsigned int lanes_below, T val, T* stage,
                                           int& cnt) {
  if (pred) stage[cnt + __popc(b & lanes_below)] = val;
  cnt += __popc(b);
}

// Loads the kP2Unroll chunks of 128 values from chunk ch0 on; values past n
// read as NaN (class 0, never sure, never listed).
__device__ __forceinline__ void p2_load(const float* __restrict__ src, long long n, long long ch0, int lane,
                                        float (&a)[kP2Unroll][4]) {
  const float* base = src + ch0 * 128 + lane;
  if ((ch0 + kP2Unroll) * 128 <= n) {
#pragma unroll
    for (int u = 0; u < kP2Unroll; ++u)
#pragma unroll
      for (int c = 0; c < 4; ++c) a[u][c] = __ldg(base + 128 * u + 32 * c);
  } else {
#pragma unroll
    for (int u = 0; u < kP2Unroll; ++u)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const long long v = (ch0 + u) * 128 + 32 * c + lane;
        a[u][c] = v < n ? __ldg(src + v) : __int_as_float(0x7fc00000);
      }
  }
}

__global__ void __launch_bounds__(kP2Threads, 2) k_pass2(const float* __restrict__ src, long long n,
                                                         uint32_t* mbits, DevState* st, Lists L) {
  extern __shared__ __align__(16) unsigned char p2_smem[];
  chain_open();
  const NoisePlan p = st->plan;
  if (p.flags & (PLAN_EMPTY | PLAN_STD)) return;
  const bool do_clip = (p.flags & PLAN_CLIP) && !(p.flags & PLAN_CLIP_FULL) && mbits != nullptr;
  if ((p.flags & PLAN_MED_FULL) && (p.flags & PLAN_MAD_FULL) && !do_clip) return;
  unsigned char* cls = p2_smem;
  for (int i = threadIdx.x; i < kClsCells / 16; i += kP2Threads)
    reinterpret_cast<uint4*>(cls)[i] = __ldg(reinterpret_cast<const uint4*>(L.cls) + i);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* const cols = reinterpret_cast<float*>(p2_smem + kClsCells);
  float* const mine = cols + threadIdx.x;  // this lane's MAD candidates
  unsigned long long* samb = reinterpret_cast<unsigned long long*>(cols + kP2Col * kP2Threads) + warp * kP2Stage;
  float* smed = reinterpret_cast<float*>(reinterpret_cast<unsigned long long*>(cols + kP2Col * kP2Threads) +
                                         kP2Warps * kP2Stage) + warp * kP2Stage;
  __syncthreads();
  const float thr_lo = p.thr_lo, thr_hi = p.thr_hi;
  const unsigned int lanes_below = (1u << lane) - 1u;
  int nmed = 0, ncol = 0, namb = 0;
  const long long nchunks = (n + 127) >> 7;
  const long long wstride = (long long)gridDim.x * kP2Warps * kP2Unroll;
  float a[kP2Unroll][4], nxt[kP2Unroll][4];
  long long ch0 = ((long long)blockIdx.x * kP2Warps + warp) * kP2Unroll;
  if (ch0 < nchunks) p2_load(src, n, ch0, lane, a);
  for (; ch0 < nchunks; ch0 += wstride) {
    if (ch0 + wstride < nchunks) p2_load(src, n, ch0 + wstride, lane, nxt);
#pragma unroll
    for (int u = 0; u < kP2Unroll; ++u) {
      const long long ch = ch0 + u;
      unsigned int k[4], sure_w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int c = 0; c < 4; ++c) k[c] = cls[__float_as_uint(a[u][c]) >> 16];
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (k[c] & CLS_MAD) mine[kP2Threads * ncol++] = a[u][c];
      // the rest concerns few chunks: one vote settles the others
      const unsigned int other = (k[0] | k[1] | k[2] | k[3]) & ~CLS_MAD;
      if (!__any_sync(0xffffffffu, other != 0u || ncol > kP2Col - 4)) continue;
      if (__any_sync(0xffffffffu, ncol > kP2Col - 4))
        column_flush(mine, ncol, L.mad, &st->n_cand_mad, L.cap.mad, &st->status);
      bool any_sure = false;  // warp-uniform
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        // the other classes present in the group, one reduction for the warp
        const unsigned int present = __reduce_or_sync(0xffffffffu, k[c]) & ~CLS_MAD;
        if (present == 0u) continue;
        if (present & CLS_SURE) sure_w[c] = __ballot_sync(0xffffffffu, (k[c] & CLS_SURE) != 0u);
        if (present & (CLS_MED | CLS_AMB)) {
          const float s = a[u][c];
          const float as = fabsf(s);
          const bool pm = (k[c] & CLS_MED) != 0u;
          const bool amb_cell = (k[c] & CLS_AMB) != 0u;  // finite: the cell is not Inf / NaN
          const bool sure = amb_cell && as > thr_hi;
          const bool pamb = amb_cell && as > thr_lo && !sure;
          sure_w[c] |= __ballot_sync(0xffffffffu, sure);
          const unsigned int bmed = __ballot_sync(0xffffffffu, pm);
          const unsigned int bamb = __ballot_sync(0xffffffffu, pamb);
          stage_push(bmed, pm, lanes_below, s, smed, nmed);
          stage_push(bamb, pamb, lanes_below, (unsigned long long)(ch * 128 + 32 * c + lane), samb, namb);
        }
        any_sure |= sure_w[c] != 0u;
      }
      if (any_sure) {
        // lane c owns mask word 4 * ch + c of this chunk (no SURE cells, so
        // no words, without a clip)
        unsigned int w = sure_w[0];
        w = lane == 1 ? sure_w[1] : w;
        w = lane == 2 ? sure_w[2] : w;
        w = lane == 3 ? sure_w[3] : w;
        if (do_clip && lane < 4 && w != 0u) atomicOr(mbits + ch * 4 + lane, w);
      }
      if (max(nmed, namb) > kP2FlushAt) {
        if (nmed > kP2FlushAt) stage_flush(smed, nmed, L.med, &st->n_cand_med, L.cap.med, &st->status);
        if (namb > kP2FlushAt) stage_flush(samb, namb, L.amb, &st->n_amb, L.cap.amb, &st->status);
      }
    }
#pragma unroll
    for (int u = 0; u < kP2Unroll; ++u)
#pragma unroll
      for (int c = 0; c < 4; ++c) a[u][c] = nxt[u][c];
  }
  stage_flush(smed, nmed, L.med, &st->n_cand_med, L.cap.med, &st->status);
  column_flush(mine, ncol, L.mad, &st->n_cand_mad, L.cap.mad, &st->status);
  stage_flush(samb, namb, L.amb, &st->n_amb, L.cap.amb, &st->status);
}

cudaError_t launch_pass2(const float* src, long long n, uint32_t* mbits, DevState* st, Lists L, int sms,
                         cudaStream_t s) {
  const long long chunks = (n + 127) / 128;
  long long want = (chunks + kP2Warps * kP2Unroll - 1) / (kP2Warps * kP2Unroll);
  int grid = (int)(want < 1 ? 1 : (want > 2LL * sms ? 2LL * sms : want));
  k_pass2<<<grid, kP2Threads, kP2Smem, s>>>(src, n, mbits, st, L);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Radix selection. MAD keys are the correctly rounded float of the exact
// |s - m| (m is the exact median, a double): rounding is monotone, so the
// order statistics of the keys are the rounded order statistics of |s - m|.
// What a pass reads of its SelJob.
struct SelIn {
  const float* list;
  const unsigned long long* count_ptr;
  int mode;
};
__device__ __forceinline__ bool sel_key(const SelIn& J, double m, float s, unsigned int* key) {
  if (!isfinite(s)) return false;
  if (J.mode == SEL_VALUE) {
    *key = fkey(s);
  } else {
    *key = fkey(__double2float_rn(fabs((double)s - m)));
  }
  return true;
}

// A candidate list of |s - m| keys (not the whole array) holds, after the
// first round, the keys themselves in place of the values: that round forms
// each key once in float64 (slow on this GPU) and the later rounds read it.
// kNoKey marks a non-finite value (no finite key is that large; read as a
// float it is a NaN, so it is no value either).
constexpr unsigned int kNoKey = 0xffffffffu;
__device__ __forceinline__ bool sel_keys_stored(const SelIn& J) {
  return J.mode == SEL_ABSDEV && J.count_ptr != nullptr;
}
__device__ __forceinline__ bool sel_key_of(const SelIn& J, bool stored, double m, float v, unsigned int* key) {
  if (stored) {
    *key = __float_as_uint(v);
    return *key != kNoKey;
  }
  return sel_key(J, m, v, key);
}

// The lists are read kSelUnroll values a thread at a time, loads first, so
// that enough of them are in flight (a list of millions of candidates is
// otherwise bound by the latency of one load per thread).
constexpr int kSelUnroll = 16;
__device__ __forceinline__ void sel_load(const float* list, unsigned long long i0,
                                         unsigned long long stride, unsigned long long count,
                                         float (&v)[kSelUnroll]) {
#pragma unroll
  for (int u = 0; u < kSelUnroll; ++u) {
    const unsigned long long i = i0 + u * stride;
    v[u] = i < count ? __ldcg(list + i) : __uint_as_float(kNoKey);  // past the end: no key either way
  }
}

// Elements in the list: the candidate count, clamped to the buffer capacity
// (count_fixed), or the whole array.
__device__ __forceinline__ unsigned long long sel_count(const SelJob& J) {
  return J.count_ptr ? min(*J.count_ptr, J.count_fixed) : J.count_fixed;
}

// Every block redoes the pick of round r-1 from its histogram (same result
// everywhere); block 0 records it.
__device__ void sel_pick(SelJob* J, int r, unsigned int* prefix, unsigned long long* rank, unsigned int* status) {
  __shared__ unsigned long long s_part[32];
  __shared__ unsigned int s_digit;
  __shared__ unsigned long long s_rank;
  const unsigned long long* h = J->hist[r - 1];
  const int tid = threadIdx.x, nt = blockDim.x;  // nt == 256 or 1024
  const int per = kSelBins / nt;
  unsigned long long loc = 0;
  for (int j = 0; j < per; ++j) loc += h[tid * per + j];
  // exclusive scan over threads
  unsigned long long incl = loc;
  for (int o = 1; o < 32; o <<= 1) {
    unsigned long long t = __shfl_up_sync(0xffffffffu, incl, o);
    if ((tid & 31) >= o) incl += t;
  }
  if ((tid & 31) == 31) s_part[tid >> 5] = incl;
  __syncthreads();
  if (tid < 32) {
    unsigned long long w = (tid < nt / 32) ? s_part[tid] : 0ull, wi = w;
    for (int o = 1; o < 32; o <<= 1) {
      unsigned long long t = __shfl_up_sync(0xffffffffu, wi, o);
      if (tid >= o) wi += t;
    }
    s_part[tid] = wi - w;
  }
  if (tid == 0) { s_digit = 0xffffffffu; s_rank = 0ull; }
  __syncthreads();
  const unsigned long long want = *rank;
  unsigned long long run = s_part[tid >> 5] + incl - loc;
  for (int j = 0; j < per; ++j) {
    const unsigned long long c = h[tid * per + j];
    if (want >= run && want < run + c) {
      s_digit = (unsigned)(tid * per + j);
      s_rank = want - run;
    }
    run += c;
  }
  __syncthreads();
  if (s_digit == 0xffffffffu) {
    if (tid == 0) atomicOr(status, (unsigned int)SC_ST_INTERNAL);
    *prefix = 0u;
    *rank = 0ull;
  } else {
    *prefix = ((*prefix) << sel_bits(r - 1)) | s_digit;
    *rank = s_rank;
  }
  __syncthreads();
}

__device__ __forceinline__ unsigned long long sel_rank0(const DevState* st, const SelJob* J, int which) {
  unsigned long long r = J->rank_lo;
  if (which == 1 && J->count_ptr != nullptr) r -= st->n_below;
  return r;
}

// The full passes serve measurements with a candidate set above capacity; the
// others have been selected from their lists by k_select.
__device__ __forceinline__ bool sel_by_full_passes(const NoisePlan& p) {
  return !(p.flags & (PLAN_EMPTY | PLAN_STD)) && (p.flags & (PLAN_MED_FULL | PLAN_MAD_FULL));
}

__device__ void sel_result(DevState* st, SelJob* J, int which, int pair);

__device__ void sel_round(DevState* st, int which, int r) {
  __shared__ unsigned int sh[kSelBins];
  SelJob* J = which ? &st->sel_mad : &st->sel_med;
  unsigned int prefix = 0u;
  unsigned long long rank = sel_rank0(st, J, which);
  const unsigned long long count = sel_count(*J);
  if (r == 0 && rank >= count) {
    if (threadIdx.x == 0 && blockIdx.x == 0) atomicOr(&st->status, (unsigned int)SC_ST_INTERNAL);
    return;
  }
  if (r > 0) {
    prefix = J->prefix[r - 1 + 0];
    rank = J->rank_in[r - 1 + 0];
    if (r == 1) { prefix = 0u; rank = sel_rank0(st, J, which); }
    sel_pick(J, r, &prefix, &rank, &st->status);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      J->prefix[r] = prefix;
      J->rank_in[r] = rank;
    }
  }
  for (int i = threadIdx.x; i < kSelBins; i += blockDim.x) sh[i] = 0u;
  __syncthreads();
  const double m = st->m;
  const int shift_prev = (r == 0) ? 32 : sel_shift(r - 1);
  const int shift = sel_shift(r);
  const unsigned int dmask = (1u << sel_bits(r)) - 1u;
  const SelIn Jl{J->list, J->count_ptr, J->mode};
  const bool stored = r > 0 && sel_keys_stored(Jl);
  // the first round of a list of |s - m| values writes their keys over them
  float* const keys_out = (r == 0 && sel_keys_stored(Jl)) ? const_cast<float*>(Jl.list) : nullptr;
  // whole warps iterate together: a warp whose 32 values share one digit (a
  // list's candidates cluster in few digits, in the first round mostly in
  // one) adds to its bin once
  const unsigned lane = threadIdx.x & 31u;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long w0 = (unsigned long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); w0 < count;
       w0 += kSelUnroll * stride) {
    float v[kSelUnroll];
    sel_load(Jl.list, w0 + lane, stride, count, v);
#pragma unroll
    for (int u = 0; u < kSelUnroll; ++u) {
      const unsigned long long i = w0 + u * stride + lane;
      unsigned int key = 0u;
      bool ok = i < count && sel_key_of(Jl, stored, m, v[u], &key);
      if (keys_out && i < count) keys_out[i] = __uint_as_float(ok ? key : kNoKey);
      ok = ok && !(shift_prev < 32 && (key >> shift_prev) != prefix);
      const unsigned digit = ok ? (key >> shift) & dmask : 0xffffffffu;
      const unsigned d0 = __shfl_sync(0xffffffffu, digit, 0);
      if (__all_sync(0xffffffffu, digit == d0)) {
        if (lane == 0 && ok) atomicAdd(&sh[d0], 32u);
      } else if (ok) {
        atomicAdd(&sh[digit], 1u);
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kSelBins; i += blockDim.x)
    if (sh[i]) atomicAdd(&J->hist[r][i], (unsigned long long)sh[i]);
}

__device__ void sel_succ(DevState* st, int which, int pair) {
  __shared__ unsigned long long s_c[8];
  __shared__ unsigned int s_m[8];
  SelJob* J = which ? &st->sel_mad : &st->sel_med;
  const unsigned long long count = sel_count(*J);
  if (sel_rank0(st, J, which) >= count) return;  // (the first round has set the error)
  unsigned int prefix = J->prefix[2];
  unsigned long long rank = J->rank_in[2];
  sel_pick(J, 3, &prefix, &rank, &st->status);
  const unsigned int key_lo = prefix;
  if (blockIdx.x == 0 && threadIdx.x == 0) J->key_lo = key_lo;
  const double m = st->m;
  const SelIn Jl{J->list, J->count_ptr, J->mode};
  const bool stored = sel_keys_stored(Jl);
  unsigned long long c = 0;
  unsigned int mn = 0xffffffffu;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i0 = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i0 < count;
       i0 += kSelUnroll * stride) {
    float v[kSelUnroll];
    sel_load(Jl.list, i0, stride, count, v);
#pragma unroll
    for (int u = 0; u < kSelUnroll; ++u) {
      unsigned int key;
      if (!sel_key_of(Jl, stored, m, v[u], &key)) continue;  // includes the places past the end
      if (key <= key_lo) ++c; else mn = min(mn, key);
    }
  }
  c = warp_sum_u64(c);
  for (int o = 16; o > 0; o >>= 1) mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) { s_c[warp] = c; s_m[warp] = mn; }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long ct = 0;
    unsigned int mt = 0xffffffffu;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { ct += s_c[w]; mt = min(mt, s_m[w]); }
    if (ct) atomicAdd(&J->c_le, ct);
    if (mt != 0xffffffffu) atomicMin(&J->min_gt, mt);
    __threadfence();
    // the last block to finish forms the result
    if (atomicAdd(&J->done, 1u) == gridDim.x - 1u) {
      __threadfence();
      sel_result(st, J, which, pair);
    }
  }
}

// (one thread, after every block's counts)
__device__ void sel_result(DevState* st, SelJob* J, int which, int pair) {
  const NoisePlan& p = st->plan;
  const unsigned long long r_hi = sel_rank0(st, J, which) + (p.k_hi - p.k_lo);
  const unsigned long long c_le = *(volatile unsigned long long*)&J->c_le;
  const unsigned int k_lo = *(volatile unsigned int*)&J->key_lo;
  unsigned int k_hi = k_lo;
  if (r_hi >= c_le) {
    k_hi = *(volatile unsigned int*)&J->min_gt;
    if (k_hi == 0xffffffffu) {
      atomicOr(&st->status, (unsigned int)SC_ST_INTERNAL);
      k_hi = k_lo;
    }
  }
  const double v_lo = (double)fkey_inv(k_lo), v_hi = (double)fkey_inv(k_hi);
  const double v = (k_hi == k_lo) ? v_lo : 0.5 * (v_lo + v_hi);
  if (which == 0) {
    st->m = v;
  } else {
    st->mad = v;
    st->sigma_cur_d = kMadToSigma * v;
    const float sg = sigma_of_mad(v);
    st->sigma_cur = sg;
    if (pair >= 0) st->sigma[pair] = sg;
    if (!(sg > 0.0f)) st->warn |= SC_WARN_ZERO_SIGMA;
  }
}

__global__ void __launch_bounds__(256) k_sel_round(DevState* st, int which, int r) {
  chain_begin();
  if (sel_by_full_passes(st->plan)) sel_round(st, which, r);
}

__global__ void __launch_bounds__(256) k_sel_succ(DevState* st, int which, int pair) {
  chain_begin();
  if (sel_by_full_passes(st->plan)) sel_succ(st, which, pair);
}

// Mostly there is nothing to do, and the eight launches return at once, about
// 1 us each. One cooperative launch in their place saved most of that (12 pairs
// on 217 x 331 x 509 voxels: 3.64 ms against 3.75), but a cooperative grid
// starts only when all of it fits: beside other lanes, another context or a
// kernel of the program that keeps an SM it waited for them to end.
cudaError_t launch_select_full(DevState* st, int pair, int sms, cudaStream_t s) {
  const unsigned grid = 2u * (unsigned)sms;
  cudaError_t e = cudaSuccess;
  for (int which = 0; which < 2 && e == cudaSuccess; ++which) {
    for (int r = 0; r < 3 && e == cudaSuccess; ++r) e = launch_chained(k_sel_round, grid, 256, 0, 0, s, st, which, r);
    if (e == cudaSuccess) e = launch_chained(k_sel_succ, grid, 256, 0, 0, s, st, which, which ? pair : -1);
  }
  return e;
}

// ---------------------------------------------------------------------------
// STD mode: sums of d = (x - K) 2^-e and of d^2 over the finite values, with K
// in the median's bin and 2^e above all magnitudes (both from the histogram:
// the squares of float32 data can overflow or underflow float32). Where K is
// so far from the mean that S2 - S1^2 / n would lose a bit (data on an offset
// of many times their spread), a second pass takes the mean as K.
//
// Each thread keeps its sums as unevaluated triples of floats: the difference,
// the square and the additions are exact in the first two parts (TwoSum, and an
// FMA for a product's error), the third takes what those leave, 2^-48 of the
// sum, rounded to 2^-24 of itself. So a thread's sums are good to float64's
// last bit, and the noise is as near to the exact one as with float64 sums
// about the mean in two passes (2^-50 either way at 10 to 400 M values; pairs
// of floats gave 2^-44 to 2^-39). The conversions and FMAs of those bound them
// at 268 us a pass on 256 x 250 x 600 voxels (the float64 pipe is slow on this
// part); this pass takes 61 us (pairs: 44, a read at the measured HBM rate: 23).
// a += x + y + low, y and low well below x.
__device__ __forceinline__ void sum3_add(float (&a)[3], float x, float y, float low) {
  float e, f, g;
  a[0] = two_sum(a[0], x, &e);
  a[1] = two_sum(a[1], e, &f);
  a[1] = two_sum(a[1], y, &g);
  a[2] = __fadd_rn(a[2], __fadd_rn(__fadd_rn(f, g), low));
}
__device__ __forceinline__ void sum3_add(float (&a)[3], float x) {
  float e, f;
  a[0] = two_sum(a[0], x, &e);
  a[1] = two_sum(a[1], e, &f);
  a[2] = __fadd_rn(a[2], f);
}
__device__ __forceinline__ double sum3_value(const float (&a)[3]) {
  return (double)a[0] + ((double)a[1] + (double)a[2]);
}

// PLAIN: neither shift nor scale.
template <bool PLAIN>
__device__ __forceinline__ void std_add(float x, float scale, float shift, float (&s1)[3], float (&s2)[3], unsigned* n) {
  if (!(fabsf(x) <= FLT_MAX)) return;  // NaN and Inf
  if (PLAIN) {
    sum3_add(s1, x);
    const float p = __fmul_rn(x, x);
    sum3_add(s2, p, __fmaf_rn(x, x, -p), 0.0f);
  } else {
    float l;  // d = h + l
    const float h = two_sum(__fmul_rn(x, scale), -shift, &l);  // (scale: a power of two)
    sum3_add(s1, h, l, 0.0f);
    // d^2 = h^2 + 2 h l + l^2, the first two as products and their errors
    const float p = __fmul_rn(h, h), h2 = __fadd_rn(h, h), q = __fmul_rn(h2, l);
    float re;
    const float r = two_sum(__fmaf_rn(h, h, -p), q, &re);
    sum3_add(s2, p, r, __fmaf_rn(l, l, __fadd_rn(re, __fmaf_rn(h2, l, -q))));
  }
  ++*n;
}

template <bool PLAIN>
__device__ __forceinline__ void std_sums(const float* __restrict__ x, long long n, float scale, float shift,
                                         float (&s1)[3], float (&s2)[3], unsigned* cnt) {
  const long long t0 = (long long)blockIdx.x * 256 + threadIdx.x, stride = (long long)gridDim.x * 256;
  const long long nq = (reinterpret_cast<uintptr_t>(x) & 15u) == 0 ? n >> 2 : 0;
  for (long long q = t0; q < nq; q += 4 * stride) {
    float4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      v[u] = q + u * stride < nq ? __ldg(reinterpret_cast<const float4*>(x) + q + u * stride)
                                 : make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      std_add<PLAIN>(v[u].x, scale, shift, s1, s2, cnt);
      std_add<PLAIN>(v[u].y, scale, shift, s1, s2, cnt);
      std_add<PLAIN>(v[u].z, scale, shift, s1, s2, cnt);
      std_add<PLAIN>(v[u].w, scale, shift, s1, s2, cnt);
    }
  }
  for (long long i = 4 * nq + t0; i < n; i += stride) std_add<PLAIN>(__ldg(x + i), scale, shift, s1, s2, cnt);
}

// The first pass, or the second, which only runs where the first pass's shift
// was too far from the mean. The last block of a pass forms the result (or
// asks for the second pass).
__global__ void __launch_bounds__(256) k_std_pass(const float* __restrict__ x, long long n, DevState* st, int second,
                                                  int pair) {
  __shared__ double s_a[8], s_b[8];
  __shared__ unsigned s_n[8];
  chain_begin();
  if ((st->plan.flags & PLAN_EMPTY) || (second && !st->std_again)) return;
  const float scale = st->std_scale, shift = __fmul_rn(st->std_shift, scale);
  float p1[3] = {0.0f, 0.0f, 0.0f}, p2[3] = {0.0f, 0.0f, 0.0f};
  unsigned cnt = 0u;
  if (scale == 1.0f && shift == 0.0f) std_sums<true>(x, n, scale, shift, p1, p2, &cnt);
  else std_sums<false>(x, n, scale, shift, p1, p2, &cnt);
  double s1 = sum3_value(p1), s2 = sum3_value(p2);
  for (int o = 16; o > 0; o >>= 1) {
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    s_a[warp] = s1;
    s_b[warp] = s2;
    s_n[warp] = cnt;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  unsigned long long ct = 0ull;
  s1 = s2 = 0.0;
  for (int w = 0; w < 8; ++w) {
    s1 += s_a[w];
    s2 += s_b[w];
    ct += s_n[w];
  }
  atomicAdd(&st->sum, s1);
  atomicAdd(&st->sum2, s2);
  atomicAdd(&st->count, ct);
  __threadfence();
  if (atomicAdd(&st->std_blocks, 1u) != gridDim.x - 1u) return;
  __threadfence();
  const double c = (double)*(volatile unsigned long long*)&st->count;
  s1 = *(volatile double*)&st->sum;
  s2 = *(volatile double*)&st->sum2;
  const double var = s2 - s1 * s1 / c;
  if (!second && c > 1.0 && !(var >= 0.5 * s2)) {
    st->std_again = 1;
    st->std_shift = __double2float_rn((double)st->std_shift + s1 / c / (double)scale);  // the mean
    st->sum = st->sum2 = 0.0;
    st->count = 0ull;
    st->std_blocks = 0u;
    return;
  }
  const double sd = c > 1.0 ? sqrt(fmax(var, 0.0) / (c - 1.0)) / (double)scale : 0.0;
  const float sg = (float)sd;
  st->sigma_cur = sg;
  st->sigma_cur_d = sd;
  if (pair >= 0) st->sigma[pair] = sg;
  if (!(sg > 0.0f)) st->warn |= SC_WARN_ZERO_SIGMA;
}

cudaError_t launch_std(const float* src, long long n, DevState* st, int pair, int sms, cudaStream_t s) {
  const long long want = (n + 4095) / 4096;  // four 16-byte loads a thread
  const int grid = (int)(want > 6LL * sms ? 6LL * sms : want);
  const cudaError_t e = launch_chained(k_std_pass, grid, 256, 0, 0, s, src, n, st, 0, pair);
  if (e != cudaSuccess) return e;
  return launch_chained(k_std_pass, grid, 256, 0, 0, s, src, n, st, 1, pair);
}

// ---------------------------------------------------------------------------
// Clip: the voxels that the candidate pass left undecided, or all of them when
// the plan asked for a full pass.
__device__ void clip_listed(const float* __restrict__ src, uint32_t* mbits, const DevState* st, const Lists& L,
                            float thr) {
  const unsigned long long na = min(st->n_amb, L.cap.amb);
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < na;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned long long v = L.amb[i];
    if (fabsf(__ldg(src + v)) > thr) atomicOr(mbits + (v >> 5), 1u << (v & 31ull));
  }
}

// resident k_clip_full blocks per SM (init_noise_attrs, which every context
// creation runs, possibly from several host threads at once)
static std::atomic<int> g_clip_blocks_per_sm{0};

// Lane l holds values l, l + 32, l + 64 and l + 96 of chunk ch (each load
// instruction reads 128 contiguous bytes), so ballot c is mask word 4 ch + c
// as it stands; 0 past n.
__device__ __forceinline__ void clip_load(const float* __restrict__ src, long long n, long long ch, int lane,
                                          float (&a)[4]) {
  const long long v0 = ch * 128 + lane;
  if (ch * 128 + 128 <= n) {
#pragma unroll
    for (int c = 0; c < 4; ++c) a[c] = __ldg(src + v0 + 32 * c);
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) a[c] = (v0 + 32 * c < n) ? __ldg(src + v0 + 32 * c) : 0.0f;
  }
}

// Sets chunk ch's detected bits: lane c < 4 owns word 4 ch + c.
__device__ __forceinline__ void clip_store(uint32_t* mbits, long long ch, int lane, float thr, const float (&a)[4]) {
  unsigned int w = 0u;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float m = fabsf(a[c]);  // NaN fails the first compare, Inf the second
    const unsigned int b = __ballot_sync(0xffffffffu, m > thr && m <= FLT_MAX);
    w = lane == c ? b : w;
  }
  if (lane < 4 && w) atomicOr(mbits + ch * 4 + lane, w);  // no return value: no wait for the word
}

__global__ void __launch_bounds__(256) k_clip_full(const float* __restrict__ src, long long n, uint32_t* mbits,
                                                   DevState* st, Lists L) {
  chain_begin();
  const NoisePlan& p = st->plan;
  if (!(p.flags & PLAN_CLIP) || (p.flags & PLAN_EMPTY)) return;
  const float sg = st->sigma_cur;
  if (!(sg > 0.0f)) return;
  const float thr = __fmul_rn(p.threshold, sg);
  if (!(p.flags & PLAN_CLIP_FULL)) {
    clip_listed(src, mbits, st, L, thr);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long nchunks = (n + 127) / 128;
  const long long stride = (long long)gridDim.x * 8;
  // two chunks a warp per iteration, all eight loads issued before a ballot
  for (long long ch = (long long)blockIdx.x * 8 + warp; ch < nchunks; ch += 2 * stride) {
    const long long ch2 = ch + stride;
    float a[4], b[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    clip_load(src, n, ch, lane, a);
    if (ch2 < nchunks) clip_load(src, n, ch2, lane, b);
    clip_store(mbits, ch, lane, thr, a);
    if (ch2 < nchunks) clip_store(mbits, ch2, lane, thr, b);
  }
}

cudaError_t launch_clip(const float* src, long long n, uint32_t* mbits, DevState* st, Lists L, int sms,
                        cudaStream_t s) {
  // one wave: as many blocks as are resident at once (a second, partial wave
  // would run on a fraction of the SMs)
  const int per_sm = g_clip_blocks_per_sm.load(std::memory_order_relaxed);
  const long long cap = (long long)(per_sm > 0 ? per_sm : 4) * sms;
  long long want = (n + 1023) / 1024;
  int grid = (int)(want < 1 ? 1 : (want > cap ? cap : want));
  return launch_chained(k_clip_full, grid, 256, 0, 0, s, src, n, mbits, st, L);
}


// ---------------------------------------------------------------------------
// After sigma_0: replacement value, bin window, fixed-point scales.
// Fixed-point shift of every pair: X_q = rint(X * 2^f) with
// max|X| * 2^f * Wf <= 2^62 (Wf >= W), so that no exact sum can overflow
// int64. The replacement value repl_d (float64) is quantised once per pair.
__device__ void fx_setup(DevState* st, double repl_d, const PairWeights& W, int n_pairs) {
  const float maxabs = __uint_as_float(st->maxabs_bits);
  const float mx = fmaxf(maxabs, __double2float_ru(repl_d));
  int ex = 0;
  frexpf(mx, &ex);  // mx < 2^ex
  if (mx == 0.0f) ex = 0;
  // f depends on the spatial kernel (through wf) but not on a spectral width up
  // to kShareMaxWz, so pairs with one spatial kernel quantise alike and can
  // share their stored spatial sums. A thread per pair.
  for (int k = threadIdx.x; k < n_pairs; k += blockDim.x) {
    const long long w = W.w[k];
    const int bits = 64 - __clzll((unsigned long long)(W.wf[k] - 1));  // bit length of wf - 1
    int f = 62 - ex - bits;
    if (f > 120) f = 120;
    if (f < -120) f = -120;
    st->fx_shift[k] = f;
    st->fx_scale[k] = ldexpf(1.0f, f);
    st->fx_inv[k] = (float)(ldexp(1.0, -f) / (double)w);
    st->fx_qrepl[k] = __double2ll_rn(ldexp(repl_d, f));
  }
}

__global__ void k_fx_setup(DevState* st, float repl_value, PairWeights W, int n_pairs) {
  if (threadIdx.x == 0) {
    st->repl_d = (double)repl_value;
    st->repl = repl_value;
  }
  fx_setup(st, (double)repl_value, W, n_pairs);
}

cudaError_t launch_fx_setup(DevState* st, float repl_value, const PairWeights& W, int n_pairs, cudaStream_t s) {
  k_fx_setup<<<1, SC_MAX_KERNELS, 0, s>>>(st, repl_value, W, n_pairs);
  return cudaGetLastError();
}

// Window of the fine histogram of the raw cube: the bin of the median of |x|
// gives the scale, and the window spans 2^-20 .. 2^12 of it (as for the
// smoothed cubes), so the plan of the sigma_0 measurement resolves 128 bins
// per octave instead of 16. The median |x| comes from kWinSample values
// spread through the cube (all of them in a smaller cube): a window 32
// octaves wide needs its scale only roughly, and the exact selection that
// follows does not depend on it (a poorly placed window costs candidates,
// never exactness). Where hardly any of them is finite, up to seven further
// samples are taken: of a cube that is blank but for one voxel in 8,000 the
// first may hold none, and full selection passes would follow. One block,
// bound by the latency of its loads: 65,536 values in four batches took 44 to
// 68 us, 8,192 in one take 9 to 10 (21 on 360 x 360 x 1464 values and 78 on
// 1200 x 1200 x 1024 in the first pass over a cube).
constexpr int kWinThreads = 1024;
constexpr long long kWinSample = 8192;
constexpr int kWinPerThread = (int)(kWinSample / kWinThreads);
constexpr int kWinRounds = 8, kWinEnough = 32;  // samples at most; threads that found a finite value
__global__ void __launch_bounds__(kWinThreads) k_window_from_sample(const float* __restrict__ x, Half16 h,
                                                                    long long plane, long long n, DevState* st) {
  extern __shared__ unsigned int wh[];  // full-range histogram of the sample
  __shared__ unsigned long long s_w[32];
  __shared__ int s_mb;
  const BinCfg full = kFullRange;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int i = t; i < kNumBins; i += kWinThreads) wh[i] = 0u;
  __syncthreads();
  // m values, one from every step of the cube (all of a cube of at most
  // kWinSample), at places that follow no row or column
  const long long m = n < kWinSample ? n : kWinSample, step = n / (m > 0 ? m : 1);
#pragma unroll 1
  for (int round = 0; round < kWinRounds; ++round) {
    float v[kWinPerThread];  // all loads in flight
#pragma unroll
    for (int j = 0; j < kWinPerThread; ++j) {
      const long long k = (long long)j * kWinThreads + t;
      const unsigned long long h32 = (unsigned)k * 2654435761u;
      long long i = k * step + (long long)(h32 * (unsigned long long)step >> 32);
      if (round > 0)  // further places anywhere in the cube
        i = (long long)__umul64hi((unsigned long long)(round * kWinSample + k) * 0x9e3779b97f4a7c15ull, (unsigned long long)n);
      v[j] = __int_as_float(0x7fc00000);
      if (k < m) v[j] = h.fmt ? half16_value(__ldg(h.bits + i), h.fmt, __ldg(h.scale + i / plane)) : __ldg(x + i);
    }
    int any = 0;
#pragma unroll
    for (int j = 0; j < kWinPerThread; ++j) {
      if (!isfinite(v[j])) continue;
      atomicAdd(&wh[bin_of(v[j], full)], 1u);
      any = 1;
    }
    if (__syncthreads_count(any) >= kWinEnough || m < kWinSample) break;
  }
  // thread t holds magnitude bins [t * per, t * per + per), both signs
  constexpr int per = (kBinsPerSign + kWinThreads - 1) / kWinThreads;
  unsigned long long c[per], loc = 0;
#pragma unroll
  for (int j = 0; j < per; ++j) {
    const int mb = t * per + j;
    c[j] = mb < kBinsPerSign ? (unsigned long long)wh[kBinsPerSign + mb] + wh[kBinsPerSign - 1 - mb] : 0ull;
    loc += c[j];
  }
  unsigned long long inc = loc;  // inclusive scan over the warp, then over the warps
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_w[warp] = inc;
  if (t == 0) s_mb = -1;
  __syncthreads();
  if (warp == 0) {
    const unsigned long long xw = s_w[lane];
    unsigned long long xi = xw;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, xi, o);
      if (lane >= o) xi += y;
    }
    s_w[lane] = xi;  // inclusive over warps; s_w[31] is the total
  }
  __syncthreads();
  const unsigned long long total = s_w[31];
  // the first magnitude bin whose cumulative count exceeds half of the sample
  unsigned long long run = (warp ? s_w[warp - 1] : 0ull) + inc - loc;
#pragma unroll
  for (int j = 0; j < per; ++j) {
    if (2 * run <= total && 2 * (run + c[j]) > total) s_mb = t * per + j;
    run += c[j];
  }
  __syncthreads();
  if (t == 0) {
    const float scale = (total > 0 && s_mb >= 0) ? (float)mag_hi(s_mb, full) : 0.0f;
    st->win = window_cfg(isfinite(scale) ? scale : 3.0e38f);
  }
}

cudaError_t launch_window_from_sample(const float* x, const Half16* h16, long long plane, long long n, DevState* st,
                                      cudaStream_t s) {
  Half16 h{};
  if (h16) h = *h16;
  k_window_from_sample<<<1, kWinThreads, kNumBins * sizeof(unsigned int), s>>>(x, h, plane, n, st);
  return cudaGetLastError();
}

__global__ void k_sigma0_done(DevState* st, float replacement, PairWeights W, int n_pairs) {
  const float s0 = st->sigma_cur;
  const double repl_d = (replacement > 0.0f) ? (double)replacement * st->sigma_cur_d : 0.0;
  if (threadIdx.x == 0) {
    st->sigma0 = s0;
    st->repl_d = repl_d;
    st->repl = __double2float_rn(repl_d);
    st->win = window_cfg(s0);
    const float mx = fmaxf(__uint_as_float(st->maxabs_bits), st->repl);
    if (s0 > 0.0f && mx > s0 * 1048576.0f) st->warn |= SC_WARN_RANGE;
  }
  fx_setup(st, repl_d, W, n_pairs);
}

cudaError_t launch_sigma0_done(DevState* st, float replacement, const PairWeights& W, int n_pairs, cudaStream_t s) {
  k_sigma0_done<<<1, SC_MAX_KERNELS, 0, s>>>(st, replacement, W, n_pairs);
  return cudaGetLastError();
}

// The latest run's sigmas for sc_copy_sigmas: out[k] = sigma_k (k < n),
// out[n] = sigma_0, all zero when the run's device-side status is an error
// (its sigmas are then meaningless).
__global__ void k_sigma_out(const DevState* st, int n, float* out) {
  const bool ok = st->status == 0u;
  for (int k = threadIdx.x; k <= n; k += blockDim.x) out[k] = ok ? (k < n ? st->sigma[k] : st->sigma0) : 0.0f;
}

cudaError_t launch_sigma_out(const DevState* st, int n, float* out, cudaStream_t s) {
  k_sigma_out<<<1, 64, 0, s>>>(st, n, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// uint8 mask <-> 1-bit working mask.
// Working mask from a caller's uint8 mask: a bit for every set voxel whose
// cube value is finite (non-finite voxels are never replaced, and no clip
// ever sets their bit, so the working mask holds finite voxels only).
//
// What bounds it: the read of the mask. A thread takes a word: two 16-byte
// loads of the mask, and of the cube only the quads with a set voxel, all in
// flight together. 512 x 512 x 256 voxels (0.5 % set): 65 us with a byte
// load a voxel, 17 now.
__device__ __forceinline__ unsigned int mask_word(const uint8_t* __restrict__ m8, long long n, long long v0, bool vec) {
  unsigned int bits = 0u;
  if (vec && v0 + 32 <= n) {
    const uint4 a = __ldg(reinterpret_cast<const uint4*>(m8 + v0)), b = __ldg(reinterpret_cast<const uint4*>(m8 + v0) + 1);
    bits = nonzero_bits(a.x) | nonzero_bits(a.y) << 4 | nonzero_bits(a.z) << 8 | nonzero_bits(a.w) << 12 |
           nonzero_bits(b.x) << 16 | nonzero_bits(b.y) << 20 | nonzero_bits(b.z) << 24 | nonzero_bits(b.w) << 28;
  } else {
    for (int i = 0; i < 32; ++i)
      if (v0 + i < n && m8[v0 + i]) bits |= 1u << i;
  }
  return bits;
}

__global__ void __launch_bounds__(256) k_pack(const uint8_t* __restrict__ m8, const float* __restrict__ cube,
                                              long long n, uint32_t* __restrict__ mbits) {
  const long long nw = (n + 31) / 32;
  const bool vec = (reinterpret_cast<uintptr_t>(m8) & 15u) == 0u && (reinterpret_cast<uintptr_t>(cube) & 15u) == 0u;
  for (long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x; w < nw; w += (long long)gridDim.x * blockDim.x) {
    const long long v0 = w * 32;
    unsigned int bits = mask_word(m8, n, v0, vec);
    if (bits != 0u) {
      unsigned int finite = 0u;
      if (vec && v0 + 32 <= n) {
        float4 x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          x[q] = (bits >> (4 * q)) & 15u ? __ldg(reinterpret_cast<const float4*>(cube + v0) + q)
                                         : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int q = 0; q < 8; ++q)
          finite |= ((isfinite(x[q].x) ? 1u : 0u) | (isfinite(x[q].y) ? 2u : 0u) | (isfinite(x[q].z) ? 4u : 0u) |
                     (isfinite(x[q].w) ? 8u : 0u))
                    << (4 * q);
      } else {
        for (int i = 0; i < 32; ++i)
          if ((bits >> i) & 1u) finite |= (isfinite(__ldg(cube + v0 + i)) ? 1u : 0u) << i;
      }
      bits &= finite;
    }
    mbits[w] = bits;
  }
}
// The same for a 16-bit cube (finiteness of the decoded value).
__global__ void k_pack16(const uint8_t* __restrict__ m8, Half16 h, long long plane, long long n,
                         uint32_t* __restrict__ mbits) {
  const long long nw = (n + 31) / 32;
  const bool vec = (reinterpret_cast<uintptr_t>(m8) & 15u) == 0u;
  for (long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x; w < nw; w += (long long)gridDim.x * blockDim.x) {
    const long long v0 = w * 32;
    const long long z0 = v0 / plane, next = (z0 + 1) * plane;
    unsigned int bits = 0u;
    for (unsigned int t = mask_word(m8, n, v0, vec); t; t &= t - 1u) {
      const int i = __ffs(t) - 1;
      const float cs = __ldg(h.scale + (v0 + i >= next ? z0 + 1 : z0));
      if (isfinite(half16_value(__ldg(h.bits + v0 + i), h.fmt, cs))) bits |= 1u << i;
    }
    mbits[w] = bits;
  }
}

cudaError_t launch_pack16(const uint8_t* m8, const Half16& h, long long plane, long long n, uint32_t* mbits,
                          cudaStream_t s) {
  long long nw = (n + 31) / 32;
  long long want = (nw + 255) / 256;
  int grid = (int)(want < 1 ? 1 : (want > 4096 ? 4096 : want));
  k_pack16<<<grid, 256, 0, s>>>(m8, h, plane, n, mbits);
  return cudaGetLastError();
}

cudaError_t launch_pack(const uint8_t* m8, const float* cube, long long n, uint32_t* mbits, cudaStream_t s) {
  long long nw = (n + 31) / 32;
  long long want = (nw + 255) / 256;
  int grid = (int)(want < 1 ? 1 : (want > 4096 ? 4096 : want));
  k_pack<<<grid, 256, 0, s>>>(m8, cube, n, mbits);
  return cudaGetLastError();
}

// uint8 mask from the working mask; with keep, OR-ed into the caller's mask
// (whose set voxels at non-finite values the working mask does not hold).
__global__ void k_expand(const uint32_t* __restrict__ mbits, long long n, uint8_t* __restrict__ m8, int keep) {
  // each thread writes 16 bytes
  const bool vec = ((reinterpret_cast<uintptr_t>(m8) & 15u) == 0);
  const long long ng = (n + 15) / 16;
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += (long long)gridDim.x * blockDim.x) {
    const long long v0 = g * 16;
    const unsigned int w = __ldg(mbits + (v0 >> 5)) >> (v0 & 31);
    if (vec && v0 + 16 <= n) {
      uint4 o = keep ? *reinterpret_cast<const uint4*>(m8 + v0) : make_uint4(0u, 0u, 0u, 0u);
      unsigned int* po = &o.x;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        unsigned int b = 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) b |= ((w >> (4 * q + i)) & 1u) << (8 * i);
        // 0x01 in every byte of the caller's word that is non-zero
        const unsigned int t = po[q];
        const unsigned int nz = ((((t & 0x7f7f7f7fu) + 0x7f7f7f7fu) | t) >> 7) & 0x01010101u;
        po[q] = keep ? (b | nz) : b;
      }
      *reinterpret_cast<uint4*>(m8 + v0) = o;
    } else {
      for (int i = 0; i < 16 && v0 + i < n; ++i)
        m8[v0 + i] = (uint8_t)((((w >> i) & 1u) != 0u || (keep && m8[v0 + i] != 0)) ? 1u : 0u);
    }
  }
}
cudaError_t launch_expand(const uint32_t* mbits, long long n, uint8_t* m8, int keep, cudaStream_t s) {
  long long ng = (n + 15) / 16;
  long long want = (ng + 255) / 256;
  int grid = (int)(want < 1 ? 1 : (want > 8192 ? 8192 : want));
  k_expand<<<grid, 256, 0, s>>>(mbits, n, m8, keep);
  return cudaGetLastError();
}

void init_noise_attrs() {
  cudaFuncSetAttribute(k_plan, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)((kNumBins + 1) * sizeof(unsigned long long)));
  cudaFuncSetAttribute(k_pass2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kP2Smem);
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_clip_full, 256, 0) != cudaSuccess) {
    cudaGetLastError();
    b = 0;
  }
  if (b > 0) g_clip_blocks_per_sm.store(b, std::memory_order_relaxed);
}

}  // namespace sc
