// Auto-flagger (SoFiA 2 Sect. 4.1): channels and spatial pixels whose noise
// deviates from the median noise across all channels / pixels by more than k
// times the MAD-based RMS are blanked.
//
//   k_chan_sample, k_chan_pass, k_chan_select
//                  the median and MAD of every channel's plane: a sample of
//                  the plane brackets the wanted rank, a pass over the whole
//                  cube counts each plane's values under its bracket and
//                  copies those inside, and a block per channel finds the
//                  rank among the copies (twice: values, then |x - m|)
//                  (and the Gaussian fit, over the plane once more)
//   k_chan_noise   one block per channel, the plane streamed from memory: STD
//                  by compensated sums, and (small planes, or no room for the
//                  copies) median and MAD by radix passes
//   k_pix_noise    one block per 16 pixels of a row: their spectra staged in
//                  shared memory, each pixel's noise by one warp (exact
//                  selections by a histogram of 256 equal steps between the
//                  smallest and the largest value)
//   k_array_stats  (sc_select.cu) median M and MAD-based RMS R of a noise array
//   k_flag         flags: |noise - M| > k R
//   k_blank        out = NaN on flagged channels and pixels, else in
//
// The noises are kept in float32; M, R and the flag test are in double.
#include <cfloat>
#include <cstdint>

#include "sc_device.cuh"
#include "sc_gaussfit.cuh"
#include "sc_internal.h"

namespace sc {
namespace flag {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kBins = 2048;
constexpr unsigned kNone = 0xffffffffu;

struct Scratch {
  unsigned hist[kBins];
  unsigned part[kWarps + 1];
  unsigned digit, rank, next, count;
  double dpart[kWarps + 1];
};

__device__ __forceinline__ void hist_add_warp(unsigned* hist, unsigned bin) {
  const unsigned peers = __match_any_sync(0xffffffffu, bin);
  if ((threadIdx.x & 31) == __ffs(peers) - 1 && bin < (unsigned)kBins) atomicAdd(&hist[bin], __popc(peers));
}

__device__ __forceinline__ unsigned block_scan_incl(unsigned v, unsigned* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  if (lane == 31) part[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const unsigned w = part[lane];
    unsigned wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += t;
    }
    part[lane] = wi - w;
  }
  __syncthreads();
  return part[warp] + x;
}

__device__ __forceinline__ double block_sum_d(double v, double* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) part[warp] = v;
  __syncthreads();
  if (warp == 0) {
    double t = lane < kWarps ? part[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) part[32] = t;
  }
  __syncthreads();
  const double r = part[32];
  __syncthreads();
  return r;
}

// |x - m| of the median m = (a + b) / 2 (a == b for an odd count), faithfully
// rounded (correctly for an odd count): -m = h + l exactly (a TwoSum of the
// halves; l is 0 for an odd count), then x + h as a sum and its error, to which
// l is added. NaN where x + h overflows.
struct Deviation {
  float h, l;
  __device__ __forceinline__ float operator()(float x) const {
    float e;
    const float t = two_sum(x, h, &e);
    return fabsf(__fadd_rn(t, __fadd_rn(e, l)));
  }
};
__device__ __forceinline__ Deviation deviation_of(float a, float b) {
  Deviation d{-a, 0.0f};
  if (a != b) d.h = two_sum(-0.5f * a, -0.5f * b, &d.l);
  return d;
}
// Its key (an overflow the largest).
__device__ __forceinline__ unsigned deviation_key(const Deviation& dev, float x) {
  const float d = dev(x);
  return fkey(d == d ? d : INFINITY);
}

// Order statistic `rank` (and, with want_next, rank + 1) of key_of(x) over
// the finite values x of src[0 .. n), streamed from memory: radix digits of
// 11, 11 and 10 bits counted in a shared histogram. All threads call it.
template <class KeyOf>
__device__ unsigned stream_select(const float* __restrict__ src, long long n, unsigned rank, KeyOf key_of,
                                  Scratch* S, bool want_next, unsigned* next) {
  const int tid = threadIdx.x, lane = tid & 31;
  unsigned prefix = 0u, pmask = 0u;
  for (int round = 0; round < 3; ++round) {
    const int shift = round == 0 ? 21 : (round == 1 ? 10 : 0);
    const unsigned dmask = round == 2 ? 0x3ffu : 0x7ffu;
    for (int i = tid; i < kBins; i += kThreads) S->hist[i] = 0u;
    __syncthreads();
    for (long long base = tid - lane; base < n; base += kThreads) {
      const long long i = base + lane;
      const float x = i < n ? __ldg(src + i) : __int_as_float(0x7fc00000);
      const unsigned k = isfinite(x) ? key_of(x) : kNone;
      hist_add_warp(S->hist, (k != kNone && (k & pmask) == prefix) ? (k >> shift) & dmask : (unsigned)kBins);
    }
    __syncthreads();
    const unsigned a = S->hist[2 * tid], b = S->hist[2 * tid + 1];
    const unsigned incl = block_scan_incl(a + b, S->part);
    const unsigned excl = incl - a - b;
    if (rank >= excl && rank < excl + a) {
      S->digit = 2u * tid;
      S->rank = rank - excl;
    } else if (rank >= excl + a && rank < incl) {
      S->digit = 2u * tid + 1u;
      S->rank = rank - excl - a;
    }
    __syncthreads();
    const unsigned d = S->digit;
    rank = S->rank;
    prefix |= d << shift;
    pmask |= dmask << shift;
    if (round == 2 && want_next) {
      if (tid == 0) S->next = (rank + 1u < S->hist[d]) ? prefix : kNone;
      __syncthreads();
      if (S->next == kNone) {
        for (int i = (int)d + 1 + tid; i < 1024; i += kThreads)
          if (S->hist[i] != 0u) atomicMin(&S->next, (prefix & ~dmask) | (unsigned)i);
        __syncthreads();
        if (S->next == kNone) {
          for (long long i = tid; i < n; i += kThreads) {
            const float x = __ldg(src + i);
            if (isfinite(x)) {
              const unsigned k = key_of(x);
              if (k > prefix) atomicMin(&S->next, k);
            }
          }
          __syncthreads();
        }
      }
      *next = S->next;
    }
    __syncthreads();
  }
  return prefix;
}

// Gaussian-fit noise of the finite values of src[0 .. n) with MAD noise
// sigma_mad > 0: the 256-bin histogram, then the fit (the MAD noise stands
// without a root). All threads call it.
__device__ double block_gauss(const float* __restrict__ src, long long n, double sigma_mad, Scratch* S) {
  const int tid = threadIdx.x, lane = tid & 31;
  const float k = gfit::scale_of(sigma_mad);
  __syncthreads();  // the selection is done with S->hist
  for (int i = tid; i < gfit::kBins; i += kThreads) S->hist[i] = 0u;
  __syncthreads();
  for (long long i = tid; i < n; i += kThreads) {
    const int b = gfit::bin_of(__ldg(src + i), k);
    if (b >= 0) atomicAdd(&S->hist[b], 1u);
  }
  __syncthreads();
  // one warp fits (four folded bins a lane, no block barriers); the others wait
  if (tid < 32) {
    const double tau = gfit::fit_tau_warp(S->hist);
    if (lane == 0) S->dpart[0] = tau;
  }
  __syncthreads();
  const double tau = S->dpart[0];
  __syncthreads();
  return tau > 0.0 ? gfit::noise_of(tau, k) : sigma_mad;
}

// Noise of the finite values of src[0 .. n) (NaN if none) in the S+C sense
// (mode SC_NOISE_MAD, _STD or _GAUSS); for MAD mode also the median m (the
// stats kernel needs it). All threads call it and get the same values.
__device__ void block_noise(const float* __restrict__ src, long long n, int mode, Scratch* S, double* sigma,
                            double* median) {
  const bool std_mode = mode == SC_NOISE_STD;
  const int tid = threadIdx.x, lane = tid & 31;
  // finite count
  unsigned c = 0u;
  for (long long i = tid; i < n; i += kThreads) c += isfinite(__ldg(src + i)) ? 1u : 0u;
  c = __reduce_add_sync(0xffffffffu, c);
  if (tid == 0) S->count = 0u;
  __syncthreads();
  if (lane == 0) atomicAdd(&S->count, c);
  __syncthreads();
  const unsigned nf = S->count;
  __syncthreads();
  if (nf == 0u) {
    *sigma = __longlong_as_double(0x7ff8000000000000LL);
    *median = *sigma;
    return;
  }
  if (std_mode) {
    float s = 0.0f, sc = 0.0f;
    for (long long i = tid; i < n; i += kThreads) {
      const float x = __ldg(src + i);
      if (isfinite(x)) neumaier_add(&s, &sc, x);
    }
    const double mean = block_sum_d((double)s + (double)sc, S->dpart) / (double)nf;
    const float mh = __double2float_rn(mean), ml = __double2float_rn(mean - (double)mh);
    float q = 0.0f, qc = 0.0f;
    for (long long i = tid; i < n; i += kThreads) {
      const float x = __ldg(src + i);
      if (isfinite(x)) {
        const float d = __fsub_rn(__fsub_rn(x, mh), ml);
        neumaier_add(&q, &qc, __fmul_rn(d, d));
      }
    }
    const double qq = block_sum_d((double)q + (double)qc, S->dpart);
    *sigma = nf > 1u ? sqrt(qq / (double)(nf - 1u)) : 0.0;
    *median = mean;
    return;
  }
  const unsigned r1 = (nf - 1u) / 2u;
  const bool even = (nf & 1u) == 0u;
  unsigned k2 = 0u;
  const unsigned k1 = stream_select(src, n, r1, [](float x) { return fkey(x); }, S, even, &k2);
  const float ma = fkey_inv(k1), mb = even ? fkey_inv(k2) : ma;
  const Deviation dev = deviation_of(ma, mb);
  unsigned a2 = 0u;
  const unsigned a1 =
      stream_select(src, n, r1, [=](float x) { return deviation_key(dev, x); }, S, even, &a2);
  const double mad = even ? 0.5 * ((double)fkey_inv(a1) + (double)fkey_inv(a2)) : (double)fkey_inv(a1);
  *sigma = kMadToSigma * mad;
  *median = even ? 0.5 * ((double)ma + (double)mb) : (double)ma;
  if (mode == SC_NOISE_GAUSS && *sigma > 0.0) *sigma = block_gauss(src, n, *sigma, S);
}

// ---- per-pixel noise: a warp per pixel ---------------------------------------
//
// What bounds it: instruction issue, with the loads of a tile before it (two
// blocks an SM hide each other's). Of 600 x 600 x 1024 voxels, the form with
// the spectrum in registers, 32 rounds of bisection for each of the four order
// statistics and one block of 8 warps an SM took 7.97 ms; this one 1.60 ms.
constexpr int kPixTile = 16;         // pixels of a row (64 bytes of each plane), a warp each
constexpr int kPixThreads = 32 * kPixTile;
constexpr int kPixPitch = kPixTile + 1;
constexpr int kSteps = 256;          // counts per warp (also the Gaussian fit's bins)
constexpr int kPixUnroll = 8;
static_assert(kSteps == gfit::kBins, "one set of counts serves both");

// f(value, its place) for a spectrum in shared memory; the lanes past its end
// get NaN. All lanes of the warp call f together.
template <class F>
__device__ __forceinline__ void for_spectrum(float* col, int nz, F f) {
  const int lane = threadIdx.x & 31;
  for (int z0 = 0; z0 < nz; z0 += 32 * kPixUnroll) {
    float v[kPixUnroll];
#pragma unroll
    for (int u = 0; u < kPixUnroll; ++u) {
      const int z = z0 + 32 * u + lane;
      v[u] = z < nz ? col[z * kPixPitch] : __int_as_float(0x7fc00000);
    }
#pragma unroll
    for (int u = 0; u < kPixUnroll; ++u) f(v[u], col + (z0 + 32 * u + lane) * kPixPitch);
  }
}

// Order statistic `rank` of a spectrum's values of(v) that are not NaN, by
// bisection on the 32-bit key.
template <class Of>
__device__ __noinline__ float warp_bisect(float* col, int nz, Of of, unsigned rank) {
  unsigned ans = 0u;
  for (int bit = 31; bit >= 0; --bit) {
    const unsigned t = ans | (1u << bit);
    unsigned c = 0u;
    for_spectrum(col, nz, [&](float x, float*) {
      const float v = of(x);
      c += (v == v && fkey(v) < t) ? 1u : 0u;
    });
    c = __reduce_add_sync(0xffffffffu, c);
    if (c <= rank) ans = t;
  }
  return fkey_inv(ans);
}

// Order statistics rank and (want_next) rank + 1 of a spectrum's values of(v)
// that are not NaN, all in [lo, hi] (both finite). counts: kSteps of shared
// memory, list: 32 floats. 256 equal steps of the range (rounded to the
// nearest, a monotone function of the value) are counted; the values of the
// rank's step are ranked directly, or, more than 32 of them, their smallest
// and largest become the next range. A range too small to divide: by bisection.
// first(v, place) is what the first count takes as of(v) (it may also replace
// the value in shared memory by that).
template <class Of, class First>
__device__ __forceinline__ void warp_select(float* col, int nz, Of of, First first, float lo, float hi, unsigned rank,
                                            bool want_next, unsigned* counts, float* list, float* v1, float* v2) {
  const unsigned lane = threadIdx.x & 31u;
  unsigned r = rank, cnt = kNone;  // rank in the range, and its values (at first: all)
  float found = lo;
  bool counted = false;
  while (lo < hi) {
    // halves, so that hi - lo cannot overflow; the step is in the low bits of
    // a sum with 1.5 * 2^23
    const float magic = 12582912.0f, h0 = -0.5f * lo, inv = (float)(kSteps - 1) / (0.5f * hi + h0);
    if (!(inv <= FLT_MAX)) {
      if (!counted) for_spectrum(col, nz, [&](float x, float* at) { first(x, at); });
      __syncwarp();
      *v1 = warp_bisect(col, nz, of, rank);
      *v2 = want_next ? warp_bisect(col, nz, of, rank + 1u) : *v1;
      return;
    }
    const auto step = [&](float v) { return __float_as_uint(__fmaf_rn(__fmaf_rn(v, 0.5f, h0), inv, magic)) & 0xffu; };
#pragma unroll
    for (int j = 0; j < kSteps / 128; ++j)
      reinterpret_cast<uint4*>(counts)[j * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    if (!counted) {
      for_spectrum(col, nz, [&](float x, float* at) {
        const float v = first(x, at);
        if (v >= lo && v <= hi) atomicAdd(counts + step(v), 1u);  // (false for NaN)
      });
    } else {
      for_spectrum(col, nz, [&](float x, float*) {
        const float v = of(x);
        if (v >= lo && v <= hi) atomicAdd(counts + step(v), 1u);
      });
    }
    counted = true;
    __syncwarp();
    const uint4 c0 = reinterpret_cast<const uint4*>(counts)[2 * lane];
    const uint4 c1 = reinterpret_cast<const uint4*>(counts)[2 * lane + 1];
    const unsigned c[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
    unsigned sum = 0u;
#pragma unroll
    for (int j = 0; j < 8; ++j) sum += c[j];
    unsigned x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (unsigned)o) x += y;
    }
    unsigned run = x - sum, d = 0u, in = 0u;
    const bool mine = r >= run && r < x;
    cnt = 0u;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (r >= run && r < run + c[j]) {
        d = 8u * lane + j;
        in = r - run;
        cnt = c[j];
      }
      run += c[j];
    }
    const int from = __ffs(__ballot_sync(0xffffffffu, mine)) - 1;  // (the range holds the rank)
    d = __shfl_sync(0xffffffffu, d, from);
    r = __shfl_sync(0xffffffffu, in, from);
    cnt = __shfl_sync(0xffffffffu, cnt, from);
    if (cnt <= 32u) {
      unsigned n = 0u;
      for_spectrum(col, nz, [&](float xv, float*) {
        const float v = of(xv);
        const bool take = v >= lo && v <= hi && step(v) == d;
        const unsigned b = __ballot_sync(0xffffffffu, take);
        if (take) list[n + __popc(b & ((1u << lane) - 1u))] = v;
        n += __popc(b);
      });
      __syncwarp();
      const float a = lane < cnt ? list[lane] : 0.0f;
      unsigned k = 0u;
      for (unsigned j = 0; j < cnt; ++j) {
        const float o = list[j];
        k += (o < a || (o == a && j < lane)) ? 1u : 0u;
      }
      __syncwarp();
      found = __shfl_sync(0xffffffffu, a, __ffs(__ballot_sync(0xffffffffu, lane < cnt && k == r)) - 1);
      if (want_next && r + 1u < cnt) {
        *v1 = found;
        *v2 = __shfl_sync(0xffffffffu, a, __ffs(__ballot_sync(0xffffffffu, lane < cnt && k == r + 1u)) - 1);
        return;
      }
      break;
    }
    unsigned kmin = kNone, kmax = 0u;
    for_spectrum(col, nz, [&](float xv, float*) {
      const float v = of(xv);
      if (v >= lo && v <= hi && step(v) == d) {
        kmin = min(kmin, fkey(v));
        kmax = max(kmax, fkey(v));
      }
    });
    found = lo = fkey_inv(__reduce_min_sync(0xffffffffu, kmin));
    hi = fkey_inv(__reduce_max_sync(0xffffffffu, kmax));
  }
  // found: ranked, or the only value of its range
  *v1 = *v2 = found;
  if (!want_next || r + 1u < cnt) return;
  // the rank was the last of its step or range: the next larger value
  unsigned above = kNone;
  for_spectrum(col, nz, [&](float xv, float*) {
    const float v = of(xv);
    if (v > found) above = min(above, fkey(v));
  });
  *v2 = fkey_inv(__reduce_min_sync(0xffffffffu, above));
}

// ---- per-channel median and MAD by passes over the whole cube ---------------
//
// What bounds it: the two passes' reads of the cube. On 600 x 600 x 1024
// voxels the form with one block per channel (seven passes over each plane by
// 304 blocks, whose planes do not fit L2 together, and a match_any histogram
// per value) took 11.3 ms; these kernels take 0.92 ms.
constexpr int kChanSample = 4096;         // values sampled per plane, four a thread
constexpr long long kChanMinPlane = 1LL << 15;  // smaller planes: one block streams them as fast
constexpr int kPassThreads = 256;
constexpr int kPassWarps = kPassThreads / 32;
constexpr int kPassRun = 1024;            // consecutive values a warp takes
constexpr int kFew = 1024;                // copies ranked directly

// A channel's bracket [lo, hi] of the wanted rank and what a pass found.
struct Chan {
  float lo, hi;
  unsigned finite, below, n;  // finite values, those under lo, copies (may exceed the room)
  Deviation dev;              // |x - m| of the median
};

// The digits whose cumulative ranges in S->hist hold ranks ra and rb, and the
// ranks within them.
__device__ __forceinline__ void find_two(Scratch* S, unsigned ra, unsigned rb, unsigned* da, unsigned* db,
                                         unsigned* ia) {
  const unsigned tid = threadIdx.x;
  __syncthreads();
  const unsigned a = S->hist[2 * tid], b = S->hist[2 * tid + 1];
  const unsigned incl = block_scan_incl(a + b, S->part), excl = incl - a - b;
  if (ra >= excl && ra < incl) {
    const bool in_a = ra < excl + a;
    S->digit = 2u * tid + (in_a ? 0u : 1u);
    S->rank = ra - excl - (in_a ? 0u : a);
  }
  if (rb >= excl && rb < incl) S->next = 2u * tid + (rb < excl + a ? 0u : 1u);
  __syncthreads();
  *da = S->digit;
  *db = S->next;
  *ia = S->rank;
  __syncthreads();
}

// Bracket of the median of of(x) over the plane, from a sample at a fixed step
// (each place moved a little, against patterns in the plane): sample ranks p
// +- 4 binomial standard deviations, located by the top 11 bits of the keys
// and then by 2048 equal steps between. Any bracket is checked by the pass's
// counts. kShift: key bits under a digit (keys below 2^(11 + kShift)).
template <int kShift, class Of, class Key>
__device__ void plane_bracket(const float* __restrict__ src, long long n, Of of, Key key, Scratch* S, float* lo,
                              float* hi) {
  const unsigned tid = threadIdx.x;
  const long long step = n / kChanSample;
  float v[4];
  unsigned c = 0u;
  for (int i = tid; i < kBins; i += kThreads) S->hist[i] = 0u;
  if (tid == 0u) S->count = 0u;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const unsigned j = u * kThreads + tid;
    v[u] = __ldg(src + j * step + ((unsigned long long)(j * 2654435761u) * (unsigned long long)step >> 32));
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const bool ok = isfinite(v[u]);
    v[u] = ok ? of(v[u]) : __int_as_float(0x7fc00000);
    if (ok) {
      ++c;
      atomicAdd(&S->hist[min(key(v[u]) >> kShift, (unsigned)kBins - 1u)], 1u);
    }
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if ((tid & 31u) == 0u) atomicAdd(&S->count, c);
  __syncthreads();
  const unsigned ns = S->count;
  *lo = -FLT_MAX;
  *hi = FLT_MAX;
  if (ns < 64u) return;
  const unsigned p = (ns - 1u) / 2u, delta = 2u * (unsigned)sqrtf((float)ns) + 4u;
  const unsigned ra = p > delta ? p - delta : 0u, rb = min(p + delta, ns - 1u);
  unsigned da, db, ia;
  find_two(S, ra, rb, &da, &db, &ia);
  const float a = fminf(fmaxf(key.value(da << kShift), -FLT_MAX), FLT_MAX);
  const float b = fminf(fmaxf(key.value((db << kShift) | ((1u << kShift) - 1u)), -FLT_MAX), FLT_MAX);
  *lo = a;
  *hi = b;
  const float inv = (float)kBins / (b - a);
  if (!(inv > 0.0f && isfinite(inv))) return;
  for (int i = tid; i < kBins; i += kThreads) S->hist[i] = 0u;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u)
    if (v[u] >= a && v[u] <= b) atomicAdd(&S->hist[min(kBins - 1, (int)((v[u] - a) * inv))], 1u);
  // the ranks among the values from the first digit on
  find_two(S, ia, ia + (rb - ra), &da, &db, &ia);
  const float w = (b - a) / (float)kBins;
  *lo = fmaxf(a, a + (float)da * w);
  *hi = fminf(b, a + (float)(db + 1u) * w);
}

// Order statistics r and (want_next) r + 1 among the n copies in list (all in
// [lo, hi], more than r of them). False (uniformly) when the step of the rank
// holds too many, or the next one lies beyond the copies.
__device__ bool list_select(const float* __restrict__ list, unsigned n, float lo, float hi, unsigned r, bool want_next,
                            Scratch* S, float* few, float* v1, float* v2) {
  const unsigned tid = threadIdx.x, lane = tid & 31u;
  const float inv = (float)kBins / (hi - lo);  // a step is a monotone function of the value
  const auto digit = [&](float v) { return (unsigned)min(kBins - 1, (int)((v - lo) * inv)); };
  for (int i = tid; i < kBins; i += kThreads) S->hist[i] = 0u;
  if (tid == 0u) S->count = 0u;
  __syncthreads();
  for (unsigned i = tid; i < n; i += kThreads) atomicAdd(&S->hist[digit(list[i])], 1u);
  unsigned d, d2, rr;
  find_two(S, r, r, &d, &d2, &rr);
  const unsigned cnt = S->hist[d];
  if (tid == 0u) S->next = kNone;
  __syncthreads();
  const bool many = cnt > (unsigned)kFew;
  unsigned above = kNone, kmin = kNone, kmax = 0u;
  for (unsigned i = tid; i < n; i += kThreads) {
    const float v = list[i];
    const unsigned dv = digit(v);
    if (dv == d) {
      kmin = min(kmin, fkey(v));
      kmax = max(kmax, fkey(v));
      if (!many) few[atomicAdd(&S->count, 1u)] = v;
    } else if (dv > d) {
      above = min(above, fkey(v));
    }
  }
  above = __reduce_min_sync(0xffffffffu, above);
  if (lane == 0u) atomicMin(&S->next, above);
  if (tid == 0u) {
    S->digit = kNone;
    S->rank = 0u;
  }
  __syncthreads();
  if (many) {  // ties? one value in the whole step is the answer
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0u) {
      atomicMin(&S->digit, kmin);
      atomicMax(&S->rank, kmax);
    }
    __syncthreads();
    const bool same = S->digit == S->rank;
    *v1 = *v2 = fkey_inv(S->digit);
    if (want_next && rr + 1u >= cnt) *v2 = fkey_inv(S->next);
    const bool ok = same && (!want_next || rr + 1u < cnt || S->next != kNone);
    __syncthreads();
    return ok;
  }
  if (tid < cnt) {
    const float v = few[tid];
    unsigned k = 0u;  // its rank in the step, ties in the order of the list
    for (unsigned j = 0; j < cnt; ++j) {
      const float o = few[j];
      k += (o < v || (o == v && j < tid)) ? 1u : 0u;
    }
    if (k == rr) S->digit = fkey(v);
    if (k == rr + 1u) S->rank = fkey(v);
  }
  __syncthreads();
  const unsigned k1 = S->digit, k2 = rr + 1u < cnt ? S->rank : S->next;
  __syncthreads();
  *v1 = fkey_inv(k1);
  *v2 = want_next ? fkey_inv(k2) : *v1;
  return !want_next || k2 != kNone;
}

}  // namespace flag

// A block per channel: the bracket of its median.
__global__ void __launch_bounds__(flag::kThreads, 1)
    k_chan_sample(const float* __restrict__ cube, long long plane, flag::Chan* ch) {
  using namespace flag;
  __shared__ Scratch S;
  float lo, hi;
  plane_bracket<21>(cube + (long long)blockIdx.x * plane, plane, [](float x) { return x; }, KeyOfValue{}, &S, &lo, &hi);
  if (threadIdx.x == 0) ch[blockIdx.x] = Chan{lo, hi, 0u, 0u, 0u, Deviation{0.0f, 0.0f}};
}

// A pass over the cube: the values (DEV: their |x - m|) of every channel under
// its bracket counted and those inside copied to its list. A warp takes runs
// of kPassRun consecutive values of a plane, its copies staged in shared memory.
template <bool DEV>
__global__ void __launch_bounds__(flag::kPassThreads, 4)
    k_chan_pass(const float* __restrict__ cube, long long plane, int nz, flag::Chan* ch, float* __restrict__ lists,
                long long room) {
  using namespace flag;
  __shared__ float stage[kPassWarps][kPassRun];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long runs = (plane + kPassRun - 1) / kPassRun, total = runs * nz;
  const long long warps = (long long)gridDim.x * kPassWarps;
  const bool vec = (plane & 3) == 0 && (reinterpret_cast<uintptr_t>(cube) & 15u) == 0;
  constexpr int kQ = kPassRun / 128;  // float4 loads a lane makes per run
  for (long long it = (long long)blockIdx.x * kPassWarps + warp; it < total; it += warps) {
    const int z = (int)(it / runs);
    const long long p0 = (it - z * runs) * kPassRun;
    const float* src = cube + z * plane + p0;
    const int left = (int)min((long long)kPassRun, plane - p0);
    const float lo = ch[z].lo, hi = ch[z].hi;
    const Deviation dev = ch[z].dev;
    float v[kQ][4];
    if (vec && left == kPassRun) {
#pragma unroll
      for (int q = 0; q < kQ; ++q) {
        const float4 f = __ldg(reinterpret_cast<const float4*>(src) + 32 * q + lane);
        v[q][0] = f.x, v[q][1] = f.y, v[q][2] = f.z, v[q][3] = f.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < kQ; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int i = 128 * q + 32 * c + lane;
          v[q][c] = i < left ? __ldg(src + i) : __int_as_float(0x7fc00000);
        }
    }
    // every lane copies to its own column: room for all its values, no votes
    unsigned finite = 0u, below = 0u;
    int n = 0;
#pragma unroll
    for (int q = 0; q < kQ; ++q)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float a = v[q][c];
        const bool ok = fabsf(a) <= FLT_MAX;  // false for NaN and Inf
        if (DEV) a = dev(a);
        else finite += ok ? 1u : 0u;
        const bool under = ok && a < lo;
        below += under ? 1u : 0u;
        if (ok && !under && a <= hi) stage[warp][32 * n++ + lane] = a;
      }
    finite = __reduce_add_sync(0xffffffffu, finite);
    below = __reduce_add_sync(0xffffffffu, below);
    int x = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    unsigned at = 0u;
    if (lane == 31) {
      if (finite) atomicAdd(&ch[z].finite, finite);
      if (below) atomicAdd(&ch[z].below, below);
      if (x) at = atomicAdd(&ch[z].n, (unsigned)x);
    }
    at = __shfl_sync(0xffffffffu, at, 31) + (unsigned)(x - n);
    float* out = lists + z * room;
    for (int i = 0; i < n; ++i)
      if ((long long)at + i < room) out[at + i] = stage[warp][32 * i + lane];
  }
}

// A block per channel: the median from its copies, and the bracket of the MAD
// (DEV false); the MAD and the noise (DEV true). Without a usable bracket, by
// radix passes over the plane.
template <bool DEV>
__global__ void __launch_bounds__(flag::kThreads, 1)
    k_chan_select(const float* __restrict__ cube, long long plane, flag::Chan* ch, const float* __restrict__ lists,
                  long long room, int mode, float* __restrict__ noise) {
  using namespace flag;
  __shared__ Scratch S;
  __shared__ float few[kFew];
  const int z = blockIdx.x;
  const float* src = cube + (long long)z * plane;
  const Chan c = ch[z];
  if (c.finite == 0u) {  // no finite voxel: no noise (and no MAD pass to prepare)
    if (DEV && threadIdx.x == 0) noise[z] = __int_as_float(0x7fc00000);
    return;
  }
  const unsigned r1 = (c.finite - 1u) / 2u;
  const bool even = (c.finite & 1u) == 0u;
  float v1 = 0.0f, v2 = 0.0f;
  bool done = (long long)c.n <= room && r1 >= c.below && r1 - c.below < c.n && c.hi > c.lo;
  if (done) done = list_select(lists + z * room, c.n, c.lo, c.hi, r1 - c.below, even, &S, few, &v1, &v2);
  if (!done) {
    unsigned k2 = 0u;
    if (DEV) {
      const Deviation dev = c.dev;
      v1 = fkey_inv(stream_select(src, plane, r1, [=](float x) { return deviation_key(dev, x); }, &S, even, &k2));
    } else {
      v1 = fkey_inv(stream_select(src, plane, r1, [](float x) { return fkey(x); }, &S, even, &k2));
    }
    v2 = even ? fkey_inv(k2) : v1;
  }
  if (DEV) {
    const double mad = even ? 0.5 * ((double)v1 + (double)v2) : (double)v1;
    double sigma = kMadToSigma * mad;
    if (mode == SC_NOISE_GAUSS && sigma > 0.0) {
      __syncthreads();  // the selection is done with the scratch
      sigma = block_gauss(src, plane, sigma, &S);
    }
    if (threadIdx.x == 0) noise[z] = __double2float_rn(sigma);
  } else {
    float lo, hi;
    const Deviation dev = deviation_of(v1, v2);
    __syncthreads();
    plane_bracket<20>(src, plane, dev, KeyOfDev{}, &S, &lo, &hi);
    if (threadIdx.x == 0) ch[z] = Chan{fmaxf(lo, 0.0f), hi, c.finite, 0u, 0u, dev};
  }
}

__global__ void __launch_bounds__(flag::kThreads, 1)
    k_chan_noise(const float* __restrict__ cube, long long plane, int nz, int mode, float* __restrict__ noise) {
  __shared__ flag::Scratch S;
  for (int z = blockIdx.x; z < nz; z += gridDim.x) {
    double sigma, m;
    flag::block_noise(cube + (long long)z * plane, plane, mode, &S, &sigma, &m);
    if (threadIdx.x == 0) noise[z] = __double2float_rn(sigma);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(flag::kPixThreads, 2) k_pix_noise(const float* __restrict__ cube, int nx, int ny,
                                                                    int nz, int mode, float* __restrict__ noise) {
  using namespace flag;
  extern __shared__ __align__(16) float pix_smem[];
  // per warp 256 counts and 32 values, then the spectra: [nz][kPixPitch]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned* const counts = reinterpret_cast<unsigned*>(pix_smem) + warp * kSteps;
  float* const list = pix_smem + kPixTile * kSteps + warp * 32;
  float* const tile = pix_smem + kPixTile * (kSteps + 32);
  const long long plane = (long long)nx * ny;
  const int xtiles = (nx + kPixTile - 1) / kPixTile;
  const long long ntiles = (long long)xtiles * ny;
  for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int y = (int)(t / xtiles), x0 = (int)(t - (long long)y * xtiles) * kPixTile;
    __syncthreads();  // the tile of the previous iteration is consumed
    {
      // two planes a warp and load, eight loads ahead
      const int px = lane & (kPixTile - 1), x = x0 + px;
      const float* src = cube + (long long)y * nx + x;
      for (int z0 = 2 * warp + (lane >> 4); z0 < nz; z0 += 2 * kPixTile * 8) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int z = z0 + 2 * kPixTile * u;
          v[u] = (z < nz && x < nx) ? __ldg(src + (long long)z * plane) : __int_as_float(0x7fc00000);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int z = z0 + 2 * kPixTile * u;
          if (z < nz) tile[z * kPixPitch + px] = __fadd_rn(v[u], __fsub_rn(v[u], v[u]));  // Inf becomes NaN
        }
      }
    }
    __syncthreads();
    if (x0 + warp >= nx) continue;
    float* const col = tile + warp;
    unsigned nf = 0u;
    float mn = FLT_MAX, mx = -FLT_MAX;
    for_spectrum(col, nz, [&](float v, float*) {
      nf += v == v ? 1u : 0u;
      mn = fminf(mn, v);
      mx = fmaxf(mx, v);
    });
    nf = __reduce_add_sync(0xffffffffu, nf);
    float out;
    if (nf == 0u) {
      out = __int_as_float(0x7fc00000);
    } else if (mode == SC_NOISE_STD) {
      float s = 0.0f, sc = 0.0f;
      for_spectrum(col, nz, [&](float v, float*) {
        if (v == v) neumaier_add(&s, &sc, v);
      });
      double ds = (double)s + (double)sc;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ds += __shfl_xor_sync(0xffffffffu, ds, o);
      const double mean = ds / (double)nf;
      const float mh = __double2float_rn(mean), ml = __double2float_rn(mean - (double)mh);
      float q = 0.0f, qc = 0.0f;
      for_spectrum(col, nz, [&](float v, float*) {
        if (v == v) {
          const float d = __fsub_rn(__fsub_rn(v, mh), ml);
          neumaier_add(&q, &qc, __fmul_rn(d, d));
        }
      });
      double dq = (double)q + (double)qc;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dq += __shfl_xor_sync(0xffffffffu, dq, o);
      out = __double2float_rn(nf > 1u ? sqrt(dq / (double)(nf - 1u)) : 0.0);
    } else {
      mn = fkey_inv(__reduce_min_sync(0xffffffffu, fkey(mn)));
      mx = fkey_inv(__reduce_max_sync(0xffffffffu, fkey(mx)));
      const unsigned r1 = (nf - 1u) / 2u;
      const bool even = (nf & 1u) == 0u;
      float ma, mb, a1, a2;
      const auto same = [](float v) { return v; };
      warp_select(col, nz, same, [](float v, float*) { return v; }, mn, mx, r1, even, counts, list, &ma, &mb);
      const Deviation dev = deviation_of(ma, mb);
      // |v - m| in place of v (an overflow stays the largest), unless the fit
      // needs the values
      const bool keep = mode == SC_NOISE_GAUSS;
      const auto clamped = [&](float v) { return v == v ? fminf(dev(v), FLT_MAX) : v; };
      const float top = fmaxf(clamped(mn), clamped(mx));
      if (keep) {
        warp_select(col, nz, clamped, [&](float v, float*) { return clamped(v); }, 0.0f, top, r1, even, counts, list, &a1,
                    &a2);
      } else {
        const auto replace = [&](float v, float* at) {
          v = clamped(v);
          if (v == v) *at = v;
          return v;
        };
        warp_select(col, nz, same, replace, 0.0f, top, r1, even, counts, list, &a1, &a2);
      }
      const double mad = even ? 0.5 * ((double)a1 + (double)a2) : (double)a1;
      double sigma = kMadToSigma * mad;
      if (mode == SC_NOISE_GAUSS && sigma > 0.0) {
        // the spectrum's 256-bin histogram in this warp's counts, then a
        // warp-wide fit over the 128 folded bins (4 a lane)
        for (int i = lane; i < gfit::kBins; i += 32) counts[i] = 0u;
        __syncwarp();
        const float ks = gfit::scale_of(sigma);
        for_spectrum(col, nz, [&](float v, float*) {
          const int b = gfit::bin_of(v, ks);  // NaN gives -1
          if (b >= 0) atomicAdd(counts + b, 1u);
        });
        __syncwarp();
        const double tau = gfit::fit_tau_warp(counts);
        if (tau > 0.0) sigma = gfit::noise_of(tau, ks);
      }
      out = __double2float_rn(sigma);
    }
    if (lane == 0) noise[(long long)y * nx + x0 + warp] = out;
  }
}

__global__ void k_flag(const float* __restrict__ noise, long long n, const double* __restrict__ stats, double k,
                       uint8_t* __restrict__ flags) {
  const double m = stats[0], r = stats[1];
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float v = noise[i];
    flags[i] = (isfinite(v) && isfinite(m) && fabs((double)v - m) > k * r) ? 1 : 0;
  }
}

// A thread keeps its pixels (VEC: four, else one) and goes through kBlankRun
// planes, four loads ahead. HBM-bound: 8 bytes a voxel; with a 64-bit division
// and a 4-byte load and store per voxel 600 x 600 x 1024 voxels took 1.03 ms,
// now 0.42 ms. out may be in.
constexpr int kBlankRun = 16;
template <bool VEC>
__global__ void __launch_bounds__(256) k_blank(const float* in, float* out, long long plane, int nz,
                                               const uint8_t* __restrict__ fchan, const uint8_t* __restrict__ fpix) {
  constexpr int kW = VEC ? 4 : 1;
  const long long q = blockIdx.x * 256LL + threadIdx.x;
  if (q * kW >= plane) return;
  const float qnan = __int_as_float(0x7fc00000);
  bool pix[kW];
#pragma unroll
  for (int c = 0; c < kW; ++c) pix[c] = fpix && fpix[q * kW + c];
  for (long long z1 = blockIdx.y * (long long)kBlankRun; z1 < nz; z1 += gridDim.y * (long long)kBlankRun) {
    for (int z0 = 0; z0 < kBlankRun && z1 + z0 < nz; z0 += 4) {
      float v[4][kW];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const long long z = z1 + z0 + u;
        if (z >= nz) break;
        const float* src = in + z * plane + q * kW;
        if constexpr (VEC) {
          const float4 f = *reinterpret_cast<const float4*>(src);
          v[u][0] = f.x, v[u][1] = f.y, v[u][2] = f.z, v[u][3] = f.w;
        } else {
          v[u][0] = *src;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const long long z = z1 + z0 + u;
        if (z >= nz) break;
        const bool ch = fchan && __ldg(fchan + z);
#pragma unroll
        for (int c = 0; c < kW; ++c) v[u][c] = ch || pix[c] ? qnan : v[u][c];
        float* dst = out + z * plane + q * kW;
        if constexpr (VEC) *reinterpret_cast<float4*>(dst) = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
        else *dst = v[u][0];
      }
    }
  }
}

// ---------------------------------------------------------------------------
namespace {
cudaError_t launch_pix(const float* cube, int nx, int ny, int nz, int mode, float* noise, int sms, cudaStream_t s) {
  const size_t smem = sizeof(float) * (flag::kPixTile * (flag::kSteps + 32) + flag::kPixPitch * (size_t)nz);
  cudaFuncSetAttribute(k_pix_noise, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const long long tiles = (long long)((nx + flag::kPixTile - 1) / flag::kPixTile) * ny;
  const int grid = (int)(tiles < 8LL * sms ? tiles : 8LL * sms);
  k_pix_noise<<<grid, flag::kPixThreads, smem, s>>>(cube, nx, ny, nz, mode, noise);
  return cudaGetLastError();
}
}  // namespace

// Room for the copies of one plane: a bracket holds about 6 % of it.
static long long chan_room(long long plane) { return (plane / 8 + 4 + 3) & ~3LL; }

size_t chan_plane_bytes(const long long dims[3], int mode) {
  const long long plane = dims[0] * dims[1];
  if (mode == SC_NOISE_STD || plane < flag::kChanMinPlane || plane >= (1LL << 32)) return 0;
  return sizeof(float) * (size_t)chan_room(plane) + ((sizeof(flag::Chan) + 15) & ~(size_t)15);
}

// Channels [0, nz) in groups of `group`, whose copies and brackets lie in scratch.
static cudaError_t launch_chan_mad(const float* cube, long long plane, int nz, int mode, void* scratch, int group,
                                   float* noise, int sms, cudaStream_t s) {
  const long long room = chan_room(plane);
  float* const lists = static_cast<float*>(scratch);
  flag::Chan* const ch = reinterpret_cast<flag::Chan*>(lists + room * group);
  const long long runs = (plane + flag::kPassRun - 1) / flag::kPassRun;
  for (int z0 = 0; z0 < nz; z0 += group) {
    const int n = nz - z0 < group ? nz - z0 : group;
    const float* const part = cube + z0 * plane;
    const long long want = (runs * n + flag::kPassWarps - 1) / flag::kPassWarps;
    const int grid = (int)(want < 4LL * sms ? want : 4LL * sms);
    k_chan_sample<<<n, flag::kThreads, 0, s>>>(part, plane, ch);
    k_chan_pass<false><<<grid, flag::kPassThreads, 0, s>>>(part, plane, n, ch, lists, room);
    k_chan_select<false><<<n, flag::kThreads, 0, s>>>(part, plane, ch, lists, room, mode, noise + z0);
    k_chan_pass<true><<<grid, flag::kPassThreads, 0, s>>>(part, plane, n, ch, lists, room);
    k_chan_select<true><<<n, flag::kThreads, 0, s>>>(part, plane, ch, lists, room, mode, noise + z0);
  }
  return cudaGetLastError();
}

cudaError_t launch_autoflag(const float* cube, const long long dims[3], double k, int channels, int pixels,
                            int mode, float* out, float* chan_noise, float* pix_noise, uint8_t* chan_flags,
                            uint8_t* pix_flags, double* stats, void* chan_scratch, int chan_group, int sms,
                            cudaStream_t s) {
  const int nx = (int)dims[0], ny = (int)dims[1], nz = (int)dims[2];
  const long long plane = (long long)nx * ny;
  cudaError_t e = cudaSuccess;
  if (channels) {
    if (chan_group > 0) {
      e = launch_chan_mad(cube, plane, nz, mode, chan_scratch, chan_group, chan_noise, sms, s);
      if (e != cudaSuccess) return e;
    } else {
      k_chan_noise<<<nz < 2 * sms ? nz : 2 * sms, flag::kThreads, 0, s>>>(cube, plane, nz, mode, chan_noise);
    }
    if ((e = launch_array_stats(chan_noise, nz, stats, s)) != cudaSuccess) return e;
    k_flag<<<(nz + 255) / 256, 256, 0, s>>>(chan_noise, nz, stats, k, chan_flags);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (pixels) {
    e = launch_pix(cube, nx, ny, nz, mode, pix_noise, sms, s);
    if (e != cudaSuccess) return e;
    if ((e = launch_array_stats(pix_noise, plane, stats + 2, s)) != cudaSuccess) return e;
    const long long g = (plane + 255) / 256;
    k_flag<<<(unsigned)(g < 16LL * sms ? g : 16LL * sms), 256, 0, s>>>(pix_noise, plane, stats + 2, k, pix_flags);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  const uint8_t* const fc = channels ? chan_flags : nullptr;
  const uint8_t* const fp = pixels ? pix_flags : nullptr;
  const bool vec = plane % 4 == 0 && ((reinterpret_cast<uintptr_t>(cube) | reinterpret_cast<uintptr_t>(out)) & 15u) == 0;
  const long long bx = ((vec ? plane / 4 : plane) + 255) / 256, by = (nz + kBlankRun - 1) / kBlankRun;
  const dim3 grid((unsigned)bx, (unsigned)(by < 65535 ? by : 65535));
  if (vec) k_blank<true><<<grid, 256, 0, s>>>(cube, out, plane, nz, fc, fp);
  else k_blank<false><<<grid, 256, 0, s>>>(cube, out, plane, nz, fc, fp);
  return cudaGetLastError();
}

}  // namespace sc
