// Exact median and MAD of one noise measurement from its candidate lists
// (SoFiA 2, Sect. 4.1).
//
//   k_select       one thread-block cluster: radix rounds over the median's
//                  list (about 1e-4 of the values), then over the MAD's (0.7 %)
//   k_mad_digits,  long lists only: the MAD's first round by all SMs, and the
//   k_mad_compact  values of its digit copied into a short list
//
// A round counts up to 2048 digits in each block's shared memory; the blocks
// of a cluster add their counts up over distributed shared memory and all take
// the same pick. The plan gives the range of keys that holds the wanted order
// statistics (the median's bins, the MAD's bracket), so a round resolves 11
// bits of that range, not of the whole float: two rounds for noise-like data.
// Where both lists are short (kOneBlock) the first block does it alone.
//
// What bounds it: latency (a round's barriers and loads; the code itself,
// which every launch fetches once, hence one copy of the round for all forms
// of keys), and for long lists the instructions that form the keys. It took
// the place of ten launches over all SMs (three rounds, the successor and the
// result, for the median and for the MAD): the 12
// measurements of a run on a 64 x 64 x 128 cube took 0.99 ms of those, and take
// 0.26 ms now. Measurements whose lists would overflow (PLAN_*_FULL) keep the full passes
// of sc_noise.cu, which read the array with all SMs; in an array of at most
// kSelectAllMax values one cluster reads it as fast, and does that too.
#include <cooperative_groups.h>

#include <cfloat>

#include "sc_device.cuh"
#include "sc_internal.h"

namespace sc {
namespace select {

namespace cg = cooperative_groups;

constexpr int kThreads = 1024;
constexpr int kBins = kSelBins, kDigitBits = 11;
constexpr unsigned kOneBlock = 16384;   // lists up to this long: one block
constexpr int kUnroll = 4;              // loads in flight per thread
constexpr unsigned kNone = 0xffffffffu; // above every key of a finite value

// |s - m| of a median m = (a + b) / 2 as a correctly rounded float, without
// the slow float64 pipe: -m = h + l exactly (a TwoSum of the halves), then the
// sum of the three floats s, h and l, its tail rounded to odd (Boldo and
// Melquiond, "Emulation of FMA and correctly rounded sums", 2008). l == 0 (an
// odd count, or equal middle values): one addition. Halving a subnormal may
// round, so medians of tiny values take float64.
__device__ __forceinline__ AbsDev abs_dev_of(float a, float b) {
  AbsDev d;
  d.m = a == b ? (double)a : 0.5 * ((double)a + (double)b);
  const float tiny = 0x1p-100f;
  d.wide = a != b && ((a != 0.0f && fabsf(a) < tiny) || (b != 0.0f && fabsf(b) < tiny)) ? 1 : 0;
  d.l = 0.0f;
  d.h = a == b ? -a : two_sum(-0.5f * a, -0.5f * b, &d.l);
  return d;
}

__device__ __forceinline__ float abs_dev(float s, const AbsDev& d) {
  if (d.wide) return __double2float_rn(fabs((double)s - d.m));
  if (d.l == 0.0f) return fabsf(__fadd_rn(s, d.h));
  float e;
  const float t = two_sum(s, d.h, &e);
  float ve;
  float v = two_sum(e, d.l, &ve);
  // v rounded to odd: an inexact v with an even significand moves one step
  // towards the rest
  const unsigned vb = __float_as_uint(v);
  if (ve != 0.0f && !(vb & 1u)) v = __uint_as_float((ve > 0.0f) == (v > 0.0f) ? vb + 1u : vb - 1u);
  const float r = __fadd_rn(t, v);
  return fabsf(isfinite(t) ? r : t);
}

enum Form { FORM_VALUE, FORM_ABSDEV, FORM_KEY };

// Key of list element v; kNone for a non-finite value.
__device__ __forceinline__ unsigned key_of(int form, float v, const AbsDev& d) {
  if (form == FORM_KEY) return __float_as_uint(v);
  if (!isfinite(v)) return kNone;
  return form == FORM_VALUE ? fkey(v) : __float_as_uint(abs_dev(v, d)) | 0x80000000u;
}

// Adds one to the digit's count for every lane (kNone: nothing); a warp whose
// lanes share a digit (ties) adds once. All lanes call it.
__device__ __forceinline__ void count_digit(unsigned* hist, unsigned dig) {
  const unsigned d0 = __shfl_sync(0xffffffffu, dig, 0);
  if (__all_sync(0xffffffffu, dig == d0)) {
    if ((threadIdx.x & 31u) == 0u && dig != kNone) atomicAdd(&hist[dig], 32u);
  } else if (dig != kNone) {
    atomicAdd(&hist[dig], 1u);
  }
}

// Digit width of the first round over a range of keys.
__device__ __forceinline__ int first_shift(unsigned klo, unsigned khi) {
  const int bits = khi > klo ? 32 - __clz(khi - klo) : 0;
  return bits > kDigitBits ? bits - kDigitBits : 0;
}

struct Smem {
  unsigned hist[2][kBins];     // this block's counts of a round (the other one is clear)
  unsigned red[2][kBins / 2];  // the cluster's counts of this block's share of the digits
  unsigned below[2];           // this block's keys under the range
  unsigned part[kThreads / 32];
  unsigned digit, rank, count, next, found, total_below;
  unsigned k1, k2;             // the result
};

// What a selection reads: order statistics rank and (want_next) rank + 1 of
// the keys of list[0 .. count), the first of them in [klo, khi]. store: the
// first round writes the keys over the list. next: the smallest key above the
// list's, for a rank + 1 beyond it.
struct Task {
  float* list;
  unsigned long long count;
  unsigned rank, klo, khi, next;
  int form, store, want_next;
};

// The order statistics into S->k1, S->k2 of every block (all nc blocks of the
// cluster call it with all threads; nc == 1: the calling block alone). False
// when the counts contradict the rank.
__device__ __noinline__ bool select_rank(int nc, Task t, const AbsDev d, Smem* S) {
  cg::cluster_group cl = cg::this_cluster();
  const int me = nc > 1 ? (int)cl.block_rank() : 0;
  const unsigned tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const unsigned first = (unsigned)me * kThreads + tid, stride = (unsigned)nc * kThreads;
  for (unsigned i = tid; i < kBins; i += kThreads) S->hist[0][i] = S->hist[1][i] = 0u;
  if (nc > 1)
    for (unsigned i = tid; i < kBins / 2; i += kThreads) S->red[0][i] = S->red[1][i] = 0u;
  if (tid < 2u) S->below[tid] = 0u;
  __syncthreads();
  const unsigned share = kBins / nc;  // digits whose cluster-wide counts this block adds up
  int shift = first_shift(t.klo, t.khi);
  unsigned rank = t.rank, a, b;
  int par = 0;
#pragma unroll 1
  for (bool first_round = true;; first_round = false) {
    unsigned under = 0u;
#pragma unroll 1
    for (unsigned long long w0 = first - lane; w0 < t.count; w0 += (unsigned long long)kUnroll * stride) {
      float v[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const unsigned long long i = w0 + lane + (unsigned long long)u * stride;
        v[u] = i < t.count ? t.list[i] : __uint_as_float(kNone);
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const unsigned k = key_of(t.form, v[u], d);
        if (t.store) {
          const unsigned long long i = w0 + lane + (unsigned long long)u * stride;
          if (i < t.count) t.list[i] = __uint_as_float(k);
        }
        under += k < t.klo ? 1u : 0u;
        count_digit(S->hist[par], (k >= t.klo && k <= t.khi && k != kNone) ? (k - t.klo) >> shift : kNone);
      }
    }
    if (t.store) t.form = FORM_KEY;
    t.store = 0;
    under = __reduce_add_sync(0xffffffffu, under);
    if (lane == 0u && under) atomicAdd(&S->below[par], under);
    if (nc == 1) {
      __syncthreads();
      a = S->hist[par][2u * tid];
      b = S->hist[par][2u * tid + 1u];
      if (tid == 0u) S->total_below = S->below[par];
    } else {
      cl.sync();  // every block's counts are complete
      for (unsigned i = tid; i < kBins; i += kThreads) {
        const unsigned c = *cl.map_shared_rank(&S->hist[par][me * share + i % share], i / share);
        if (c) atomicAdd(&S->red[par][i % share], c);
      }
      cl.sync();  // every block's sums are complete
      a = *cl.map_shared_rank(&S->red[par][(2u * tid) % share], (2u * tid) / share);
      b = *cl.map_shared_rank(&S->red[par][(2u * tid + 1u) % share], (2u * tid + 1u) / share);
      if (warp == 0u) {
        unsigned s = lane < (unsigned)nc ? *cl.map_shared_rank(&S->below[par], lane) : 0u;
        s = __reduce_add_sync(0xffffffffu, s);
        if (lane == 0u) S->total_below = s;
      }
    }
    // the digit that holds the rank
    unsigned x = a + b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
      if ((int)lane >= o) x += y;
    }
    if (lane == 31u) S->part[warp] = x;
    if (tid == 0u) {
      S->found = 0u;
      S->next = kNone;
    }
    __syncthreads();
    const unsigned p = S->part[lane];
    unsigned excl = __reduce_add_sync(0xffffffffu, lane < warp ? p : 0u) + x - a - b;
    // later rounds' ranges start at a picked digit: nothing under them counts
    excl += first_round ? S->total_below : 0u;
    if (rank >= excl && rank < excl + a + b) {
      const bool in_a = rank < excl + a;
      S->digit = 2u * tid + (in_a ? 0u : 1u);
      S->rank = rank - excl - (in_a ? 0u : a);
      S->count = in_a ? a : b;
      S->found = 1u;
    }
    // the other buffers for the next round (their readers are past a barrier)
    for (unsigned i = tid; i < kBins; i += kThreads) S->hist[par ^ 1][i] = 0u;
    if (nc > 1)
      for (unsigned i = tid; i < kBins / 2; i += kThreads) S->red[par ^ 1][i] = 0u;
    if (tid == 0u) S->below[par ^ 1] = 0u;
    __syncthreads();
    if (S->found == 0u) {
      if (nc > 1) cl.sync();  // (no block leaves while another reads its counts)
      return false;
    }
    rank = S->rank;
    const unsigned digit = S->digit;
    if (shift == 0) {
      unsigned k2 = t.klo + digit;
      if (tid == 0u) S->k1 = k2;
      if (t.want_next && rank + 1u >= S->count) {
        // the next non-empty digit of this round
        if (a && 2u * tid > digit) atomicMin(&S->next, 2u * tid);
        else if (b && 2u * tid + 1u > digit) atomicMin(&S->next, 2u * tid + 1u);
        __syncthreads();
        const unsigned next = S->next;
        __syncthreads();  // every thread has read it before it is written again
        if (next != kNone) {
          k2 = t.klo + next;
        } else {
          // the smallest key above this round's range
          unsigned mn = kNone;
#pragma unroll 1
          for (unsigned long long i = first; i < t.count; i += stride) {
            const unsigned k = key_of(t.form, t.list[i], d);
            if (k > t.khi) mn = min(mn, k);
          }
          mn = __reduce_min_sync(0xffffffffu, mn);
          if (lane == 0u && mn != kNone) atomicMin(&S->next, mn);
          __syncthreads();
          k2 = min(t.next, S->next);
          if (nc > 1) {
            cl.sync();  // every block's minimum is complete
#pragma unroll 1
            for (int r = 0; r < nc; ++r) k2 = min(k2, *cl.map_shared_rank(&S->next, r));
          }
        }
      }
      if (tid == 0u) S->k2 = k2;
      __syncthreads();
      if (nc > 1) cl.sync();  // no block still reads another's counts
      return k2 != kNone;
    }
    const unsigned span = (1u << shift) - 1u;
    t.klo += digit << shift;
    t.khi = t.khi - t.klo < span ? t.khi : t.klo + span;
    shift = shift > kDigitBits ? shift - kDigitBits : 0;
    par ^= 1;
  }
}

}  // namespace select

// part: PART_ALL, or with the MAD's first round by all SMs in between,
// PART_MEDIAN and then PART_MAD. all: full passes are done here as well.
enum { PART_ALL, PART_MEDIAN, PART_MAD };
__global__ void __launch_bounds__(select::kThreads, 1)
    k_select(DevState* st, const float* src, long long n, Lists L, int pair, int part, int all) {
  using namespace select;
  __shared__ Smem S;
  chain_begin();
  cg::cluster_group cl = cg::this_cluster();
  const NoisePlan& p = st->plan;
  const int flags = p.flags;
  if (flags & (PLAN_EMPTY | PLAN_STD)) return;
  const bool med_full = (flags & PLAN_MED_FULL) != 0, mad_full = (flags & PLAN_MAD_FULL) != 0;
  if (!all && (med_full || mad_full)) return;  // the full passes follow
  const unsigned long long n_med = med_full ? (unsigned long long)n : min(st->n_cand_med, L.cap.med);
  const unsigned long long n_mad = mad_full ? (unsigned long long)n : min(st->n_cand_mad, L.cap.mad);
  const bool shortened = part == PART_MAD && st->mad_short;
  const bool solo = (part == PART_MAD || n_med <= kOneBlock) &&
                    (part == PART_MEDIAN || (shortened ? (unsigned long long)st->n_mad_short : n_mad) <= kOneBlock);
  const int me = (int)cl.block_rank(), nc = solo ? 1 : (int)cl.num_blocks();
  if (solo && me != 0) return;
  const bool lead = me == 0 && threadIdx.x == 0;
  const bool even = p.k_hi != p.k_lo;
  AbsDev d = st->dev;
#pragma unroll 1
  for (int which = part == PART_MAD ? 1 : 0; which < (part == PART_MEDIAN ? 1 : 2); ++which) {
    Task t;
    t.want_next = even ? 1 : 0;
    t.next = kNone;
    t.store = 0;
    if (which == 0) {
      // the median's bins hold both middle values, the first of rank below_med
      t.list = med_full ? const_cast<float*>(src) : L.med;
      t.count = n_med;
      t.form = FORM_VALUE;
      t.rank = (unsigned)(p.k_lo - (med_full ? 0ull : p.below_med));
      t.klo = fkey(__double2float_rd(bin_lo_value(p.b_med_lo, p.cfg)));
      t.khi = fkey(__double2float_ru(bin_hi_value(p.b_med_hi, p.cfg)));
    } else if (shortened) {
      // the values of the first round's digit
      t.list = L.med;
      t.count = st->n_mad_short;
      t.form = FORM_KEY;
      t.rank = st->mad_rank;
      t.klo = st->mad_klo;
      t.khi = st->mad_khi;
      t.next = st->mad_next;
    } else {
      // T1 < MAD <= T2 where the plan has a bracket
      t.list = mad_full ? const_cast<float*>(src) : L.mad;
      t.count = n_mad;
      t.form = part == PART_MAD ? FORM_KEY : FORM_ABSDEV;
      t.store = part == PART_ALL && !mad_full ? 1 : 0;
      t.rank = (unsigned)(p.k_lo - (mad_full ? 0ull : p.n_B));
      t.klo = p.has_B ? fkey(p.T1) : fkey(0.0f);
      t.khi = fkey(p.T2);
    }
    const bool ok = select_rank(nc, t, d, &S);
    if (!ok) {
      if (lead) atomicOr(&st->status, (unsigned int)SC_ST_INTERNAL);
      return;
    }
    const float v1 = fkey_inv(S.k1), v2 = fkey_inv(S.k2);
    if (which == 0) {
      d = abs_dev_of(v1, v2);
      if (lead) {
        st->m = d.m;
        st->dev = d;
        st->mad_next = kNone;
        st->n_mad_short = 0u;
        st->mad_below = 0u;
      }
      if (part == PART_MEDIAN)  // for the first round of the MAD
        for (int i = me * kThreads + threadIdx.x; i < kBins; i += nc * kThreads) st->mad_digits[i] = 0u;
      __syncthreads();  // the result is read before the next selection writes it
    } else {
      const double mad = S.k1 == S.k2 ? (double)v1 : 0.5 * ((double)v1 + (double)v2);
      const float sg = sigma_of_mad(mad);
      if (lead) {
        st->mad = mad;
        st->sigma_cur_d = kMadToSigma * mad;
        st->sigma_cur = sg;
        if (pair >= 0) st->sigma[pair] = sg;
        if (!(sg > 0.0f)) st->warn |= SC_WARN_ZERO_SIGMA;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// The MAD's first round over a long list, by all SMs: the keys over the list's
// values and the counts of the digits of [T1, T2].
constexpr int kMadThreads = 512;
constexpr int kMadUnroll = 8;
__device__ __forceinline__ bool mad_by_grid(const NoisePlan& p) {
  return !(p.flags & (PLAN_EMPTY | PLAN_STD | PLAN_MED_FULL | PLAN_MAD_FULL));
}

__global__ void __launch_bounds__(kMadThreads) k_mad_digits(DevState* st, Lists L) {
  using namespace select;
  __shared__ unsigned hist[kBins];
  chain_begin();
  const NoisePlan& p = st->plan;
  if (!mad_by_grid(p)) return;
  for (int i = threadIdx.x; i < kBins; i += kMadThreads) hist[i] = 0u;
  __syncthreads();
  const AbsDev d = st->dev;
  const unsigned klo = p.has_B ? fkey(p.T1) : fkey(0.0f), khi = fkey(p.T2);
  const int shift = first_shift(klo, khi);
  const unsigned long long count = min(st->n_cand_mad, L.cap.mad), stride = (unsigned long long)gridDim.x * kMadThreads;
  const unsigned lane = threadIdx.x & 31u;
  unsigned under = 0u;
  for (unsigned long long w0 = (unsigned long long)blockIdx.x * kMadThreads + threadIdx.x - lane; w0 < count;
       w0 += kMadUnroll * stride) {
    float v[kMadUnroll];
#pragma unroll
    for (int u = 0; u < kMadUnroll; ++u) {
      const unsigned long long i = w0 + lane + u * stride;
      v[u] = i < count ? L.mad[i] : __uint_as_float(kNone);
    }
#pragma unroll
    for (int u = 0; u < kMadUnroll; ++u) {
      const unsigned long long i = w0 + lane + u * stride;
      const unsigned k = key_of(FORM_ABSDEV, v[u], d);
      if (i < count) L.mad[i] = __uint_as_float(k);
      under += k < klo ? 1u : 0u;
      count_digit(hist, (k >= klo && k <= khi && k != kNone) ? (k - klo) >> shift : kNone);
    }
  }
  under = __reduce_add_sync(0xffffffffu, under);
  if (lane == 0u && under) atomicAdd(&st->mad_below, under);
  __syncthreads();
  for (int i = threadIdx.x; i < kBins; i += kMadThreads)
    if (hist[i]) atomicAdd(&st->mad_digits[i], hist[i]);
}

// Every block picks the digit that holds the rank; its keys go to L.med (the
// median's list is done with), unless there are too many, and the smallest key
// above them to mad_next.
__global__ void __launch_bounds__(kMadThreads) k_mad_compact(DevState* st, Lists L) {
  using namespace select;
  __shared__ unsigned part[kMadThreads / 32], s_digit, s_rank, s_count;
  chain_begin();
  const NoisePlan& p = st->plan;
  if (!mad_by_grid(p)) return;
  const unsigned tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  constexpr int kPer = kBins / kMadThreads;
  static_assert(kPer == 4, "four digits per thread");
  const uint4 c = reinterpret_cast<const uint4*>(st->mad_digits)[tid];
  const unsigned cc[4] = {c.x, c.y, c.z, c.w}, sum = c.x + c.y + c.z + c.w;
  unsigned x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if ((int)lane >= o) x += y;
  }
  if (lane == 31u) part[warp] = x;
  if (tid == 0u) s_count = 0u;
  __syncthreads();
  unsigned run = st->mad_below + x - sum;
  for (unsigned k = 0; k < warp; ++k) run += part[k];
  const unsigned rank = (unsigned)(p.k_lo - p.n_B);
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    if (rank >= run && rank < run + cc[j]) {
      s_digit = kPer * tid + j;
      s_rank = rank - run;
      s_count = cc[j];
    }
    run += cc[j];
  }
  __syncthreads();
  // nothing found (the next selection reports it) or too many: no short list
  const bool fits = s_count > 0u && (unsigned long long)s_count <= L.cap.med;
  unsigned klo = p.has_B ? fkey(p.T1) : fkey(0.0f), khi = fkey(p.T2);
  const int shift = first_shift(klo, khi);
  klo += s_digit << shift;
  const unsigned span = (1u << shift) - 1u;
  khi = khi - klo < span ? khi : klo + span;
  if (blockIdx.x == 0 && tid == 0u) {
    st->mad_short = fits ? 1 : 0;
    st->mad_rank = s_rank;
    st->mad_klo = klo;
    st->mad_khi = khi;
  }
  if (!fits) return;
  const unsigned long long count = min(st->n_cand_mad, L.cap.mad), stride = (unsigned long long)gridDim.x * kMadThreads;
  unsigned mn = kNone;
  for (unsigned long long w0 = (unsigned long long)blockIdx.x * kMadThreads + tid - lane; w0 < count;
       w0 += kMadUnroll * stride) {
    unsigned k[kMadUnroll];
#pragma unroll
    for (int u = 0; u < kMadUnroll; ++u) {
      const unsigned long long i = w0 + lane + u * stride;
      k[u] = i < count ? __float_as_uint(__ldcg(L.mad + i)) : kNone;
    }
#pragma unroll
    for (int u = 0; u < kMadUnroll; ++u) {
      if (k[u] > khi) mn = min(mn, k[u]);
      const bool in = k[u] >= klo && k[u] <= khi && k[u] != kNone;
      const unsigned bal = __ballot_sync(0xffffffffu, in);
      if (bal) {
        unsigned at = 0u;
        if (lane == 0u) at = atomicAdd(&st->n_mad_short, (unsigned)__popc(bal));
        at = __shfl_sync(0xffffffffu, at, 0) + (unsigned)__popc(bal & ((1u << lane) - 1u));
        if (in) L.med[at] = __uint_as_float(k[u]);
      }
    }
  }
  mn = __reduce_min_sync(0xffffffffu, mn);
  if (lane == 0u && mn != kNone) atomicMin(&st->mad_next, mn);
}

// ---------------------------------------------------------------------------
// Median and 1.4826 MAD of the finite values of an array (stats[0], stats[1];
// NaN if there is none), by one cluster: 0.36 M values took one block of
// 1,024 threads, with eight passes and a match_any per value, 0.89 ms; they
// take 0.17 ms.
__global__ void __launch_bounds__(select::kThreads, 1) k_array_stats(const float* x, long long n, double* stats) {
  using namespace select;
  __shared__ Smem S;
  cg::cluster_group cl = cg::this_cluster();
  const bool solo = n <= (long long)kOneBlock;
  const int me = (int)cl.block_rank(), nc = solo ? 1 : (int)cl.num_blocks();
  if (solo && me != 0) return;
  if (threadIdx.x == 0) S.total_below = 0u;
  __syncthreads();
  unsigned c = 0u;
  for (long long i = (long long)me * kThreads + threadIdx.x; i < n; i += (long long)nc * kThreads)
    c += isfinite(x[i]) ? 1u : 0u;
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(&S.total_below, c);
  __syncthreads();
  unsigned nf = S.total_below;
  if (nc > 1) {
    cl.sync();
    nf = 0u;
    for (int r = 0; r < nc; ++r) nf += *cl.map_shared_rank(&S.total_below, r);
    cl.sync();  // the counts are read before a selection writes there
  }
  __syncthreads();
  const bool lead = me == 0 && threadIdx.x == 0;
  Task t;
  t.list = const_cast<float*>(x);  // (read only: nothing is stored)
  t.count = (unsigned long long)n;
  t.rank = nf ? (nf - 1u) / 2u : 0u;
  t.want_next = nf && !(nf & 1u) ? 1 : 0;
  t.next = kNone;
  t.store = 0;
  AbsDev d{};
  double sigma = __longlong_as_double(0x7ff8000000000000LL), m = sigma;
  bool ok = nf > 0u;
#pragma unroll 1
  for (int which = 0; which < 2 && ok; ++which) {
    t.form = which ? FORM_ABSDEV : FORM_VALUE;
    t.klo = which ? fkey(0.0f) : fkey(-FLT_MAX);
    t.khi = which ? fkey(INFINITY) : fkey(FLT_MAX);
    ok = select_rank(nc, t, d, &S);
    if (!ok) break;  // (not reached: the counts come from the same values)
    const float a = fkey_inv(S.k1), b = fkey_inv(S.k2);
    __syncthreads();
    if (which == 0) {
      d = abs_dev_of(a, b);
      m = d.m;
    } else {
      sigma = kMadToSigma * (a == b ? (double)a : 0.5 * ((double)a + (double)b));
    }
  }
  if (lead) {
    stats[0] = m;
    stats[1] = sigma;
  }
}

namespace {
// One cluster of `blocks` blocks as a launch configuration.
struct ClusterLaunch {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  ClusterLaunch(unsigned blocks, cudaStream_t s) {
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(select::kThreads);
    cfg.stream = s;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = blocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
  }
};
cudaError_t launch_part(DevState* st, const float* src, long long n, const Lists& L, int pair, int part, int all,
                        unsigned blocks, cudaStream_t s) {
  return launch_chained(k_select, blocks, select::kThreads, 0, blocks, s, st, src, n, L, pair, part, all);
}
}  // namespace

cudaError_t launch_array_stats(const float* x, long long n, double* stats, cudaStream_t s) {
  ClusterLaunch c(8u, s);
  return cudaLaunchKernelEx(&c.cfg, k_array_stats, x, n, stats);
}

void init_select_attrs() { cudaFuncSetAttribute(k_select, cudaFuncAttributeNonPortableClusterSizeAllowed, 1); }

// One cluster: of 8 blocks up to kSelectAllMax values, of 16 above (the MAD's
// list of a 217 x 331 x 509 cube, 0.25 M values, takes 37 us then, 50 with 8).
// Arrays of more than kSelectGridMin values take the MAD's first round by all
// SMs. The four launches start before one another's ends, so the line lies
// where they win on a whole run: 12 pairs on 217 x 331 x 509 voxels (36.6 M)
// 3.64 ms against 3.70 with one cluster, 20 pairs on 256 x 312 x 640 (51 M)
// 7.60 against 7.84; a line at 2^24 gave the same. On 360 x 360 x 1464 voxels
// the launches take 46 us of a measurement against 73, on 1200 x 1200 x 1024
// 66 against 304.
cudaError_t launch_select_lists(DevState* st, const float* src, long long n, Lists L, int pair, int sms,
                                cudaStream_t s, int* launches) {
  const int all = n <= kSelectAllMax ? 1 : 0;
  if (n <= kSelectGridMin) {
    *launches = 1;
    return launch_part(st, src, n, L, pair, PART_ALL, all, all ? 8u : 16u, s);
  }
  *launches = 4;
  cudaError_t e = launch_part(st, src, n, L, pair, PART_MEDIAN, all, 8u, s);
  if (e != cudaSuccess) return e;
  if ((e = launch_chained(k_mad_digits, 2 * sms, kMadThreads, 0, 0, s, st, L)) != cudaSuccess) return e;
  if ((e = launch_chained(k_mad_compact, 2 * sms, kMadThreads, 0, 0, s, st, L)) != cudaSuccess) return e;
  return launch_part(st, src, n, L, pair, PART_MAD, all, 8u, s);
}

}  // namespace sc
