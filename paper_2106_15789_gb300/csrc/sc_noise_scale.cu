// Local noise normalisation (SoFiA 2 Sect. 4.1, windows of 31 pixels and
// channels in the speed test of Sect. 5): the cube is divided by the noise
// level measured in a window around each voxel's cell.
//
//   k_noise_window  one block per cell (persistent over cells): the noise of
//                   the chosen mode over the finite voxels of the cell's
//                   window, clipped to the cube, which is streamed from
//                   memory: MAD by two exact selections (the median, then the
//                   median of the float32 values |x - m|, rounded correctly
//                   for an odd count and faithfully for an even one), STD by
//                   two passes of compensated float32 sums combined in double.
//                   Writes the cell's noise (double) and the float32
//                   reciprocal used below.
//   k_noise_apply   out = in * (1 / sigma) per voxel (NaN where the input is
//                   not finite or the cell has no positive noise).
//
// Cells are gx x gy x gz voxels (the last one along an axis may be shorter);
// a cell's window is centred on voxel start + (extent - 1) / 2 of each axis.
//
// A selection takes one pass over the window: a sample of it (every 8th voxel
// of a row, kept in shared memory) brackets the wanted rank, the pass counts
// the values under the bracket and every lane copies those of its own inside
// it (4 % of them, to its own column of shared memory: no votes; where few
// columns of the window are finite, also to a common pool), and the rank is
// found among the copies by one histogram of 2048 equal steps of the bracket
// and a direct ranking inside one step. A bracket that misses its rank, or
// holds more values than the copies' room, costs radix passes over the window
// instead, so the result is exact whatever the data.
//
// What bounds it: instruction issue of the two passes (2.8 of 4 slots a cycle
// while a block is resident); the 7 windows that share a voxel read it from
// L2. Blocks of 256 threads, four to an SM, hide each other's barriers and
// loads. On 360 x 360 x 1464 voxels (48,668 windows of 31^3) the earlier form,
// one block of 1,024 threads per SM with the window in shared memory,
// warp-aggregated (match_any) histograms and up to 40 barriers a window, took
// 16.9 ms; this one 5.2 ms.
#include <cfloat>
#include <cstdint>

#include "sc_device.cuh"
#include "sc_gaussfit.cuh"
#include "sc_internal.h"

namespace sc {
namespace nscale {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kBlocksPerSm = 4;
constexpr int kBins = 2048;              // steps of a bracket; radix digits of 11, 11 and 10 bits
constexpr unsigned kNone = 0xffffffffu;  // above the key of every finite value
constexpr int kLaneCap = 20;             // copies each thread keeps of its values in a bracket
constexpr int kPool = 512;               // and those beyond, for the block
constexpr int kSampleSlots = 16;         // sampled voxels per thread
constexpr int kUnroll = 8;               // loads in flight per thread
constexpr int kFewCap = 256;             // copies ranked directly

struct Geo {
  long long nx, ny, nz;
  int wx, wy, wz;     // window (odd)
  int gx, gy, gz;     // cell size
  int ncx, ncy, ncz;  // cells per axis
};

// Window of the cell with index c along an axis of length n: [lo, hi).
__device__ __forceinline__ void window_range(int c, int g, int w, long long n, long long* lo, long long* hi) {
  const long long start = (long long)c * g;
  const long long extent = min((long long)g, n - start);
  const long long centre = start + (extent - 1) / 2;
  const int r = (w - 1) / 2;
  *lo = max(centre - r, 0LL);
  *hi = min(centre + r + 1, n);
}

struct Scratch {
  float cand[kLaneCap * kThreads];        // a column per thread
  float pool[kPool];
  float sample[kSampleSlots * kThreads];  // a column per thread; NaN: no finite voxel
  union {
    alignas(16) unsigned hist[kBins];
    float few[kFewCap];
  };
  unsigned part[kWarps];
  unsigned digit[2], rank[2], n_few, next, finite, below, n_copies, n_pool, n_sample;
  float v1;
  double dpart[kWarps];
};

// A window: voxel (x, y, z) at base + z plane + y nx + x. A row goes to a
// group of 2^lw lanes (the smallest power of two that covers it, up to 32), a
// plane's rows to 2^wy of the block's warps, in turns, and its planes to the
// 8 / 2^wy sets of warps that leaves.
struct Win {
  const float* base;
  long long plane, nx;
  int lx, ly, lz, lw, wy;
  __device__ __forceinline__ void split() {
    lw = lx > 16 ? 5 : (lx > 8 ? 4 : (lx > 4 ? 3 : 2));
    const int need = (ly + (32 >> lw) - 1) >> (5 - lw);
    wy = need > 4 ? 3 : (need > 2 ? 2 : (need > 1 ? 1 : 0));
  }
  __device__ __forceinline__ int step() const { return 1 << (wy + 5 - lw); }  // rows of a turn
  __device__ __forceinline__ int turns() const { return (ly + step() - 1) / step(); }
  __device__ __forceinline__ int sets() const { return kWarps >> wy; }
  // Most voxels one thread takes.
  __device__ __forceinline__ int share() const {
    return turns() * ((lz + sets() - 1) / sets()) * ((lx + (1 << lw) - 1) >> lw);
  }
};

// f(v) for every voxel v of the window, NaN in the lanes left over; all lanes
// of a warp call f together, kUnroll loads ahead. The turn and the plane are
// the same for all lanes, so a lane adds its own fixed offset to an address
// that a warp shares. FAST: planes of three or four turns (17 to 32 rows of
// more than 16 voxels) get code of their own, two planes at a time with a
// quarter of the address arithmetic; for the passes over every voxel. Other
// windows take the general loop: a MAD noise costs 3.9 ps a window voxel at 31^3,
// 4.8 at 31 x 33 x 31 and 6.9 at 33^3 (11^3 and 15^3, copied whole, 17.9 and 8.3;
// 17^3, sampled and too small to fill its lanes, 14.8).
template <bool FAST, class F>
__device__ __forceinline__ void for_window(const Win& w, F f) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int group = 1 << w.lw, step = w.step(), turns = w.turns(), sets = w.sets();
  const int y0 = ((warp & ((1 << w.wy) - 1)) << (5 - w.lw)) + (lane >> w.lw), z0 = warp >> w.wy;
  const int total = z0 < w.lz ? turns * ((w.lz - z0 + sets - 1) / sets) : 0;
  const long long turn = step * w.nx, wrap = sets * w.plane - turns * turn;
  for (int x0 = 0; x0 < w.lx; x0 += group) {
    const int dx = x0 + (lane & (group - 1));
    const int rows = dx < w.lx ? w.ly - y0 : 0;  // rows left from the lane's first one on
    const float* const mine = w.base + z0 * w.plane + y0 * w.nx + dx;
    if (FAST && turns > 2 && turns <= 4) {
      const float* q = mine;
      const long long jump = sets * w.plane;
      const int planes = total / turns;
      const bool ok[4] = {0 < rows, step < rows, 2 * step < rows, 3 * step < rows};
      for (int z = 0; z < planes; z += 2, q += 2 * jump) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          v[u] = __int_as_float(0x7fc00000);
          if (ok[u & 3] && (u < 4 || z + 1 < planes)) v[u] = __ldg(q + (u >> 2) * jump + (u & 3) * turn);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) f(v[u]);
      }
      continue;
    }
    long long at = 0;
    int k = 0;
    for (int t0 = 0; t0 < total; t0 += kUnroll) {
      float v[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        v[u] = __int_as_float(0x7fc00000);
        if (k * step < rows && t0 + u < total) v[u] = __ldg(mine + at);
        at += turn;
        if (++k == turns) {
          k = 0;
          at += wrap;
        }
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) f(v[u]);
    }
  }
}

// Clears the histogram (a barrier follows before it is counted into).
__device__ __forceinline__ void clear_hist(Scratch* S) {
  uint4* h = reinterpret_cast<uint4*>(S->hist);
  h[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
  h[threadIdx.x + kThreads] = make_uint4(0u, 0u, 0u, 0u);
}

// The digits whose cumulative ranges in S->hist hold ranks ra and rb, and the
// ranks within them (S->digit, S->rank). Barriers before and after.
__device__ __forceinline__ void find_digits(Scratch* S, unsigned ra, unsigned rb) {
  static_assert(kBins == 8 * kThreads, "eight digits per thread");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __syncthreads();
  unsigned c[8], sum = 0u;
  const uint4 h0 = reinterpret_cast<const uint4*>(S->hist)[2 * tid], h1 = reinterpret_cast<const uint4*>(S->hist)[2 * tid + 1];
  c[0] = h0.x, c[1] = h0.y, c[2] = h0.z, c[3] = h0.w, c[4] = h1.x, c[5] = h1.y, c[6] = h1.z, c[7] = h1.w;
#pragma unroll
  for (int j = 0; j < 8; ++j) sum += c[j];
  unsigned x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  if (lane == 31) S->part[warp] = x;
  __syncthreads();
  unsigned run = x - sum;
  for (int k = 0; k < warp; ++k) run += S->part[k];
  if (ra < run + sum && rb >= run) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (ra >= run && ra < run + c[j]) {
        S->digit[0] = 8u * tid + j;
        S->rank[0] = ra - run;
      }
      if (rb >= run && rb < run + c[j]) {
        S->digit[1] = 8u * tid + j;
        S->rank[1] = rb - run;
      }
      run += c[j];
    }
  }
  __syncthreads();
}

// The MAD value of x: the float of |x - m| with m = (a + b) / 2 (a == b for an
// odd count: one correctly rounded subtraction). For an even count, x - a/2
// and then - b/2 are taken exactly as sums of two floats and added back, which
// rounds the exact difference faithfully (within one unit in the last place)
// in single precision, without the slow FP64 pipe.
struct AbsDev {
  float a, b;
  bool even;
  __device__ __forceinline__ float operator()(float x) const {
    if (!even) return fabsf(__fsub_rn(x, a));
    float e1, e2;
    const float t = two_sum(x, -0.5f * a, &e1);
    const float u = two_sum(t, -0.5f * b, &e2);
    return fabsf(__fadd_rn(u, __fadd_rn(e1, e2)));
  }
};
struct Value {
  __device__ __forceinline__ float operator()(float x) const { return x; }
};

// Order statistics r and (want_next) r + 1 of of(x) over the finite voxels x of
// the window, by radix passes over it (digits of 11, 11 and 10 bits).
template <class Of>
__device__ __noinline__ void select_window(const Win& w, Of of, unsigned r, bool want_next, Scratch* S, float* v1,
                                           float* v2) {
  const int tid = threadIdx.x;
  unsigned prefix = 0u, pmask = 0u;
  for (int round = 0; round < 3; ++round) {
    const int shift = round == 0 ? 21 : (round == 1 ? 10 : 0);
    const unsigned dmask = round == 2 ? 0x3ffu : 0x7ffu;
    __syncthreads();
    clear_hist(S);
    __syncthreads();
    for_window<false>(w, [&](float v) {
      const unsigned k = isfinite(v) ? fkey(of(v)) : kNone;
      const bool in = k != kNone && (k & pmask) == prefix;
      const unsigned d = in ? (k >> shift) & dmask : kNone;
      const unsigned d0 = __shfl_sync(0xffffffffu, d, 0);  // ties are added at once
      if (__all_sync(0xffffffffu, d == d0)) {
        if ((threadIdx.x & 31) == 0 && d != kNone) atomicAdd(&S->hist[d], 32u);
      } else if (d != kNone) {
        atomicAdd(&S->hist[d], 1u);
      }
    });
    find_digits(S, r, r);
    r = S->rank[0];
    const unsigned d = S->digit[0];
    prefix |= d << shift;
    pmask |= dmask << shift;
    if (round == 2) {
      *v1 = *v2 = fkey_inv(prefix);
      if (want_next && r + 1u >= S->hist[d]) {  // the next order statistic is another value
        if (tid == 0) S->next = kNone;
        __syncthreads();
        unsigned mn = kNone;
        for_window<false>(w, [&](float v) {
          const unsigned k = isfinite(v) ? fkey(of(v)) : 0u;
          if (k > prefix) mn = min(mn, k);
        });
        mn = __reduce_min_sync(0xffffffffu, mn);
        if ((tid & 31) == 0) atomicMin(&S->next, mn);
        __syncthreads();
        *v2 = fkey_inv(S->next);
      }
    }
  }
  __syncthreads();
}

// Order statistics r and (want_next) r + 1 among the copies (all in [lo, hi],
// more than r of them); for a next one outside them, nxt(): its value. False
// (uniformly) when too many copies share the step of the rank.
template <class Next>
__device__ bool select_cand(int n, float lo, float hi, unsigned r, bool want_next, Scratch* S, float* v1, float* v2,
                            Next nxt) {
  const int tid = threadIdx.x, lane = tid & 31;
  // f(v) for this thread's n copies, kThreads apart, and its part of the pool
  const int np = (int)S->n_pool;
  const auto copies = [&](auto f) {
    for (int i = 0; i < n; ++i) f(S->cand[i * kThreads + tid]);
    for (int i = tid; i < np; i += kThreads) f(S->pool[i]);
  };
  // the step of a copy: a monotone function of its value
  const float inv = (float)kBins / (hi - lo);
  const auto digit = [&](float v) { return min(kBins - 1, (int)((v - lo) * inv)); };
  clear_hist(S);
  if (tid == 0) {
    S->n_few = 0u;
    S->next = kNone;
  }
  __syncthreads();
  copies([&](float v) { atomicAdd(&S->hist[digit(v)], 1u); });
  find_digits(S, r, r);
  const int d = (int)S->digit[0];
  const unsigned rr = S->rank[0], cnt = S->hist[d];
  if (cnt > (unsigned)kFewCap) {
    // ties? one value in the whole step is the answer
    __syncthreads();  // (the digit and the counts are read)
    if (tid == 0) {
      S->digit[0] = kNone;
      S->digit[1] = 0u;
    }
    __syncthreads();
    unsigned kmin = kNone, kmax = 0u;
    copies([&](float v) {
      if (digit(v) != d) return;
      kmin = min(kmin, fkey(v));
      kmax = max(kmax, fkey(v));
    });
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) {
      atomicMin(&S->digit[0], kmin);
      atomicMax(&S->digit[1], kmax);
    }
    __syncthreads();
    const bool same = S->digit[0] == S->digit[1];
    *v1 = *v2 = fkey_inv(S->digit[0]);
    __syncthreads();
    return same && (!want_next || rr + 1u < cnt);
  }
  __syncthreads();  // the counts are read: their memory becomes the step's values
  unsigned above = kNone;
  copies([&](float v) {
    const int dv = digit(v);
    if (dv == d) S->few[atomicAdd(&S->n_few, 1u)] = v;
    else if (dv > d) above = min(above, fkey(v));
  });
  if (want_next) {
    above = __reduce_min_sync(0xffffffffu, above);
    if (lane == 0) atomicMin(&S->next, above);
  }
  __syncthreads();
  if (tid < (int)cnt) {
    const float v = S->few[tid];
    unsigned k = 0u;  // its rank in the step, ties in the order of the list
    for (int j = 0; j < (int)cnt; ++j) {
      const float o = S->few[j];
      k += (o < v || (o == v && j < tid)) ? 1u : 0u;
    }
    if (k == rr) S->v1 = v;
    if (want_next && k == rr + 1u) S->next = fkey(v);
  }
  __syncthreads();
  *v1 = *v2 = S->v1;
  if (want_next) *v2 = S->next != kNone ? fkey_inv(S->next) : nxt();
  return true;
}

// Counts the values under lo and copies those in [lo, hi] to the thread's
// column (n of them) and, once that is full, to the pool.
struct Collect {
  float lo, hi;
  Scratch* S;
  int n;
  unsigned below;
  __device__ __forceinline__ void operator()(float a) {  // (NaN: neither)
    const bool under = a < lo;
    below += under ? 1u : 0u;
    if (a <= hi && !under) {
      if (n < kLaneCap) {
        S->cand[n * kThreads + threadIdx.x] = a;
        ++n;
      } else {
        const unsigned i = atomicAdd(&S->n_pool, 1u);
        if (i < (unsigned)kPool) S->pool[i] = a;
      }
    }
  }
  // Adds a pass's counts up (S->below, n_copies, n_pool cleared before it).
  __device__ __forceinline__ void finish() const {
    const unsigned b = __reduce_add_sync(0xffffffffu, below), c = __reduce_add_sync(0xffffffffu, (unsigned)n);
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(&S->below, b);
      atomicAdd(&S->n_copies, c);
    }
  }
};

// Bracket [lo, hi] of sample rank p of of(x) over the ns finite sampled voxels
// (`slots` per thread): 2.5 binomial standard deviations either side (a sample
// at fixed places scatters less; wider ones overflow the columns where few
// voxels are finite), located by the keys' bits from kShift on and
// then by 2048 equal steps between. Any bracket is checked by the pass's counts.
template <int kShift, class Of, class Key>
__device__ void sample_bracket(Scratch* S, int slots, Of of, Key key, unsigned ns, unsigned p, float* lo, float* hi) {
  const float* const mine = S->sample + threadIdx.x;
  clear_hist(S);
  __syncthreads();
  for (int i = 0; i < slots; ++i) {
    const float v = of(mine[i * kThreads]);
    if (v == v) atomicAdd(&S->hist[min(key(v) >> kShift, (unsigned)kBins - 1u)], 1u);
  }
  const unsigned delta = (unsigned)(1.25f * sqrtf((float)ns)) + 4u;
  const unsigned ra = p > delta ? p - delta : 0u, rb = min(p + delta, ns - 1u);
  find_digits(S, ra, rb);
  const float a = fminf(fmaxf(key.value(S->digit[0] << kShift), -FLT_MAX), FLT_MAX);
  const float b = fminf(fmaxf(key.value((S->digit[1] << kShift) | ((1u << kShift) - 1u)), -FLT_MAX), FLT_MAX);
  const unsigned ia = S->rank[0];
  *lo = a;
  *hi = b;
  const float inv = (float)kBins / (b - a);
  __syncthreads();
  if (!(inv > 0.0f && inv <= FLT_MAX)) return;
  clear_hist(S);
  __syncthreads();
  for (int i = 0; i < slots; ++i) {
    const float v = of(mine[i * kThreads]);
    if (v >= a && v <= b) atomicAdd(&S->hist[min(kBins - 1, (int)((v - a) * inv))], 1u);
  }
  // the ranks among the values from the first digit on
  find_digits(S, ia, ia + (rb - ra));
  const float step = (b - a) / (float)kBins;
  *lo = fmaxf(a, a + (float)S->digit[0] * step);
  *hi = fminf(b, a + (float)(S->digit[1] + 1u) * step);
  __syncthreads();
}

// Samples every 8th voxel (of rows over 4,096 voxels fewer) of every rstep-th
// row, the offset moving with the row, into the threads' columns; returns the
// slots used, and adds the finite ones to S->n_sample.
__device__ __forceinline__ int take_sample(const Win& w, Scratch* S) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int lstep = 3;
  while ((w.lx >> lstep) >= 32 * kSampleSlots) ++lstep;
  const int rows = w.ly * w.lz, sx = (w.lx + (1 << lstep) - 1) >> lstep;
  const int ls = sx > 16 ? 5 : (sx > 8 ? 4 : (sx > 4 ? 3 : (sx > 2 ? 2 : 1)));  // 2^ls lanes share a row
  const int turns = (sx + (1 << ls) - 1) >> ls, at_once = kWarps << (5 - ls);   // rows of a slot
  int rstep = 1;
  while (turns * (((rows + rstep - 1) / rstep + at_once - 1) / at_once) > kSampleSlots) ++rstep;
  const int groups = ((rows + rstep - 1) / rstep + at_once - 1) / at_once;
  const int q0 = (warp << (5 - ls)) + (lane >> ls);  // the thread's first sampled row
  const int inc = at_once * rstep, dz = inc / w.ly, dy = inc - dz * w.ly;
  unsigned c = 0u;
  int slot = 0;
  for (int t = 0; t < turns; ++t) {
    int q = q0, z = q0 * rstep / w.ly, y = q0 * rstep - z * w.ly;
    const int j = (t << ls) + (lane & ((1 << ls) - 1));
    for (int g0 = 0; g0 < groups; g0 += 4) {
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int dx = (j << lstep) + ((3 * q) & 7);
        v[u] = __int_as_float(0x7fc00000);
        if (z < w.lz && dx < w.lx) v[u] = __ldg(w.base + z * w.plane + y * w.nx + dx);
        q += at_once;
        y += dy;
        z += dz;
        if (y >= w.ly) {
          y -= w.ly;
          ++z;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (g0 + u >= groups) break;
        const bool ok = isfinite(v[u]);
        S->sample[(slot++) * kThreads + tid] = ok ? v[u] : __int_as_float(0x7fc00000);
        c += ok ? 1u : 0u;
      }
    }
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if (lane == 0 && c) atomicAdd(&S->n_sample, c);
  return slot;
}

__device__ __forceinline__ double block_sum_d(double v, double* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) part[warp] = v;
  __syncthreads();
  double t = 0.0;
#pragma unroll
  for (int k = 0; k < kWarps; ++k) t += part[k];
  __syncthreads();
  return t;
}

// Exact median and MAD noise of the window's finite voxels (NaN if none).
__device__ double window_mad(const Win& w, Scratch* S) {
  const int tid = threadIdx.x, lane = tid & 31;
  Collect col;
  col.S = S;
  // a window whose threads' shares fit their columns is copied whole
  const bool whole = w.share() <= kLaneCap;
  float lo = -FLT_MAX, hi = FLT_MAX;
  unsigned ns = 0u;
  int slots = 0;
  if (tid == 0) S->finite = S->below = S->n_copies = S->n_pool = S->n_sample = 0u;
  __syncthreads();
  if (!whole) {
    slots = take_sample(w, S);
    __syncthreads();
    ns = S->n_sample;
    if (ns >= 64u) sample_bracket<21>(S, slots, Value{}, KeyOfValue{}, ns, (ns - 1u) / 2u, &lo, &hi);
  }
  const bool bracket = whole || ns >= 64u;
  unsigned finite = 0u;
  col.lo = lo;
  col.hi = hi;
  col.n = 0;
  col.below = 0u;
  for_window<true>(w, [&](float v) {
    const bool ok = fabsf(v) <= FLT_MAX;  // false for NaN and Inf
    finite += ok ? 1u : 0u;
    col(ok ? v : __int_as_float(0x7fc00000));
  });
  finite = __reduce_add_sync(0xffffffffu, finite);
  if (lane == 0) atomicAdd(&S->finite, finite);
  col.finish();
  __syncthreads();
  const unsigned nf = S->finite;
  if (nf == 0u) return __longlong_as_double(0x7ff8000000000000LL);  // no finite voxel
  const unsigned r1 = (nf - 1u) / 2u;
  const bool even = (nf & 1u) == 0u;
  // the copies are complete and hold the rank
  const auto holds = [&] {
    return S->n_pool <= (unsigned)kPool && r1 >= S->below && r1 - S->below < S->n_copies + S->n_pool;
  };
  unsigned below = S->below;
  bool done = bracket && holds();
  // the smallest and largest of the copies' values, as their bracket
  const auto ends = [&](bool both) {
    if (tid == 0) {
      S->digit[0] = kNone;
      S->digit[1] = 0u;
    }
    __syncthreads();
    unsigned kmin = kNone, kmax = 0u;
    for (int i = 0; i < col.n; ++i) {
      const unsigned k = fkey(S->cand[i * kThreads + tid]);
      kmin = min(kmin, k);
      kmax = max(kmax, k);
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) {
      atomicMin(&S->digit[0], kmin);
      atomicMax(&S->digit[1], kmax);
    }
    __syncthreads();
    lo = both ? fkey_inv(S->digit[0]) : 0.0f;
    hi = fkey_inv(S->digit[1]);
    __syncthreads();
  };
  if (whole) ends(true);
  // the smallest value of(x) above hi in the window
  const auto above = [&](auto of, float top) {
    unsigned mn = kNone;
    for_window<false>(w, [&](float v) {
      const float a = isfinite(v) ? of(v) : __int_as_float(0x7fc00000);
      if (a > top) mn = min(mn, fkey(a));
    });
    mn = __reduce_min_sync(0xffffffffu, mn);
    __syncthreads();
    if (lane == 0) atomicMin(&S->next, mn);
    __syncthreads();
    return fkey_inv(S->next);
  };
  float ma = 0.0f, mb = 0.0f;
  if (done)
    done = select_cand(col.n, lo, hi, r1 - below, even, S, &ma, &mb, [&] { return above(Value{}, hi); });
  if (!done) select_window(w, Value{}, r1, even, S, &ma, &mb);
  if (!even) mb = ma;
  __syncthreads();
  // the MAD: the same order statistics of |x - m|, m = (ma + mb) / 2
  const AbsDev dev{ma, mb, even};
  float d1 = 0.0f, d2 = 0.0f;
  if (whole) {  // the copies are all finite voxels
    for (int i = 0; i < col.n; ++i) S->cand[i * kThreads + tid] = dev(S->cand[i * kThreads + tid]);
    ends(false);
    done = select_cand(col.n, 0.0f, hi, r1, even, S, &d1, &d2, [&] { return d1; });
  } else {
    done = ns >= 64u;
    if (done) {
      if (tid == 0) S->below = S->n_copies = S->n_pool = 0u;
      sample_bracket<20>(S, slots, dev, KeyOfDev{}, ns, (unsigned)(((unsigned long long)r1 * ns) / nf), &col.lo,
                         &col.hi);
      col.n = 0;
      col.below = 0u;
      for_window<true>(w, [&](float v) { col(dev(v)); });  // NaN and Inf voxels: |v - m| is NaN or Inf
      col.finish();
      __syncthreads();
      below = S->below;
      done = holds();
    }
    if (done)
      done = select_cand(col.n, col.lo, col.hi, r1 - below, even, S, &d1, &d2, [&] { return above(dev, col.hi); });
  }
  if (!done) select_window(w, dev, r1, even, S, &d1, &d2);
  const double mad = even ? 0.5 * ((double)d1 + (double)d2) : (double)d1;
  return kMadToSigma * mad;
}

}  // namespace nscale

__global__ void __launch_bounds__(nscale::kThreads, nscale::kBlocksPerSm)
    k_noise_window(const float* __restrict__ cube, nscale::Geo g, int mode, double* __restrict__ sig_out,
                   float* __restrict__ rinv_out) {
  using namespace nscale;
  __shared__ Scratch S;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long n_cells = (long long)g.ncx * g.ncy * g.ncz;
  Win w;
  w.plane = g.nx * g.ny;
  w.nx = g.nx;
  for (long long cell = blockIdx.x; cell < n_cells; cell += gridDim.x) {
    const int cx = (int)(cell % g.ncx);
    const int cy = (int)((cell / g.ncx) % g.ncy);
    const int cz = (int)(cell / ((long long)g.ncx * g.ncy));
    long long x0, x1, y0, y1, z0, z1;
    window_range(cx, g.gx, g.wx, g.nx, &x0, &x1);
    window_range(cy, g.gy, g.wy, g.ny, &y0, &y1);
    window_range(cz, g.gz, g.wz, g.nz, &z0, &z1);
    w.base = cube + z0 * w.plane + y0 * g.nx + x0;
    w.lx = (int)(x1 - x0);
    w.ly = (int)(y1 - y0);
    w.lz = (int)(z1 - z0);
    w.split();
    __syncthreads();  // the previous cell is done with the scratch
    double sigma;
    if (mode == SC_NOISE_STD) {
      // float32 sums with Neumaier compensation per thread (the FP64 pipe is
      // slow on this part), combined in double across the block
      float s = 0.0f, sc = 0.0f;
      unsigned finite = 0u;
      for_window<false>(w, [&](float v) {
        if (isfinite(v)) {
          neumaier_add(&s, &sc, v);
          ++finite;
        }
      });
      finite = __reduce_add_sync(0xffffffffu, finite);
      if (lane == 0) S.part[warp] = finite;
      const double sum = block_sum_d((double)s + (double)sc, S.dpart);
      unsigned nf = 0u;
      for (int k = 0; k < kWarps; ++k) nf += S.part[k];
      if (nf == 0u) {
        sigma = __longlong_as_double(0x7ff8000000000000LL);  // NaN: no finite voxel
      } else {
        const double mean = sum / (double)nf;
        const float mh = __double2float_rn(mean), ml = __double2float_rn(mean - (double)mh);
        float q = 0.0f, qc = 0.0f;
        for_window<false>(w, [&](float v) {
          if (isfinite(v)) {
            const float d = __fsub_rn(__fsub_rn(v, mh), ml);
            neumaier_add(&q, &qc, __fmul_rn(d, d));
          }
        });
        const double qq = block_sum_d((double)q + (double)qc, S.dpart);
        sigma = nf > 1u ? sqrt(qq / (double)(nf - 1u)) : 0.0;
      }
    } else {
      sigma = window_mad(w, &S);
      if (mode == SC_NOISE_GAUSS && sigma > 0.0) {
        // the window's 256-bin histogram, then a one-warp fit; the MAD noise
        // stands without a root
        const float k = gfit::scale_of(sigma);
        __syncthreads();  // the selection is done with S.hist
        for (int i = tid; i < gfit::kBins; i += kThreads) S.hist[i] = 0u;
        __syncthreads();
        for_window<false>(w, [&](float v) {
          const int b = gfit::bin_of(v, k);
          if (b >= 0) atomicAdd(&S.hist[b], 1u);
        });
        __syncthreads();
        if (warp == 0) {
          const double tau = gfit::fit_tau_warp(S.hist);
          if (lane == 0) S.dpart[0] = tau;
        }
        __syncthreads();
        const double tau = S.dpart[0];
        if (tau > 0.0) sigma = gfit::noise_of(tau, k);
      }
    }
    if (tid == 0) {
      sig_out[cell] = sigma;
      rinv_out[cell] = sigma > 0.0 ? __double2float_rn(1.0 / sigma) : __int_as_float(0x7fc00000);
    }
  }
}

// One warp per (y, z) row; four voxels per lane step when the rows allow
// 16-byte accesses.
__global__ void __launch_bounds__(256) k_noise_apply(const float* in, float* out, nscale::Geo g,
                                                     const float* __restrict__ rinv, int vec) {
  const int lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  const long long rows = g.ny * g.nz;
  const float qnan = __int_as_float(0x7fc00000);
  for (long long row = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); row < rows; row += warps) {
    const long long z = row / g.ny, y = row - z * g.ny;
    const float* rr = rinv + ((z / g.gz) * g.ncy + y / g.gy) * (long long)g.ncx;
    const float* src = in + row * g.nx;
    float* dst = out + row * g.nx;
    if (vec) {
      const int nq = (int)(g.nx >> 2);
      for (int q = lane; q < nq; q += 32) {
        const int x = 4 * q;
        int c = x / g.gx, r = x - c * g.gx;  // cell and position in it of voxel x
        const float4 v = reinterpret_cast<const float4*>(src)[q];
        float o[4];
        const float vin[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          o[k] = isfinite(vin[k]) ? __fmul_rn(vin[k], __ldg(rr + c)) : qnan;
          if (++r == g.gx) {
            ++c;
            r = 0;
          }
        }
        reinterpret_cast<float4*>(dst)[q] = make_float4(o[0], o[1], o[2], o[3]);
      }
    } else {
      for (int x = lane; x < g.nx; x += 32) {
        const float v = src[x];
        dst[x] = isfinite(v) ? __fmul_rn(v, __ldg(rr + x / g.gx)) : qnan;
      }
    }
  }
}

namespace {
nscale::Geo make_geo(const long long dims[3], const int window[3], const int grid[3]) {
  nscale::Geo g;
  g.nx = dims[0];
  g.ny = dims[1];
  g.nz = dims[2];
  g.wx = window[0];
  g.wy = window[1];
  g.wz = window[2];
  g.gx = grid[0];
  g.gy = grid[1];
  g.gz = grid[2];
  g.ncx = (int)((g.nx + g.gx - 1) / g.gx);
  g.ncy = (int)((g.ny + g.gy - 1) / g.gy);
  g.ncz = (int)((g.nz + g.gz - 1) / g.gz);
  return g;
}
}  // namespace

cudaError_t launch_noise_window(const float* cube, const long long dims[3], const int window[3], const int grid[3],
                                int noise_mode, double* sig_dev, float* rinv_dev, int sms, cudaStream_t s) {
  const nscale::Geo g = make_geo(dims, window, grid);
  const long long cells = (long long)g.ncx * g.ncy * g.ncz;
  const long long most = (long long)nscale::kBlocksPerSm * sms;
  const int blocks = (int)(cells < most ? cells : most);
  k_noise_window<<<blocks, nscale::kThreads, 0, s>>>(cube, g, noise_mode, sig_dev, rinv_dev);
  return cudaGetLastError();
}

cudaError_t launch_noise_apply(const float* cube, const long long dims[3], const int window[3], const int grid[3],
                               float* out, const float* rinv_dev, int sms, cudaStream_t s) {
  const nscale::Geo g = make_geo(dims, window, grid);
  const long long rows = g.ny * g.nz;
  const long long want = (rows + 7) / 8;  // eight warps (rows) per block
  const int blocks = (int)(want < 16LL * sms ? want : 16LL * sms);
  const int vec = (g.nx % 4 == 0) && (reinterpret_cast<uintptr_t>(cube) & 15u) == 0 &&
                  (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
  k_noise_apply<<<blocks, 256, 0, s>>>(cube, out, g, rinv_dev, vec);
  return cudaGetLastError();
}

}  // namespace sc
