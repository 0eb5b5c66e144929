// Linker (SoFiA 2 Sect. 4.3): friends-of-friends components of a detection
// mask, numbered in raster order, with size filters.
//
// The mask is a few per cent full and its detections are runs (maximal row
// segments of mask voxels; single voxels when r_xy = 0), so the work is done
// on bits and runs, numbered in raster order:
//
//   k_lk_pack     the mask as bits, the bits where runs start, and the runs
//                 before every word (within its chunk of 8,192 voxels)
//   k_scan_block  the runs before every chunk, and their number
//   k_lk_init     every run its own root
//   k_lk_union    friends-of-friends between runs, lock-free union-find with
//                 the larger root hung under the smaller, so a component's
//                 root is its first run
//   k_lk_flatten  every run points at its root; roots counted
//   k_lk_number   ids 1, 2, ... in the order of the roots (after a scan)
//   k_lk_extents  bounding box and voxel count of every component
//   k_cc_keep, k_cc_compact  the size filters and the ids that remain
//   k_lk_expand   the labels, written once
//
// The numbers of runs, detections and kept ones stay on the device (Totals):
// the buffers are those of the last call (or a guess), each kernel returns
// where they are too small, and the host, which reads the numbers once at the
// end, grows them and starts over in that case. A cube of 2 M voxels takes
// 175 us so, and took 203 with a stop to size each buffer.
//
// What bounds it: reading the mask (1 byte a voxel) and writing the labels
// (4), then the union's scattered reads of the bits (in L2: an eighth of a
// byte a voxel each). With labels as the union-find's memory and a byte read
// per voxel and neighbour, seven passes over labels and mask, 640 x 640 x
// 1024 voxels (1.2 % set) took 7.1 ms; this form takes 1.6 ms.
#include <climits>
#include <cstdint>

#include "sc_device.cuh"
#include "sc_internal.h"

namespace sc {
namespace link {

constexpr int kThreads = 256;
constexpr int kChunk = 32 * kThreads;  // voxels of a chunk: a mask word per thread
constexpr int kBatch = 512;            // runs of a chunk worked on at a time
constexpr int kFlat = 4096;            // runs per numbering chunk (1024 threads x 4)

struct Geo {
  int nx, ny, nz;
  long long n;
  int rxy, rz;
};

// The mask's runs: bits, run starts, and the runs before each word and chunk.
struct Runs {
  unsigned* bits;
  unsigned* starts;
  unsigned short* word_off;  // within the word's chunk
  int* chunk_off;            // [chunks + 1] after the scan: before each chunk, and their number
};

__device__ __forceinline__ int find_root(int* parent, int x) {
  int p = parent[x];
  while (p != x) {
    const int gp = parent[p];
    if (gp != p) parent[x] = gp;  // path halving (a benign race: any ancestor will do)
    x = p;
    p = gp;
  }
  return x;
}

// Links the trees of a and b, the larger root under the smaller.
__device__ __forceinline__ void unite(int* parent, int a, int b) {
  while (true) {
    a = find_root(parent, a);
    b = find_root(parent, b);
    if (a == b) return;
    if (a > b) {
      const int t = a;
      a = b;
      b = t;
    }
    const int old = atomicCAS(&parent[b], b, a);
    if (old == b) return;  // b was still a root and now hangs under a
    b = old;               // b got a parent meanwhile: retry from there
  }
}

// Index of the run that holds mask voxel v: the runs that start at or before it, less one.
__device__ __forceinline__ int run_of(const Runs& R, long long v) {
  const long long w = v >> 5;
  const unsigned upto = 0xffffffffu >> (31 - (int)(v & 31));
  return __ldg(R.chunk_off + v / kChunk) + (int)__ldg(R.word_off + w) + __popc(__ldg(R.starts + w) & upto) - 1;
}

// Voxels of the run that starts at v, at most `most` (the rest of its row).
__device__ __forceinline__ int run_length(const unsigned* __restrict__ bits, long long v, int most) {
  long long w = v >> 5;
  int at = (int)(v & 31), len = 0;
  while (true) {
    const unsigned gaps = ~(__ldg(bits + w) >> at);  // (zeros shifted in at the top end the word's ones)
    const int ones = gaps ? min(__ffs(gaps) - 1, 32 - at) : 32;
    len += ones;
    if (ones < 32 - at || len >= most) return min(len, most);
    ++w;
    at = 0;
  }
}

}  // namespace link

using link::Geo;
using link::Runs;
using Totals = LinkTotals;

namespace link {
// A thread's word (32 voxels) of the block's chunk: its bits, where runs start,
// and the runs before it and in all of the chunk. A run starts at a set voxel
// whose predecessor is not set or lies in another row. All threads call it.
struct Word {
  unsigned bits, starts;
  int off, total;
};
__device__ __forceinline__ Word pack_word(const uint8_t* __restrict__ mask, const Geo& g, int* part) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long v0 = 32 * ((long long)blockIdx.x * kThreads + tid);
  unsigned bits = 0u;
  if (v0 + 32 <= g.n && (reinterpret_cast<uintptr_t>(mask) & 15u) == 0) {
    const uint4* m = reinterpret_cast<const uint4*>(mask + v0);
    const uint4 a = __ldg(m), b = __ldg(m + 1);
    bits = nonzero_bits(a.x) | nonzero_bits(a.y) << 4 | nonzero_bits(a.z) << 8 | nonzero_bits(a.w) << 12 |
           nonzero_bits(b.x) << 16 | nonzero_bits(b.y) << 20 | nonzero_bits(b.z) << 24 | nonzero_bits(b.w) << 28;
  } else if (v0 < g.n) {
    for (int i = 0; i < 32 && v0 + i < g.n; ++i) bits |= (mask[v0 + i] ? 1u : 0u) << i;
  }
  unsigned before = __shfl_up_sync(0xffffffffu, bits, 1) >> 31;
  if (lane == 0) before = (v0 > 0 && v0 <= g.n && mask[v0 - 1]) ? 1u : 0u;
  unsigned starts = bits;
  if (g.rxy >= 1) {
    unsigned row = 0u;  // voxels with x = 0
    const unsigned x0 = (unsigned)v0 % (unsigned)g.nx;
    for (unsigned p = x0 ? (unsigned)g.nx - x0 : 0u; p < 32u; p += (unsigned)g.nx) row |= 1u << p;
    starts = bits & (~(bits << 1 | before) | row);
  }
  const int c = __popc(starts);
  int x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) part[warp] = x;
  __syncthreads();
  int off = x - c, total = 0;
  for (int k = 0; k < kThreads / 32; ++k) {
    if (k < warp) off += part[k];
    total += part[k];
  }
  return Word{bits, starts, off, total};
}
}  // namespace link

// A block per chunk, a mask word per thread.
__global__ void __launch_bounds__(link::kThreads) k_lk_pack(const uint8_t* __restrict__ mask, Geo g, Runs R) {
  using namespace link;
  __shared__ int part[kThreads / 32];
  const Word a = pack_word(mask, g, part);
  const long long w = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (32 * w < g.n) {
    R.bits[w] = a.bits;
    R.starts[w] = a.starts;
    R.word_off[w] = (unsigned short)a.off;
  }
  if (threadIdx.x == 0) R.chunk_off[blockIdx.x] = a.total;
}

// Exclusive scan of a[0 .. len) in place by one block of 1024 threads, eight
// values a thread, the next eight loaded meanwhile; a[len] and *total receive
// the sum. The length is t.scan_length(of, per, len): nothing happens where
// the totals it comes from do not fit.
__global__ void __launch_bounds__(1024) k_scan_block(int* a, long long len, Totals t, int of, int per, int* total) {
  __shared__ int part[32];
  constexpr int kPer = 8;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  len = t.scan_length(of, per, len);
  if (len < 0) return;
  int carry = 0;
  int nx[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) nx[k] = kPer * tid + k < len ? a[kPer * tid + k] : 0;
  for (long long t0 = 0; t0 < len; t0 += 1024 * kPer) {
    const long long i0 = t0 + kPer * tid, j0 = i0 + 1024 * kPer;
    int v[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      v[k] = nx[k];
      sum += v[k];
      nx[k] = j0 + k < len ? a[j0 + k] : 0;
    }
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) part[warp] = x;
    __syncthreads();
    const int p = part[lane];
    int run = carry + __reduce_add_sync(0xffffffffu, lane < warp ? p : 0) + x - sum;
    carry += __reduce_add_sync(0xffffffffu, p);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      if (i0 + k < len) a[i0 + k] = run;
      run += v[k];
    }
    __syncthreads();  // the parts are read before the next tile writes them
  }
  if (tid == 0) {
    a[len] = carry;
    *total = carry;
  }
}

__global__ void k_lk_init(int* parent, Totals t) {
  if (!t.runs_fit()) return;
  const int n = t.n[0];
  for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < n; r += (long long)gridDim.x * blockDim.x)
    parent[r] = (int)r;
}

namespace link {
// Runs `from` .. of a chunk (at most kBatch) with their coordinates, in shared
// memory: the first voxel, x and x + length - 1, y, z.
struct Batch {
  unsigned short at[kChunk];  // places of the chunk's runs in it
  int xs[kBatch], xe[kBatch], y[kBatch], z[kBatch];
};

// The places of the chunk's runs (their number is returned). All threads call it.
__device__ __forceinline__ int chunk_runs(const Runs& R, const Geo& g, Batch* B) {
  const int tid = threadIdx.x;
  const int n = __ldg(R.chunk_off + blockIdx.x + 1) - __ldg(R.chunk_off + blockIdx.x);
  if (n == 0) return 0;
  const long long w = (long long)blockIdx.x * kThreads + tid;
  if (32 * w < g.n) {
    unsigned s = __ldg(R.starts + w);
    for (int i = __ldg(R.word_off + w); s; ++i, s &= s - 1u) B->at[i] = (unsigned short)(32 * tid + __ffs(s) - 1);
  }
  __syncthreads();
  return n;
}

__device__ __forceinline__ void load_batch(const Runs& R, const Geo& g, int from, int count, Batch* B) {
  const unsigned plane = (unsigned)g.nx * (unsigned)g.ny;  // (fewer than 2^31 voxels in all)
  for (int i = threadIdx.x; i < count; i += kThreads) {
    const unsigned v = blockIdx.x * (unsigned)kChunk + B->at[from + i];
    const unsigned z = v / plane, rem = v - z * plane, y = rem / (unsigned)g.nx, x = rem - y * (unsigned)g.nx;
    B->z[i] = (int)z;
    B->y[i] = (int)y;
    B->xs[i] = (int)x;
    B->xe[i] = (int)x + (g.rxy >= 1 ? run_length(R.bits, v, g.nx - (int)x) : 1) - 1;
  }
  __syncthreads();
}
}  // namespace link

// A block per chunk. Every run links to the next run of its row within reach
// and to every run that meets its reach in each friend row after it in raster
// order (dz > 0, or dz == 0 and dy > 0); the other half of the relation is the
// mirror of these. The pairs (run, friend row) go to the threads side by side.
__global__ void __launch_bounds__(link::kThreads) k_lk_union(Geo g, Runs R, int* parent, Totals t) {
  using namespace link;
  __shared__ Batch B;
  __shared__ int reach[kLinkMaxRadius + 1];  // largest |dx| with dx^2 + dy^2 <= r_xy^2
  const int tid = threadIdx.x;
  if (!t.runs_fit()) return;
  if (tid <= g.rxy) {
    int d = 0;
    while ((d + 1) * (d + 1) + tid * tid <= g.rxy * g.rxy) ++d;
    reach[tid] = d;
  }
  const int n = chunk_runs(R, g, &B);
  if (n == 0) return;
  const int first = __ldg(R.chunk_off + blockIdx.x);
  const int wide = 2 * g.rxy + 1, rows = 1 + g.rxy + g.rz * wide;  // the run's own row first
  for (int from = 0; from < n; from += kBatch) {
    const int count = min(kBatch, n - from);
    load_batch(R, g, from, count, &B);
    for (int it = tid; it < count * rows; it += kThreads) {
      const int k = it / count, i = it - k * count;
      const int me = first + from + i;
      int dz = 0, dy = k, lo, hi;
      if (k > g.rxy) {
        dz = 1 + (k - 1 - g.rxy) / wide;
        dy = (k - 1 - g.rxy) % wide - g.rxy;
      }
      const int z = B.z[i] + dz, y = B.y[i] + dy;
      if (z >= g.nz || y < 0 || y >= g.ny) continue;
      if (k == 0) {  // (further runs in reach chain to the next one)
        lo = B.xe[i] + 2;
        hi = min(g.nx - 1, B.xe[i] + g.rxy);
      } else {
        const int d = reach[abs(dy)];
        lo = max(0, B.xs[i] - d);
        hi = min(g.nx - 1, B.xe[i] + d);
      }
      if (lo > hi) continue;
      const long long row = ((long long)z * g.ny + y) * g.nx, a = row + lo, b = row + hi;
      for (long long w = a >> 5; w <= b >> 5; ++w) {
        unsigned in = __ldg(R.bits + w);
        if (w == a >> 5) in &= 0xffffffffu << (a & 31);
        if (w == b >> 5) in &= 0xffffffffu >> (31 - (b & 31));
        if (!in) continue;
        // runs that start in the window, and one that reaches into it
        unsigned s = __ldg(R.starts + w) & in;
        if (w == a >> 5 && (in >> (a & 31) & 1u)) s |= 1u << (a & 31);
        if (k == 0) s &= 0u - s;
        for (; s; s &= s - 1u) unite(parent, me, run_of(R, 32 * w + __ffs(s) - 1));
        if (k == 0) break;
      }
    }
    __syncthreads();  // the batch is overwritten by the next one
  }
}

// Every run points at its root afterwards, and counts[block] holds the roots
// of each kFlat runs. The walks only read: halving paths here could overwrite
// a run's final root with an older ancestor read before it. A run is a root
// exactly when its walk ends at itself, whatever other threads write.
__global__ void __launch_bounds__(1024) k_lk_flatten(int* parent, int* __restrict__ counts, Totals t) {
  __shared__ int s_roots;
  if (!t.runs_fit()) return;
  const long long nruns = t.n[0];
  for (long long blk = blockIdx.x; blk * link::kFlat < nruns; blk += gridDim.x) {
    if (threadIdx.x == 0) s_roots = 0;
    __syncthreads();
    const long long base = blk * link::kFlat + 4LL * threadIdx.x;
    int c = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const long long r = base + k;
      if (r < nruns) {
        int x = (int)r, p = parent[r];
        while (p != x) {
          x = p;
          p = parent[x];
        }
        if (x == (int)r) ++c;
        else parent[r] = x;
      }
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&s_roots, c);
    __syncthreads();
    if (threadIdx.x == 0) counts[blk] = s_roots;
  }
}

// parent[root] = -(id) with ids 1, 2, ... in the order of the roots.
__global__ void __launch_bounds__(1024) k_lk_number(int* parent, const int* __restrict__ off, Totals t) {
  __shared__ int part[32];
  if (!t.all_fit()) return;
  const long long nruns = t.n[0];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (long long blk = blockIdx.x; blk * link::kFlat < nruns; blk += gridDim.x) {
    const long long base = blk * link::kFlat + 4LL * tid;
    bool root[4];
    int c = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const long long r = base + k;
      root[k] = r < nruns && parent[r] == (int)r;
      c += root[k] ? 1 : 0;
    }
    int x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) part[warp] = x;
    __syncthreads();
    const int p = part[lane];
    int id = off[blk] + __reduce_add_sync(0xffffffffu, lane < warp ? p : 0) + x - c;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (root[k]) parent[base + k] = -(++id);
    __syncthreads();  // the parts are read before the next chunk writes them
  }
}

// A block per chunk: every run's component id to run_id, and the bounding box
// and voxel count of each component, ext[7 * (id - 1) ...] = x_min, x_max,
// y_min, y_max, z_min, z_max, count. Lanes of a warp with the same id combine
// first, so a component's seven words see one atomic per group.
__global__ void __launch_bounds__(link::kThreads) k_lk_extents(Geo g, Runs R, const int* __restrict__ parent,
                                                               int* __restrict__ run_id, int* ext, Totals t) {
  using namespace link;
  __shared__ Batch B;
  if (!t.all_fit()) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const int n = chunk_runs(R, g, &B);
  if (n == 0) return;
  const int first = __ldg(R.chunk_off + blockIdx.x);
  for (int from = 0; from < n; from += kBatch) {
    const int count = min(kBatch, n - from);
    load_batch(R, g, from, count, &B);
    for (int i0 = tid - lane; i0 < count; i0 += kThreads) {
      const int i = i0 + lane;
      int id = 0, xs = 0, xe = 0, y = 0, z = 0;
      if (i < count) {
        const int r = first + from + i, p = __ldg(parent + r);
        id = p < 0 ? -p : -__ldg(parent + p);
        run_id[r] = id;
        xs = B.xs[i];
        xe = B.xe[i];
        y = B.y[i];
        z = B.z[i];
      }
      const unsigned peers = __match_any_sync(0xffffffffu, id);  // lanes of the same component
      const int xmin = __reduce_min_sync(peers, xs), xmax = __reduce_max_sync(peers, xe);
      const int ymin = __reduce_min_sync(peers, y), ymax = __reduce_max_sync(peers, y);
      const int zmin = __reduce_min_sync(peers, z), zmax = __reduce_max_sync(peers, z);
      const int voxels = __reduce_add_sync(peers, xe - xs + 1);
      if (id > 0 && lane == __ffs(peers) - 1) {
        int* e = ext + 7LL * (id - 1);
        atomicMin(e + 0, xmin);
        atomicMax(e + 1, xmax);
        atomicMin(e + 2, ymin);
        atomicMax(e + 3, ymax);
        atomicMin(e + 4, zmin);
        atomicMax(e + 5, zmax);
        atomicAdd(e + 6, voxels);
      }
    }
    __syncthreads();  // the batch is overwritten by the next one
  }
}

__global__ void k_cc_ext_init(int* ext, Totals t) {
  if (!t.all_fit()) return;
  const int ncomp = t.n[1];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ncomp; i += gridDim.x * blockDim.x) {
    int* e = ext + 7LL * i;
    e[0] = e[2] = e[4] = INT_MAX;
    e[1] = e[3] = e[5] = -1;
    e[6] = 0;
  }
}

__global__ void k_cc_keep(const int* __restrict__ ext, Totals t, int min_xy, int min_z, int max_xy, int max_z,
                          int* keep, int* flag) {
  if (!t.all_fit()) return;
  const int ncomp = t.n[1];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ncomp; i += gridDim.x * blockDim.x) {
    const int* e = ext + 7LL * i;
    const int sx = e[1] - e[0] + 1, sy = e[3] - e[2] + 1, sz = e[5] - e[4] + 1;
    bool k = sx >= min_xy && sy >= min_xy && sz >= min_z;
    if (max_xy > 0) k = k && sx <= max_xy && sy <= max_xy;
    if (max_z > 0) k = k && sz <= max_z;
    keep[i] = flag[i] = k ? 1 : 0;
  }
}

// After the exclusive scan of the keep flags: the kept rows moved to the
// front of out (ids 1 .. kept), and new_id[i] = id of detection i + 1 or 0.
__global__ void k_cc_compact(const int* __restrict__ ext, const int* keep_flag, const int* __restrict__ keep_off,
                             Totals t, int* out, int* new_id) {
  if (!t.all_fit()) return;
  const int ncomp = t.n[1];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ncomp; i += gridDim.x * blockDim.x) {
    if (keep_flag[i]) {
      const int j = keep_off[i];
      for (int c = 0; c < 7; ++c) out[7LL * j + c] = ext[7LL * i + c];
      new_id[i] = j + 1;
    } else {
      new_id[i] = 0;
    }
  }
}

// The labels, four voxels a thread: 0, or the new id of the voxel's component.
__global__ void __launch_bounds__(256) k_lk_expand(Geo g, Runs R, const int* __restrict__ run_id,
                                                   const int* __restrict__ new_id, int* __restrict__ lab, Totals t) {
  if (!t.all_fit()) return;
  const bool vec = (reinterpret_cast<uintptr_t>(lab) & 15u) == 0;
  const long long quads = (g.n + 3) / 4;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < quads; q += (long long)gridDim.x * blockDim.x) {
    const long long v = 4 * q;
    const unsigned in = __ldg(R.bits + (v >> 5)) >> (v & 31) & 0xfu;
    int l[4] = {0, 0, 0, 0};
    if (in) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (in >> k & 1u) l[k] = __ldg(new_id + __ldg(run_id + link::run_of(R, v + k)) - 1);
    }
    if (vec && v + 4 <= g.n) {
      *reinterpret_cast<int4*>(lab + v) = make_int4(l[0], l[1], l[2], l[3]);
    } else {
      for (int k = 0; k < 4 && v + k < g.n; ++k) lab[v + k] = l[k];
    }
  }
}

// The same where the bits lie in the memory of the labels: they are taken from
// the mask once more, a block per chunk and a word per thread.
__global__ void __launch_bounds__(link::kThreads) k_lk_expand_mask(const uint8_t* __restrict__ mask, Geo g,
                                                                   const int* __restrict__ chunk_off,
                                                                   const int* __restrict__ run_id,
                                                                   const int* __restrict__ new_id,
                                                                   int* __restrict__ lab, Totals t) {
  using namespace link;
  __shared__ int part[kThreads / 32];
  if (!t.all_fit()) return;
  const Word a = pack_word(mask, g, part);
  const long long v0 = 32 * ((long long)blockIdx.x * kThreads + threadIdx.x);
  int run = __ldg(chunk_off + blockIdx.x) + a.off - 1;
  for (int i = 0; i < 32 && v0 + i < g.n; ++i) {
    run += (int)(a.starts >> i & 1u);
    lab[v0 + i] = a.bits >> i & 1u ? __ldg(new_id + __ldg(run_id + run) - 1) : 0;
  }
}

// ---------------------------------------------------------------------------
namespace {
inline int grid_for(long long n, int sms, int threads) {
  const long long want = (n + threads - 1) / threads;
  const long long cap = 16LL * sms;
  return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}
size_t up16(size_t v) { return (v + 15) & ~(size_t)15; }
Runs runs_at(void* bits, int* chunk_off, long long n) {
  const size_t words = (size_t)((n + 31) / 32);
  unsigned char* b = static_cast<unsigned char*>(bits);
  Runs R;
  R.bits = reinterpret_cast<unsigned*>(b);
  R.starts = reinterpret_cast<unsigned*>(b + up16(4 * words));
  R.word_off = reinterpret_cast<unsigned short*>(b + 2 * up16(4 * words));
  R.chunk_off = chunk_off;
  return R;
}
long long chunks_of(long long n) { return (n + link::kChunk - 1) / link::kChunk; }
}  // namespace

size_t link_bits_bytes(long long n) {
  const size_t words = (size_t)((n + 31) / 32);
  return 2 * up16(4 * words) + up16(2 * words);
}
size_t link_chunk_bytes(long long n) { return up16(4 * (size_t)(chunks_of(n) + 1)); }
size_t link_runs_bytes(long long nruns) {
  return up16(4 * (size_t)(2 * nruns + (nruns + link::kFlat - 1) / link::kFlat + 1));
}
size_t link_comp_bytes(long long ncomp) { return 4 * (size_t)(16 * ncomp + 1); }

cudaError_t launch_link(const uint8_t* mask, const long long dims[3], int r_xy, int r_z, int min_xy, int min_z,
                        int max_xy, int max_z, void* bits, int* chunk_off, int* runs, long long max_runs, int* comp,
                        long long max_comp, int* totals, int* lab, int** ext_out, int sms, cudaStream_t s,
                        int* launches) {
  const Geo g{(int)dims[0], (int)dims[1], (int)dims[2], dims[0] * dims[1] * dims[2], r_xy, r_z};
  const Runs R = runs_at(bits ? bits : lab, chunk_off, g.n);
  const Totals t{totals, max_runs, max_comp};
  const long long chunks = chunks_of(g.n), flat = (max_runs + link::kFlat - 1) / link::kFlat;
  int *const parent = runs, *const run_id = runs + max_runs, *const counts = runs + 2 * max_runs;
  // per component: extents, kept extents, keep flags (scanned: one more), new ids
  int *const ext = comp, *const kept = ext + 7 * max_comp, *const new_id = kept + 7 * max_comp;
  int* const keep = new_id + max_comp;
  const int flat_grid = (int)(flat < 8LL * sms ? flat : 8LL * sms);
  // a total that a kernel leaves unwritten (what it counts did not fit) is 0
  const cudaError_t e = cudaMemsetAsync(totals, 0, 3 * sizeof(int), s);
  if (e != cudaSuccess) return e;
  k_lk_pack<<<(unsigned)chunks, link::kThreads, 0, s>>>(mask, g, R);
  k_scan_block<<<1, 1024, 0, s>>>(R.chunk_off, chunks, t, LINK_SCAN_LEN, 1, totals);
  k_lk_init<<<grid_for(max_runs, sms, 256), 256, 0, s>>>(parent, t);
  k_lk_union<<<(unsigned)chunks, link::kThreads, 0, s>>>(g, R, parent, t);
  k_lk_flatten<<<flat_grid, 1024, 0, s>>>(parent, counts, t);
  k_scan_block<<<1, 1024, 0, s>>>(counts, 0, t, LINK_SCAN_RUNS, link::kFlat, totals + 1);
  k_cc_ext_init<<<grid_for(max_comp, sms, 256), 256, 0, s>>>(ext, t);
  k_lk_number<<<flat_grid, 1024, 0, s>>>(parent, counts, t);
  k_lk_extents<<<(unsigned)chunks, link::kThreads, 0, s>>>(g, R, parent, run_id, ext, t);
  k_cc_keep<<<grid_for(max_comp, sms, 256), 256, 0, s>>>(ext, t, min_xy, min_z, max_xy, max_z, keep, new_id);
  k_scan_block<<<1, 1024, 0, s>>>(keep, 0, t, LINK_SCAN_COMPS, 1, totals + 2);
  k_cc_compact<<<grid_for(max_comp, sms, 256), 256, 0, s>>>(ext, new_id, keep, t, kept, new_id);
  if (bits) k_lk_expand<<<grid_for((g.n + 3) / 4, sms, 256), 256, 0, s>>>(g, R, run_id, new_id, lab, t);
  else k_lk_expand_mask<<<(unsigned)chunks, link::kThreads, 0, s>>>(mask, g, R.chunk_off, run_id, new_id, lab, t);
  *launches = 13;
  *ext_out = kept;
  return cudaGetLastError();
}

}  // namespace sc
