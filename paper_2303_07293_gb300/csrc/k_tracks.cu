// k_tracks.cu — linking the per-velocity detections of one object into tracks.
//
// The search reports per-velocity local maxima (Sec. 2.1); a moving object
// yields detections at neighbouring trial velocities and positions, and the
// tracker reports tracks with speed, position angle, pixel coordinates and
// S/N.  Two detections of a field are linked when their pixels differ by at
// most r_xy in x and y and their velocity indices by at most r_v in a and b;
// a track is a connected component, represented by its detection of highest
// S/N (ties: the first in (field, k, y, x) order) with the component's size.
//
// The detections arrive sorted by (field, k, y, x), so a detection's
// neighbours at one velocity are a contiguous run.  A table of where each
// velocity's detections begin (built where it is not much larger than the
// list) leaves a few to look at; without it, or where a velocity has many, a
// binary search on the packed keys finds the rows.  Every pair is met once,
// from its earlier detection.  58 717 detections of a 121^2 grid: 439 us with
// five binary searches over the records for each of nine velocities, 172 with
// the table's 10.  Components come from a lock-free union-find
// (a root is hooked under the smaller root with a compare-and-swap, so every
// component's root is its first detection); tracks are listed in root order.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "st_internal.h"

namespace st {

namespace {

__device__ __forceinline__ uint64_t key_of(const st_candidate& c) {
  return cand_key(c.field, c.k, c.y, c.x);
}

// First index in [lo, hi) whose key is >= want (hi: none).
__device__ __forceinline__ int lower_bound(const uint64_t* __restrict__ keys, int lo, int hi,
                                           uint64_t want) {
  while (lo < hi) {
    const int mid = lo + (hi - lo) / 2;
    if (__ldg(keys + mid) < want) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

__device__ int find_root(int* parent, int x) {
  for (;;) {
    const int p = ((volatile int*)parent)[x];
    if (p == x) return x;
    const int gp = ((volatile int*)parent)[p];
    if (gp != p) ((volatile int*)parent)[x] = gp;  // path halving (stays inside the set)
    x = p;
  }
}

__device__ void unite(int* parent, int a, int b) {
  for (;;) {
    int ra = find_root(parent, a), rb = find_root(parent, b);
    if (ra == rb) return;
    if (ra > rb) {
      const int t = ra;
      ra = rb;
      rb = t;
    }
    // hook the larger root under the smaller one
    const int old = atomicCAS(&parent[rb], rb, ra);
    if (old == rb) return;
    b = old;  // rb gained a parent meanwhile: retry from there
    a = ra;
  }
}

__global__ void k_link_init(const st_candidate* __restrict__ c, uint64_t* __restrict__ keys,
                            int* parent, unsigned long long* best, int* count, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  keys[i] = key_of(c[i]);
  parent[i] = (int)i;
  best[i] = 0ull;
  count[i] = 0;
}

// start[base[field] + k]: the first detection of (field, k) or later ones, for
// all velocities of all fields and one past the last.
__global__ void k_link_index(const uint64_t* __restrict__ keys, int n,
                             const FieldDev* __restrict__ fds, int n_fields, int64_t n_start,
                             int* __restrict__ start) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v > n_start) return;
  int64_t base = 0;
  int f = 0;
  while (f < n_fields && v - base >= (int64_t)fds[f].nvx * fds[f].nvy) {
    base += (int64_t)fds[f].nvx * fds[f].nvy;
    ++f;
  }
  start[v] = f < n_fields ? lower_bound(keys, 0, n, cand_key(f, (int)(v - base), 0, 0)) : n;
}

constexpr int kScan = 24;  // detections of a velocity that are looked at one by one

__global__ void k_link(const uint64_t* __restrict__ keys, int n, const FieldDev* __restrict__ fds,
                       const int* __restrict__ start, int r_xy, int r_v, int* parent) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  const uint64_t me = keys[i];
  const int field = (int)(me >> 56), k = (int)((me >> 30) & 0x3ffffffu);
  const int my_y = (int)((me >> 15) & 0x7fffu), my_x = (int)(me & 0x7fffu);
  const FieldDev& fd = fds[field];
  const int nvx = fd.nvx, nvy = fd.nvy;
  const int a = k % nvx, b = k / nvx;
  const int xlo = max(my_x - r_xy, 0), xhi = min(my_x + r_xy, fd.W - 1);
  const int ylo = max(my_y - r_xy, 0), yhi = min(my_y + r_xy, fd.H - 1);
  int64_t base = 0;
  if (start)
    for (int f = 0; f < field; ++f) base += (int64_t)fds[f].nvx * fds[f].nvy;
  // velocities at or after this one's in the list's order
  for (int b2 = b; b2 <= min(b + (int64_t)r_v, (int64_t)nvy - 1); ++b2) {
    for (int a2 = b2 == b ? a : max((int64_t)a - r_v, (int64_t)0);
         a2 <= min(a + (int64_t)r_v, (int64_t)nvx - 1); ++a2) {
      const int k2 = b2 * nvx + a2;
      int lo = i + 1, hi = n;
      if (start) {
        lo = max(__ldg(start + base + k2), i + 1);
        hi = __ldg(start + base + k2 + 1);
      }
      if (hi - lo <= kScan) {
        for (int j = lo; j < hi; ++j) {
          const uint64_t q = __ldg(keys + j);
          const int y = (int)((q >> 15) & 0x7fffu), x = (int)(q & 0x7fffu);
          if ((q >> 30) == (cand_key(field, k2, 0, 0) >> 30) && y >= ylo && y <= yhi &&
              x >= xlo && x <= xhi)
            unite(parent, i, j);
        }
        continue;
      }
      for (int y2 = ylo; y2 <= yhi; ++y2) {
        const uint64_t last = cand_key(field, k2, y2, xhi);
        lo = lower_bound(keys, lo, hi, cand_key(field, k2, y2, xlo));
        for (; lo < hi; ++lo) {
          if (__ldg(keys + lo) > last) break;
          unite(parent, i, lo);
        }
      }
    }
  }
}

// Order-preserving map of an FP32 value to uint32 (larger float, larger key).
__device__ __forceinline__ uint32_t ordered(float v) {
  const uint32_t u = __float_as_uint(v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

constexpr int kBlock = 256;

// Best detection and size of each component; the block's number of roots.
__global__ void __launch_bounds__(kBlock)
    k_link_reduce(const st_candidate* __restrict__ c, int64_t n, int* parent,
                  unsigned long long* best, int* count, int* __restrict__ block_roots) {
  const int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  bool root = false;
  if (i < n) {
    const int r = find_root(parent, (int)i);
    // highest S/N, then the smallest index
    const unsigned long long key =
        ((unsigned long long)ordered(c[i].snr) << 32) | (0xffffffffu - (uint32_t)i);
    atomicMax(&best[r], key);
    atomicAdd(&count[r], 1);
    root = r == (int)i;
  }
  const int roots = __syncthreads_count(root);
  if (threadIdx.x == 0) block_roots[blockIdx.x] = roots;
}

// Exclusive prefix sums of the blocks' roots in place (one block); the total
// after them.
__global__ void __launch_bounds__(1024) k_link_scan(int* __restrict__ v, int blocks) {
  __shared__ int sh[32];
  int carry = 0;
  for (int b0 = 0; b0 < blocks; b0 += 1024) {
    const int b = b0 + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x = b < blocks ? v[b] : 0;
    int s = x;
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, s, d);
      if (lane >= d) s += o;
    }
    if (lane == 31) sh[warp] = s;
    __syncthreads();
    if (warp == 0) {
      int t = sh[lane];
      for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, t, d);
        if (lane >= d) t += o;
      }
      sh[lane] = t;
    }
    __syncthreads();
    const int before = carry + (warp ? sh[warp - 1] : 0) + s - x;
    if (b < blocks) v[b] = before;
    carry += sh[31];
    __syncthreads();
  }
  if (threadIdx.x == 0) v[blocks] = carry;
}

__global__ void __launch_bounds__(kBlock)
    k_link_emit(const st_candidate* __restrict__ c, int64_t n, const FieldDev* __restrict__ fds,
                const double* __restrict__ grid, const int* __restrict__ parent,
                const int* __restrict__ block_roots, const unsigned long long* best,
                const int* count, st_track* __restrict__ out, int64_t cap) {
  __shared__ int warp_roots[kBlock / 32];
  const int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool root = i < n && parent[i] == (int)i;
  const unsigned m = __ballot_sync(0xffffffffu, root);
  if (lane == 0) warp_roots[warp] = __popc(m);
  __syncthreads();
  int64_t pos = block_roots[blockIdx.x] + __popc(m & ((1u << lane) - 1u));
  for (int w = 0; w < warp; ++w) pos += warp_roots[w];
  if (!root || pos >= cap) return;
  const int64_t rep = 0xffffffffu - (uint32_t)(best[i] & 0xffffffffull);
  const st_candidate r = c[rep];
  const FieldDev& fd = fds[r.field];
  const double* g = grid + 4 * r.field;  // vx0, dvx, vy0, dvy
  const double vx = __dadd_rn(g[0], __dmul_rn((double)(r.k % fd.nvx), g[1]));
  const double vy = __dadd_rn(g[2], __dmul_rn((double)(r.k / fd.nvx), g[3]));
  double pa = atan2(-vx, -vy) * (180.0 / 3.14159265358979323846);
  if (pa < 0.0) pa += 360.0;
  st_track t;
  t.x = r.x;
  t.y = r.y;
  t.k = r.k;
  t.field = r.field;
  t.stack = r.stack;
  t.snr = r.snr;
  t.n_cov = r.n_cov;
  t.members = count[i];
  t.vx = (float)vx;
  t.vy = (float)vy;
  t.speed = (float)hypot(vx, vy);
  t.pa = (float)pa;
  out[pos] = t;
}

}  // namespace

namespace {
// Entries of the table of velocities: none where the list is much shorter
// (a search of the keys a velocity costs about 20 loads).
int64_t link_starts(int64_t n, int64_t velocities) {
  return velocities <= 8 * n + 65536 ? velocities + 1 : 0;
}
}  // namespace

int64_t link_workspace_bytes(int64_t n, int64_t velocities) {
  return n * (int64_t)(sizeof(uint64_t) + sizeof(unsigned long long) + 2 * sizeof(int)) +
         ((n + kBlock - 1) / kBlock + 1 + link_starts(n, velocities)) * (int64_t)sizeof(int);
}

int launch_link_tracks(const st_candidate* c, int64_t n, const FieldDev* fds, int n_fields,
                       int64_t velocities, const double* grid, int r_xy, int r_v, void* ws,
                       st_track* out, int64_t cap, int* h_count, int64_t* n_tracks,
                       cudaStream_t s) {
  *n_tracks = 0;
  if (n <= 0) return 0;
  const unsigned blocks = (unsigned)((n + kBlock - 1) / kBlock);
  unsigned long long* best = (unsigned long long*)ws;
  uint64_t* keys = (uint64_t*)(best + n);
  int* parent = (int*)(keys + n);
  int* count = parent + n;
  int* block_roots = count + n;  // blocks + 1
  const int64_t n_start = link_starts(n, velocities);
  int* start = n_start ? block_roots + blocks + 1 : nullptr;
  int launches = 5;
  k_link_init<<<blocks, kBlock, 0, s>>>(c, keys, parent, best, count, n);
  if (start) {
    k_link_index<<<(unsigned)((n_start + 255) / 256), 256, 0, s>>>(keys, (int)n, fds, n_fields,
                                                                   velocities, start);
    ++launches;
  }
  k_link<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(keys, (int)n, fds, start, r_xy, r_v, parent);
  k_link_reduce<<<blocks, kBlock, 0, s>>>(c, n, parent, best, count, block_roots);
  k_link_scan<<<1, 1024, 0, s>>>(block_roots, (int)blocks);
  k_link_emit<<<blocks, kBlock, 0, s>>>(c, n, fds, grid, parent, block_roots, best, count, out,
                                        cap);
  cudaMemcpyAsync(h_count, block_roots + blocks, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (cudaStreamSynchronize(s) != cudaSuccess) return -1;
  *n_tracks = *h_count;
  return launches;
}

}  // namespace st
