// k_stack_runs.cu — register-window shift-and-stack kernel that sums frames
// with equal relative shifts once (nearest sampling), for sm_103a.
//
// The search of Sec. 1 / Sec. 2.1 adds, for every trial velocity, N shifted
// frames per pixel.  Within a tile of adjacent velocities most of those
// additions repeat each other: on one frame the 4 y-velocities of a tile read
// the same pixel column at row offsets that form one of 15 staircases, and
// over a night's frames few staircases occur (about 9 for steps of at most
// half a pixel).  So the frames of a tile are taken sorted by staircase
// (k_run_order), and a thread adds the window of its column (8 rows and the
// staircase's height) into ONE running sum per x-velocity.  Where the
// staircase changes, mostly one y-velocity's offset does: the running sum at
// the old offset is added to its accumulators and the sum at the new offset
// subtracted; at the end the sum, at the last offset, is added to all.  Per
// frame and x-velocity that is about 4.7 paired adds instead of 16, and a
// window column is loaded once for all adjacent x-velocities whose shifts
// agree.
//
// The additions of one output are then not in frame order, and the resolver's
// bit-exact sums are: the kernel is a filter.  It keeps every point whose sum
// reaches the threshold less a margin, a bound of the rounding of both orders
// (run_margin in st_internal.h), and the resolver re-forms each kept point's sum in frame order and applies the
// threshold itself, as it does for the other stack kernels.
//
// * Item: 32 x 32 pixels, up to 16 x-velocities (4 groups of 4; a field's
//   groups are spread evenly over its tiles) and 4 y-velocities.  16 consumer
//   warps: warp = (group, row quarter); lane l owns column X0 + l.  A producer
//   warp stages frames by TMA (box 44 x 35 FP32) in a ring of 2 stages of 16
//   frames, one CTA per SM, as in k_stack_fast.cu.  (8 groups x 2 row halves
//   leave more warps without a group: 1024^2 x 64, 161^2 velocities, 62.9 ms
//   against 56.2.)
// * Per frame a warp reads one word: the window's offset in the ring, which
//   of the 4 x-velocities step to the next column (3 bits and a direction),
//   the staircase's height and whether its run ends.  A switch on (steps,
//   height) picks straight-line code for 1..4 columns of 8..11 rows.
// * The accumulators (4 x 4 velocities x 8 rows a thread) are read and written
//   only at run ends, so they live in tensor memory (128 of the 512 columns
//   per warp: 16 warps fill the SM's 256 KB); the registers hold the run sums
//   (4 x 12 rows).
//
// What bounds it: shared-memory reads.  Per 4096 additions of the plain
// definition a warp needs about 15 row loads (32 lanes x 4 bytes, one
// wavefront each), 18 paired adds and 15 other instructions, against 64
// paired adds at the FP32 pipe's rate alone; 86 instructions in all on 64
// frames, 75 on 256 (the ends of runs, stages and items are the rest), issue
// slots 53 % and shared-memory wavefronts 43 % busy on 64 frames (58 % on 256), where
// warps wait for the slowest at each stage.  Measured against the frame-order kernel
// (rates in additions of the plain definition, 40.3 T/s the FP32 pipe's):
// 1024^2 x 64, 161^2 velocities 86.7 -> 56.7 ms (30.7 T/s); 2048^2 x 256, 101^2
// 491 -> 246 ms (44.6 T/s); six FP16 fields of 46..120 frames, 61^2 85.7 -> 47.5
// ms.  Stages of 8 frames: 62.3, 273, 51.0 ms.
#include <cuda.h>
#include <cuda_runtime.h>

#include <climits>
#include <new>

#include <type_traits>

#include "st_pending.cuh"
#include "st_runs.inc"
#include "st_stack_field.cuh"
#include "st_tma.cuh"

namespace st {

namespace {

constexpr int kG = 4;            // x-velocities per group (one warp's)
constexpr int kXG = 4;           // groups per item
constexpr int kRG = 4;           // row quarters per item
constexpr int kRows = 8;         // rows per warp
constexpr int kTY = kRG * kRows;
constexpr int kF = 16, kS = 2;   // frames per stage, stages of the ring
constexpr int kCW = kXG * kRG;   // consumer warps
constexpr int kThreads = 32 * (kCW + 1);
constexpr int kBoxH = kTY + 3;
constexpr int kItemSlots = 8;
constexpr uint32_t kAccCols = kG * kMB * kRows;  // tensor-memory columns of a warp: 128
constexpr int kShiftBias = 32768;

template <typename T>
constexpr int box_w() { return sizeof(T) == 4 ? 44 : 48; }
template <typename T>
constexpr int box_bytes() { return (box_w<T>() * kBoxH * (int)sizeof(T) + 127) & ~127; }

// A frame's word for one warp (bits 0..17: byte offset of the window in the ring).
constexpr int kPatBit = 18;              // bits 18..21: at a run's end, the next run's pattern
constexpr uint32_t kRunEnd = 1u << 22, kStageEnd = 1u << 23;
constexpr int kCaseBit = 26;             // bits 26..31: steps (3 bits), rows - 8 (2 bits) and
                                         // direction (1: the columns step towards lower x)

// A group's entry in xg: bits 0..15 shift of the first velocity + kShiftBias,
// bits 16..18 the steps, bit 19 their direction (1: towards lower x).
__device__ __forceinline__ int xg_shift(uint32_t e) { return (int)(e & 0xffffu) - kShiftBias; }
__device__ __forceinline__ int xg_last(uint32_t e) {
  const int n = __popc((e >> 16) & 7u);
  return xg_shift(e) + ((e >> 19) & 1u ? -n : n);
}

// First group of x-velocity tile t (tiles of equal size to one group).
__host__ __device__ __forceinline__ int tile_group(int nG, int nT, int t) {
  return (int)((int64_t)t * nG / nT);
}

// xg, and the largest column offset of a tile's box.
__global__ void k_run_shifts(const int32_t* __restrict__ sx, int N, int nvx, int nG, int nT,
                             int align, uint32_t* __restrict__ xg, int* __restrict__ bad) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < (int64_t)N * nG) {
    const int64_t i = idx / nG;
    const int g = (int)(idx % nG);
    const int32_t* row = sx + i * nvx;
    int prev = row[min(g * kG, nvx - 1)], dir = 0;
    bool no = prev < -32000 || prev > 32000;
    uint32_t e = (uint32_t)((prev + kShiftBias) & 0xffff);
    for (int j = 1; j < kG; ++j) {
      const int s = row[min(g * kG + j, nvx - 1)], d = s - prev;
      no |= d < -1 || d > 1 || (dir != 0 && d != 0 && d != dir);
      if (d != 0) {
        dir = d;
        e |= 1u << (15 + j);
      }
      prev = s;
    }
    if (dir < 0) e |= 1u << 19;
    xg[idx] = e;
    if (no) atomicMax(&bad[0], 1);
  } else if (idx < (int64_t)N * (nG + nT)) {
    const int64_t k = idx - (int64_t)N * nG, i = k / nT;
    const int t = (int)(k % nT);
    const int a0 = tile_group(nG, nT, t) * kG;
    const int a1 = min(tile_group(nG, nT, t + 1) * kG, nvx) - 1;
    int mn = INT_MAX, mx = INT_MIN;
    for (int a = a0; a <= a1; ++a) {
      const int s = sx[i * nvx + a];
      mn = min(mn, s);
      mx = max(mx, s);
    }
    // (shifts of one frame are monotone in the velocity: the producer takes
    // the tile's ends)
    const int s0 = sx[i * nvx + a0], s1 = sx[i * nvx + a1];
    if (mn != min(s0, s1) || mx != max(s0, s1)) atomicMax(&bad[0], 1);
    atomicMax(&bad[1], mx - (mn & ~(align - 1)));
  }
}

// ord: one warp per y-velocity tile B lists the frames by pattern, in frame
// order within a pattern: (lowest shift, frame | id << 16 | height << 20 | end
// of a run that another follows << 22 | that run's pattern << 23).
__global__ void k_run_order(const unsigned char* __restrict__ pat, const int4* __restrict__ yt,
                            int N, int nB, int2* ord) {
  const int B = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32);
  const int lane = threadIdx.x & 31;
  if (B >= nB) return;
  // (neighbours differ at one y-velocity by 1, but for two pairs)
  const int order[kPatterns] = {7, 3, 6, 5, 1, 2, 4, 0, 8, 9, 11, 12, 10, 13, 14};
  int at = 0;  // frames listed so far
  for (int k = 0; k < kPatterns; ++k) {
    const int id = order[k], from = at;
    const int height = max(max(pat_off(id, 0), pat_off(id, 1)), max(pat_off(id, 2), pat_off(id, 3)));
    for (int i0 = 0; i0 < N; i0 += 32) {
      const int i = i0 + lane;
      const bool mine = i < N && pat[(int64_t)i * nB + B] == id;
      const unsigned m = __ballot_sync(0xffffffffu, mine);
      if (mine)
        ord[(int64_t)B * N + at + __popc(m & ((1u << lane) - 1u))] =
            make_int2(yt[(int64_t)i * nB + B].x,
                      (int)((unsigned)i | (unsigned)id << 16 | (unsigned)height << 20));
      at += __popc(m);
    }
    __syncwarp();
    if (lane == 0 && at > from && from > 0)
      ord[(int64_t)B * N + from - 1].y |= (int)(1u << 22 | (unsigned)id << 23);
    __syncwarp();
  }
}

// Items of a field: super-tiles of at most 4 x 4 pixel tiles (of equal size, so
// that few lie beyond the frame), then velocity tiles, then the tiles of the
// super-tile (neighbouring CTAs share footprints in L2).
struct Supers {
  int nx, ny;  // super-tiles
  int w, h;    // tiles of one
};
__host__ __device__ __forceinline__ Supers supers_of(const FastField& ff) {
  const int tx = (ff.W + kTX - 1) / kTX, ty = (ff.H + kTY - 1) / kTY;
  Supers s;
  s.nx = (tx + kSuper - 1) / kSuper;
  s.ny = (ty + kSuper - 1) / kSuper;
  s.w = (tx + s.nx - 1) / s.nx;
  s.h = (ty + s.ny - 1) / s.ny;
  return s;
}
__host__ __device__ __forceinline__ int64_t items_of(const FastField& ff) {
  const Supers s = supers_of(ff);
  return (int64_t)s.nx * s.ny * s.w * s.h * ff.nT * ff.nB;
}

struct Item {
  int f;  // index into the launch's fields (-1: no more work)
  int X0, Y0, A, B;
  // by the producer: the first run's pattern, the tile's groups, the frames,
  // and the threshold of a point that every frame covers, less the margin
  int pat, g0, ng, N;
  float thr;
};
__device__ __forceinline__ Item decode(const FastField& ff, int f, int64_t L) {
  const int nVT = ff.nT * ff.nB;
  const Supers s = supers_of(ff);
  const int sub = (int)(L % (s.w * s.h));
  const int64_t rest = L / (s.w * s.h);
  const int vt = (int)(rest % nVT), stile = (int)(rest / nVT);
  Item it{};
  it.f = f;
  it.X0 = ((stile % s.nx) * s.w + sub % s.w) * kTX;
  it.Y0 = ((stile / s.nx) * s.h + sub / s.w) * kTY;
  it.A = vt % ff.nT;
  it.B = vt / ff.nT;
  return it;
}

// Offsets of a pattern's 4 y-velocities, 2 bits each.
__device__ __forceinline__ uint32_t pattern_offsets(int id) {
  const int up = id < 8 ? id : 0, down = id < 8 ? 0 : id - 7;
  const int u1 = up & 1, u2 = (up >> 1) & 1, u3 = up >> 2;
  const int d1 = down & 1, d2 = (down >> 1) & 1, d3 = down >> 2;
  return (uint32_t)((d1 + d2 + d3) | (u1 + d2 + d3) << 2 | (u1 + u2 + d3) << 4 |
                    (u1 + u2 + u3) << 6);
}

// The sums of a warp's 4 x-velocities: pair q holds rows q and q + 4 of the
// window, as an accumulator's pair m holds output rows m and m + 4, so a
// staircase offset c adds pair m + c to pair m whatever its parity.
constexpr int kPairs = kRows / 2 + 3;
template <int C>
__device__ __forceinline__ void add_moved(float2 (&a)[8], const unsigned long long* s) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    float2 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(s[(k / 4) * kPairs + k % 4 + C]));
    a[k] = __fadd2_rn(a[k], v);
  }
}

// ---- tensor memory: 16 columns of this warp's 32 lanes
__device__ __forceinline__ void tm_load16(uint32_t addr, float2 (&v)[8]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(addr)
      : "memory");
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = make_float2(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1]));
}
// Points of one x- and y-velocity at or above the threshold (bit r: row r), to
// the pending list.
__device__ __noinline__ void emit(uint32_t mask, int x, int y0, int bv, int av, const FastField& ff,
                                  Pending* pend, int64_t cap, Counters* ctr) {
  if (x >= ff.W || av >= ff.nvx || bv >= ff.nvy) mask = 0u;
  while (__any_sync(0xffffffffu, mask != 0u)) {
    const bool has = mask != 0u;
    const int y = y0 + (has ? __ffs(mask) - 1 : 0);
    mask &= has ? mask - 1u : 0u;
    const Pending rec{x, y, bv * ff.nvx + av, ff.field, 0.0f, -1};
    push_pending(has && y < ff.H, rec, pend, cap, ctr);
  }
}

// A consumer warp's part of an item: row quarter and group.  Each quarter's
// groups start at another scheduler, so that the warps without a group (fewer
// than 4 in a tile) fall on different ones.  (Read afresh: the thread index
// lives in no register.)
struct Role {
  int lane, part, group;
  uint32_t tm;  // from the CTA's tensor memory: the warp's lanes and columns
};
__device__ __forceinline__ Role role_of() {
  uint32_t t;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
  const int warp = (int)(t >> 5);
  Role r;
  r.lane = (int)(t & 31);
  r.part = warp / kXG;
  r.group = (warp + r.part) % kXG;
  r.tm = ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * kAccCols;
  return r;
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 1) k_stack_runs(const __grid_constant__ RunArgs p) {
  constexpr int kBox = box_bytes<T>();
  constexpr int kAlign = 16 / (int)sizeof(T);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // barriers and words, laid out as the PTX block addresses them
  struct Ring {
    uint64_t full[kS], empty[kS];
    uint32_t words[kS * kXG * kF + 1];  // (one is read ahead of the last)
  };
  __shared__ __align__(16) Ring rg;
  uint64_t* full_bar = rg.full;
  uint64_t* empty_bar = rg.empty;
  uint32_t* words = rg.words;
  __shared__ int item_inside[kItemSlots];        // frames of an item fully inside
  __shared__ int item_done[kItemSlots];          // consumer warps done with it
  __shared__ Item item_info[kItemSlots];
  __shared__ uint32_t tm_base;
  if (p.d_use && *p.d_use == 0) return;  // (uniform over the grid)
  unsigned char* ring = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < kS; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], kCW);
    }
    mbar_init_fence();
  }
  if (tid < kItemSlots) item_inside[tid] = item_done[tid] = 0;
  if (blockIdx.x == 0 && tid == 0) p.ctr->runs = 1u;
  if (warp == kCW) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                     smem_u32(&tm_base))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  if (warp == kCW) {
    // ---------------------------------------------------------------- producer
    // Lane l stages frame l % kF of a stage (lanes below kF its copy) and writes
    // the words of groups l / kF, ...  The order entry is read two stages
    // ahead and the groups' entries one stage ahead.
    constexpr int kLG = 32 / kF, kLaneGroups = (kXG + kLG - 1) / kLG;
    const int fi = lane % kF, hg = lane / kF;
    int f = 0, acq_f = -1;
    int64_t base = 0, f_items = items_of(*p.ff[0]);
    auto locate = [&](int64_t L) -> Item {
      Item it{};
      it.f = -1;
      if (L >= p.n_items) return it;
      while (L >= base + f_items) {
        base += f_items;
        f_items = items_of(*p.ff[++f]);
      }
      return decode(*p.ff[f], f, L - base);
    };
    auto take = [&]() -> int64_t {
      int64_t L = 0;
      if (lane == 0) L = (int64_t)atomicAdd(p.work, 1ull);
      return __shfl_sync(0xffffffffu, L, 0);
    };
    struct Entry {
      int2 o;                    // order entry
      uint32_t first, last;      // the tile's first and last group
      uint32_t g[kLaneGroups];   // this lane's groups
      bool valid;
    };
    // a stage: item and stage index; its item's field in registers
    struct Where {
      Item it;
      int st, spi, N, nG, g0, ng, W, H;
      const int2* ord;
      const uint32_t* xg;
      float thr;
    };
    auto where_of = [&](const Item& it) {
      Where w{};
      w.it = it;
      if (it.f < 0) {
        w.spi = 1;
        return w;
      }
      const FastField& ff = *p.ff[it.f];
      w.N = ff.N;
      w.spi = (ff.N + kF - 1) / kF;
      w.nG = ff.nG;
      w.W = ff.W;
      w.H = ff.H;
      w.g0 = tile_group(ff.nG, ff.nT, it.A);
      w.ng = tile_group(ff.nG, ff.nT, it.A + 1) - w.g0;
      w.ord = ff.ord + (int64_t)it.B * ff.N;
      w.xg = ff.xg;
      w.thr = __ldg(ff.thr + max(ff.N, ff.nmin)) -
              (p.d_margin ? __ldg(p.d_margin + ff.field) : p.margin[it.f]);
      return w;
    };
    auto next = [&](const Where& w) {
      Where n = w;
      if (w.it.f >= 0 && ++n.st == w.spi) n = where_of(locate(take()));
      return n;
    };
    auto load_order = [&](const Where& w, Entry& e) {
      const int k = w.st * kF + fi;
      e.valid = w.it.f >= 0 && k < w.N;
      if (e.valid) e.o = __ldg(w.ord + k);
    };
    auto load_groups = [&](const Where& w, Entry& e) {
      if (!e.valid) return;
      const uint32_t* row = w.xg + (int64_t)(e.o.y & 0xffff) * w.nG + w.g0;
      e.first = __ldg(row);
      e.last = __ldg(row + w.ng - 1);
#pragma unroll
      for (int q = 0; q < kLaneGroups; ++q)
        e.g[q] = kLG * q + hg < w.ng ? __ldg(row + kLG * q + hg) : 0u;
    };
    Where w0 = where_of(locate(take())), w1 = next(w0);
    Entry e0{}, e1{};
    load_order(w0, e0);
    load_order(w1, e1);
    load_groups(w0, e0);
    int slot = 0, item = 0;
    int64_t seq = 0;
    for (;;) {
      const bool done = w0.it.f < 0;
      const Where w2 = next(w1);
      Entry e2{};
      load_order(w2, e2);
      load_groups(w1, e1);
      const CUtensorMap* map = done ? nullptr : p.maps[w0.it.f];
      if (!done && w0.it.f != acq_f) {
        if (lane == 0) {
          tmap_acquire(map);
          tma_prefetch_desc(map);
        }
        acq_f = w0.it.f;
      }
      if (seq >= kS && !mbar_wait_sleep(&empty_bar[slot], (uint32_t)(seq / kS - 1) & 1u,
                                        kStackWaitNs, kProducerSleepNs)) {
        if (lane == 0) atomicOr(&p.ctr->error, ERR_TIMEOUT);
        break;  // consumers time out on the missing stage (bounded)
      }
      if (w0.st == 0 && lane == 0) {
        Item it = w0.it;
        it.pat = (e0.o.y >> 16) & 15;
        it.g0 = w0.g0;
        it.ng = w0.ng;
        it.N = w0.N;
        it.thr = w0.thr;
        item_info[item % kItemSlots] = it;
      }
      const bool copies = e0.valid && hg == 0;
      const unsigned nc = __popc(__ballot_sync(0xffffffffu, copies));
      if (lane == 0 && nc)
        mbar_expect_tx(&full_bar[slot], (uint32_t)(kBoxH * box_w<T>() * sizeof(T)) * nc);
      if (e0.valid) {
        const int lo = min(xg_shift(e0.first), xg_last(e0.last));
        const int hi = max(xg_shift(e0.first), xg_last(e0.last));
        const int xs = lo & ~(kAlign - 1);
        const unsigned oy = (unsigned)e0.o.y;
        const int height = (int)(oy >> 20) & 3;
        const uint32_t fixed = (uint32_t)((slot * kF + fi) * kBox) |
                               (uint32_t)height << (kCaseBit + 3) | ((oy >> 23) & 15u) << kPatBit |
                               ((oy >> 22) & 1u ? kRunEnd : 0u) |
                               (fi == kF - 1 || w0.st * kF + fi == w0.N - 1 ? kStageEnd : 0u);
#pragma unroll
        for (int q = 0; q < kLaneGroups; ++q) {
          const int g = kLG * q + hg;
          const uint32_t e = e0.g[q];
          if (g < w0.ng)
            words[(slot * kXG + g) * kF + fi] =
                fixed + (uint32_t)((xg_shift(e) - xs) * (int)sizeof(T)) +
                (((e >> 16) & 7u) << kCaseBit) + (((e >> 19) & 1u) << (kCaseBit + 5));
        }
        if (hg == 0) {
          const bool inside = w0.it.X0 + lo >= 0 && w0.it.X0 + kTX - 1 + hi < w0.W &&
                              w0.it.Y0 + e0.o.x >= 0 &&
                              w0.it.Y0 + kTY - 1 + e0.o.x + height < w0.H;
          if (inside) atomicAdd(&item_inside[item % kItemSlots], 1);
          tma_load_3d(ring + (size_t)(slot * kF + fi) * kBox, map, w0.it.X0 + xs,
                      w0.it.Y0 + e0.o.x, (int)(oy & 0xffffu), &full_bar[slot]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&full_bar[slot]);
      if (++slot == kS) slot = 0;
      ++seq;
      if (done) break;
      if (w1.st == 0) ++item;
      w0 = w1;
      e0 = e1;
      w1 = w2;
      e1 = e2;
    }
    // the last use of each ring slot completes before the CTA may exit (only
    // the latest phase of a slot can be waited on)
    if (lane == 0)
      for (int64_t sq = seq > kS ? seq - kS : 0; sq < seq; ++sq)
        mbar_wait(&full_bar[sq % kS], (uint32_t)(sq / kS) & 1u, kStackWaitNs);
    __syncwarp();
  } else {
    // --------------------------------------------------------------- consumers
    // (Nothing but the item number, the slot and its phase lives across the
    // PTX block: 96 registers a thread hold its 56 of sums and little else.)
    uint32_t slot = 0, ph = 0;
    for (int item = 0;; ++item) {
      if (!__all_sync(0xffffffffu, mbar_wait(&full_bar[slot], ph, kStackWaitNs))) {
        if (lane == 0) atomicOr(&p.ctr->error, ERR_TIMEOUT);  // leave (warp-uniform)
        break;
      }
      if (item_info[item % kItemSlots].f < 0) break;
      unsigned long long sums[kG * kPairs];
#pragma unroll
      for (int k = 0; k < kG * kPairs; ++k) sums[k] = 0ull;
      uint32_t off = pattern_offsets(item_info[item % kItemSlots].pat);
      {
        const Role r = role_of();
        const Item it = item_info[item % kItemSlots];
        int stages = (it.N + kF - 1) / kF;
        if (r.group >= it.ng) stages = -stages;
        const uint32_t base = smem_u32(&rg), my_words = smem_u32(rg.words + r.group * kF);
        const uint32_t lane_base =
            smem_u32(ring) + (uint32_t)((r.part * kRows * box_w<T>() + r.lane) * (int)sizeof(T));
        const uint32_t tm = tm_base + r.tm;
        __syncwarp();  // the item description is read before the block
        if constexpr (std::is_same<T, float>::value)
          asm volatile(ST_RUN_ITEM_F32 ST_RUN_OPERANDS(sums, slot, ph, off, stages, base, my_words,
                                                       lane_base, tm));
        else if constexpr (std::is_same<T, __half>::value)
          asm volatile(ST_RUN_ITEM_F16 ST_RUN_OPERANDS(sums, slot, ph, off, stages, base, my_words,
                                                       lane_base, tm));
        else
          asm volatile(ST_RUN_ITEM_BF16 ST_RUN_OPERANDS(sums, slot, ph, off, stages, base, my_words,
                                                        lane_base, tm));
      }
      if (slot == kS) {
        if ((threadIdx.x & 31) == 0) atomicOr(&p.ctr->error, ERR_TIMEOUT);
        break;
      }
      // read the item again (still in its slot: the producer is fewer than
      // kItemSlots items ahead), so that nothing of it lives across the block
      const Role r = role_of();
      const int lane = r.lane, part = r.part, group = r.group;
      const uint32_t tm = tm_base + r.tm;
      const Item it = item_info[item % kItemSlots];
      const FastField& ff = *p.ff[it.f];
      const int N = it.N, g0 = it.g0;
      const bool active = group < it.ng;
      if (active) {
        // ---- the accumulators against the thresholds (less the margin)
        const int n_full = item_inside[item % kItemSlots];
        const int x = it.X0 + lane, y0 = it.Y0 + part * kRows;
        const float thr_n = it.thr;
#pragma unroll 1
        for (int j = 0; j < kMB; ++j) {
          const int bv = it.B * kMB + j;
          int ny = 0;
          if (n_full != N) {
            // edge item: n_cov >= nx + ny - N, with nx / ny the frames whose
            // x / y sample is inside (ny at the warp's least covered row)
            const int bvc = min(bv, ff.nvy - 1), y = y0 + lane % kRows;
            ny = count_shifts(ff.covy + (int64_t)bvc * ff.cov_len, __ldg(ff.cov_ymin + bvc),
                              __ldg(ff.cov_ymax + bvc), N, -y, ff.H - 1 - y);
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) ny = min(ny, __shfl_xor_sync(0xffffffffu, ny, d));
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {  // x-velocities 2h, 2h + 1
            float2 a[8];
            if ((off >> (8 + 2 * j)) & 1u) {
              tm_load16(tm + (uint32_t)(j * kG * kRows + 16 * h), a);
            } else {
#pragma unroll
              for (int k = 0; k < 8; ++k) a[k] = make_float2(0.0f, 0.0f);
            }
            const unsigned long long* v = sums + 2 * h * kPairs;
            switch ((off >> (2 * j)) & 3u) {
              case 0: add_moved<0>(a, v); break;
              case 1: add_moved<1>(a, v); break;
              case 2: add_moved<2>(a, v); break;
              default: add_moved<3>(a, v); break;
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const int av = (g0 + group) * kG + 2 * h + q;
              float thr = thr_n;
              if (n_full != N) {
                const int avc = min(av, ff.nvx - 1);
                const int nx = count_shifts(ff.covx + (int64_t)avc * ff.cov_len,
                                            __ldg(ff.cov_xmin + avc), __ldg(ff.cov_xmax + avc), N,
                                            -x, ff.W - 1 - x);
                thr = __ldg(ff.thr + min(max(max(n_full, ff.nmin), nx + ny - N), N)) -
                      (p.d_margin ? __ldg(p.d_margin + ff.field) : p.margin[it.f]);
              }
              const float2* b = a + 4 * q;
              const float top = fmaxf(fmaxf(fmaxf(b[0].x, b[0].y), fmaxf(b[1].x, b[1].y)),
                                      fmaxf(fmaxf(b[2].x, b[2].y), fmaxf(b[3].x, b[3].y)));
              if (__any_sync(0xffffffffu, top >= thr)) {
                uint32_t mask = 0u;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                  mask |= (uint32_t)(b[k].x >= thr) << k;
                  mask |= (uint32_t)(b[k].y >= thr) << (k + 4);
                }
                emit(mask, x, y0, bv, av, ff, p.pend, p.cap, p.ctr);
              }
            }
          }
        }
      }
      // release the item's slots: the last warp done with it clears them
      __syncwarp();
      if (lane == 0 && atomicAdd(&item_done[item % kItemSlots], 1) == kCW - 1) {
        item_inside[item % kItemSlots] = 0;
        item_done[item % kItemSlots] = 0;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == kCW)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tm_base));
}

}  // namespace

int run_box_w(int storage) { return storage == ST_F32 ? box_w<float>() : box_w<__half>(); }
int run_box_h() { return kBoxH; }
int64_t run_items(const FastField& ff) { return items_of(ff); }

RunPlan* run_plan_build(const FieldDev& fd, int nB) {
  RunPlan* rp = new (std::nothrow) RunPlan();
  if (!rp) return nullptr;
  rp->nG = (fd.nvx + kG - 1) / kG;
  rp->nT = (rp->nG + kXG - 1) / kXG;
  if (cudaMalloc(&rp->xg, sizeof(uint32_t) * (size_t)fd.N * rp->nG) != cudaSuccess ||
      cudaMalloc(&rp->ord, sizeof(int2) * (size_t)fd.N * nB) != cudaSuccess ||
      cudaMalloc(&rp->bad, sizeof(int) * 2) != cudaSuccess ||
      cudaMalloc(&rp->d_map, sizeof(CUtensorMap)) != cudaSuccess ||
      cudaMallocHost(&rp->h_bad, sizeof(int) * 2) != cudaSuccess) {
    run_plan_free(rp);
    return nullptr;
  }
  return rp;
}

void run_plan_free(RunPlan* rp) {
  if (!rp) return;
  cudaFree(rp->xg);
  cudaFree(rp->ord);
  cudaFree(rp->bad);
  cudaFree(rp->d_map);
  if (rp->h_bad) cudaFreeHost(rp->h_bad);
  delete rp;
}

void run_prepare(const FieldDev& fd, const unsigned char* pat, const int4* yt, int nB,
                 RunPlan* rp, cudaStream_t s) {
  cudaMemsetAsync(rp->bad, 0, sizeof(int) * 2, s);
  const int64_t n = (int64_t)fd.N * (rp->nG + rp->nT);
  k_run_shifts<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(
      fd.sx, fd.N, fd.nvx, rp->nG, rp->nT, fd.storage == ST_F32 ? 4 : 8, rp->xg, rp->bad);
  k_run_order<<<(unsigned)((nB + 3) / 4), 128, 0, s>>>(pat, yt, fd.N, nB, rp->ord);
  cudaMemcpyAsync(rp->h_bad, rp->bad, sizeof(int) * 2, cudaMemcpyDeviceToHost, s);
}

void run_finish(const FieldDev& fd, RunPlan* rp) {
  rp->fits = rp->h_bad[0] == 0 && rp->h_bad[1] <= run_box_w(fd.storage) - kTX;
}

int launch_runs(const RunArgs& a, int storage, int sms, cudaStream_t s) {
  const void* fn = storage == ST_F32   ? (const void*)k_stack_runs<float>
                   : storage == ST_F16 ? (const void*)k_stack_runs<__half>
                                       : (const void*)k_stack_runs<__nv_bfloat16>;
  const size_t smem = 128 + (size_t)kS * kF * (storage == ST_F32 ? box_bytes<float>()
                                                                 : box_bytes<__half>());
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return -1;
  const int64_t grid = a.n_items < sms ? a.n_items : sms;
  if (grid < 1) return 0;
  void* args[1] = {const_cast<RunArgs*>(&a)};
  if (cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(kThreads), args, smem, s) != cudaSuccess)
    return -1;
  return 1;
}

}  // namespace st
