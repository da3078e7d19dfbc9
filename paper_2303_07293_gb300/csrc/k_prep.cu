// k_prep.cu — time offsets and shift tables (FP64), robust per-frame sky
// statistics (FP64, deterministic) and normalisation into the storage cube.
//
// Shift tables: linear motion with no position-angle constraint (Sec. 2.1):
// frame i is sampled at p + v*dt_i, dt_i = t_i - t_ref, v = v0 + a*dv.  Every
// FP64 operation is an explicit _rn intrinsic so no multiply-add is fused.
//
// Sky statistics: the per-frame sky level and standard deviation used for
// frame QC in Sec. 2.1, read as a kappa-sigma clipped mean and population
// standard deviation (kappa = 3, at most 5 statistics, stop when the kept set
// is unchanged).
//
// What bounds it: each statistic is one pass over the cube, so HBM, provided
// the FP64 pipe (about 2 operations per SM clock) stays out of the loop: at
// 6.8 TB/s an SM receives 5.4 pixels per clock.  The sums are therefore held
// as integers.  A frame's pixels are taken relative to a pivot p near its
// mean and scaled by a power of two, ds = (x - p) 2^-r in [-1, 1] (exact by
// the choice of p and r), and ds and ds^2 are split by adding and subtracting
// large constants into parts on fixed grids (2^-22 and 2^-45; what the square
// has beyond, its rounding error too, on 2^-47 and 2^-70) whose integer codes
// add up without error.
// The few pixels outside [-1, 1] (outliers, before they are clipped) are
// summed in FP64.  So the sums lose only what lies below 2^-46 of the range
// in ds below 2^-22 of it, and below 2^-71 in the squares, whatever the order,
// and a pass computes count, mean and variance together (5 passes; a mean pass
// and a variance pass are not needed).  Measured against extended precision
// (12288 pixels, levels of 0 to 40 deviations): sigma within 2^-52.
// Membership is a comparison with the first and last FP32 value that the
// FP64 rule keeps.  A sample of the frame gives p and r of the first pass,
// the statistics of each pass those of the next.
// Measured on a 2048^2 x 256 FP32 cube (4.29 GB): a pass 1.15 ms, 3.7 TB/s
// (issue slots: 33 instructions a pixel), the statistics 5.8 ms; with FP64
// sums they took 104 ms in 6 passes.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "st_internal.h"

namespace st {

namespace {

__global__ void k_shift_tables(const double* __restrict__ t, int N, double t_ref, double v0,
                               double dv, int nv, int mode, int32_t* __restrict__ s,
                               float* __restrict__ f) {
  int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)N * nv) return;
  int i = (int)(idx / nv), a = (int)(idx % nv);
  double dt = __dsub_rn(t[i], t_ref);
  double v = __dadd_rn(v0, __dmul_rn((double)a, dv));
  double p = __dmul_rn(v, dt);
  if (mode == ST_NEAREST) {
    s[idx] = (int32_t)floor(__dadd_rn(p, 0.5));
    if (f) f[idx] = 0.0f;
  } else {
    double fl = floor(p);
    s[idx] = (int32_t)fl;
    if (f) f[idx] = (float)__dsub_rn(p, fl);
  }
}

constexpr int kSkyBlocks = 64;    // blocks (and partial sums) per frame, at most
constexpr int kSkyThreads = 256;
constexpr int kSkyFlush = 256;    // pixels per thread between flushes of the 32-bit sums
constexpr int kSkyIters = 5;
constexpr double kKappa = 3.0;
constexpr int kSample = 2048;     // pixels sampled for the pivot and the range

// Per-frame state of the clipping.
struct SkyState {
  double mu, sigma;     // statistics of the last kept set
  double pivot;         // p (an FP32 value)
  float scale, offset;  // ds = fma(x, scale, offset): scale = 2^-r, offset = -p 2^-r
  int r;
  int done;
  float lo, hi;         // kept set of the next pass: lo <= x <= hi
  float plo, phi;       // and of the pass before it
  unsigned arrived;     // blocks of the running pass that have stored their partials
  unsigned pad;
};
static_assert(sizeof(SkyState) == 64, "state of a frame: 8 doubles");

// Partial sums of one block.
struct SkyPartial {
  long long d1, d2;      // codes of ds on the grids 2^-22 and 2^-45
  long long s1, s2;      // codes of ds^2 on the same grids
  long long s3, s4;      // codes of what ds^2 has beyond, on 2^-47 and 2^-70
  long long n, changed;  // kept pixels; pixels whose membership changed
  double w1, w2;         // kept pixels outside [-1, 1]: sums of x - p and (x - p)^2
};
static_assert(sizeof(SkyPartial) == 80, "partial sums of a block: 10 doubles");

// x + kM1 has ulp 2^-22 for |x| <= 1, x + kM2 2^-45 for |x| <= 2^-23, and
// x + kM3 2^-47 for |x| <= 2^-25, x + kM4 2^-70 for |x| <= 2^-48: the sum's
// bits less the constant's are the code of x rounded to that grid.
constexpr float kM1 = 3.0f, kM2 = 0x1.8p-22f, kM3 = 0x1.8p-24f, kM4 = 0x1.8p-47f;

__device__ __forceinline__ bool kept64(float x, double mu, double thr) {
  return fabs(__dsub_rn((double)x, mu)) <= thr;
}

// The first and last FP32 value that |x - mu| <= thr (in FP64) keeps; the
// rule is monotone on either side of mu and rounding leaves each end within
// two steps.  (First > last: it keeps none.)
__device__ void kept_interval(double mu, double thr, float* lo, float* hi) {
  float a = __double2float_rn(mu - thr), b = __double2float_rn(mu + thr);
  for (int q = 0; q < 3 && kept64(nextafterf(a, -INFINITY), mu, thr); ++q)
    a = nextafterf(a, -INFINITY);
  for (int q = 0; q < 3 && !kept64(a, mu, thr); ++q) a = nextafterf(a, INFINITY);
  for (int q = 0; q < 3 && kept64(nextafterf(b, INFINITY), mu, thr); ++q)
    b = nextafterf(b, INFINITY);
  for (int q = 0; q < 3 && !kept64(b, mu, thr); ++q) b = nextafterf(b, -INFINITY);
  const float big = 3.402823466e38f;  // (infinite pixels are never kept)
  *lo = fmaxf(a, -big);
  *hi = fminf(b, big);
}

// Pivot and range of the next pass: 2^r >= reach (a multiple of the deviation
// that holds the pixels to sum) about a pivot of few bits near mu; a mean
// within 1.6 ranges of zero takes the pivot 0 and a range that holds it.
// Either way x - p is exact: in the first case every |x| in range is at least
// half the range (its last bit is no finer than 2^-24 of the range).
__device__ void set_range(SkyState& st, double mu, double reach) {
  const bool spread = reach > 0.0;
  reach = fmax(reach, fabs(mu) * 0x1p-20);
  int r = reach > 0.0 ? ilogb(reach) + 1 : -200;
  double p = 0.0;
  if (fabs(mu) < 1.6 * ldexp(1.0, r)) {
    reach += fabs(mu);
    r = reach > 0.0 ? ilogb(reach) + 1 : -200;
  } else {
    const double g = ldexp(1.0, r - 6);
    p = spread && fabs(mu) < g * 0x1p23 ? rint(mu / g) * g : (double)(float)mu;
  }
  if (r < -100 || r > 100 || !isfinite(p)) {
    st.r = 0;
    st.pivot = isfinite(mu) ? mu : 0.0;
    st.scale = INFINITY;  // no pixel is in range: every sum in FP64, about mu
    st.offset = 0.0f;
  } else {
    st.r = r;
    st.pivot = p;
    st.scale = (float)ldexp(1.0, -r);
    st.offset = (float)ldexp(-p, -r);
  }
}

// One block per frame: a sample's clipped mean and deviation give the pivot
// and the range of the first pass (a poor guess costs time, not accuracy).
__global__ void __launch_bounds__(kSkyThreads)
    k_sky_guess(const float* __restrict__ raw, int64_t npix, SkyState* __restrict__ state) {
  __shared__ float sh[3][kSkyThreads / 32];
  const float* x = raw + (int64_t)blockIdx.x * npix;
  const int tid = threadIdx.x;
  float v[kSample / kSkyThreads];
#pragma unroll
  for (int q = 0; q < kSample / kSkyThreads; ++q) {
    const int64_t k = (int64_t)q * kSkyThreads + tid;
    // evenly spread, each moved within its share of the frame
    const int64_t step = npix / kSample;
    const int64_t j = npix <= kSample ? k : k * step + (int64_t)(k * 2654435761ull % (uint64_t)step);
    v[q] = j < npix ? x[j] : INFINITY;
  }
  // the mean and the deviation (1.25 mean absolute deviations) of what lies
  // within 4 deviations, from the whole sample on
  float mu = 0.0f, sd = 0x1p120f;
  for (int it = 0; it < 5; ++it) {
    float n = 0.0f, s1 = 0.0f, s2 = 0.0f;
#pragma unroll
    for (int q = 0; q < kSample / kSkyThreads; ++q) {
      const float d = v[q] - mu;
      const bool in = fabsf(v[q]) < 0x1p100f && fabsf(d) <= 4.0f * sd;
      n += in ? 1.0f : 0.0f;
      s1 += in ? d : 0.0f;
      s2 += in ? fabsf(d) : 0.0f;
    }
    for (int d = 16; d > 0; d >>= 1) {
      n += __shfl_down_sync(0xffffffffu, n, d);
      s1 += __shfl_down_sync(0xffffffffu, s1, d);
      s2 += __shfl_down_sync(0xffffffffu, s2, d);
    }
    __syncthreads();
    if ((tid & 31) == 0) {
      sh[0][tid >> 5] = n;
      sh[1][tid >> 5] = s1;
      sh[2][tid >> 5] = s2;
    }
    __syncthreads();
    n = s1 = s2 = 0.0f;
    for (int w = 0; w < kSkyThreads / 32; ++w) {
      n += sh[0][w];
      s1 += sh[1][w];
      s2 += sh[2][w];
    }
    if (!(n > 0.0f)) break;
    // (the first deviations are taken about 0: too wide, never too narrow)
    mu += s1 / n;
    sd = 1.25f * s2 / n;
  }
  if (tid != 0) return;
  SkyState st{};
  st.lo = st.plo = -3.402823466e38f;  // the first statistics: every finite pixel
  st.hi = st.phi = 3.402823466e38f;
  if (sd == 0x1p120f) sd = 0.0f;  // no sample
  set_range(st, (double)mu, 4.5 * (double)sd);
  state[blockIdx.x] = st;
}

// 32-bit sums of codes: a thread's pixels since the last flush.
struct Codes {
  uint32_t d1 = 0, d2 = 0, s1 = 0, s2 = 0, s3 = 0, s4 = 0;
  __device__ __forceinline__ static uint32_t bits(float2 t) {
    return __float_as_uint(t.x) + __float_as_uint(t.y);
  }
  __device__ __forceinline__ void add(float2 ds) {
    const float2 m1 = make_float2(kM1, kM1), m2 = make_float2(kM2, kM2);
    const float2 m3 = make_float2(kM3, kM3), m4 = make_float2(kM4, kM4);
    const float2 neg = make_float2(-1.0f, -1.0f);
    float2 t = __fadd2_rn(ds, m1);
    d1 += bits(t);
    d2 += bits(__fadd2_rn(__fadd2_rn(ds, __ffma2_rn(t, neg, m1)), m2));
    // (an fma, so that the rounded square and a sum after it stay two operations)
    const float2 s = __ffma2_rn(ds, ds, make_float2(0.0f, 0.0f));
    t = __fadd2_rn(s, m1);
    s1 += bits(t);
    const float2 a = __ffma2_rn(t, neg, m1);  // -(s on the first grid)
    t = __fadd2_rn(__fadd2_rn(s, a), m2);
    s2 += bits(t);
    // the square less both parts: its rounding error and what a square below
    // 2^-22 has beyond the second grid (ties there would all round one way)
    const float2 e = __ffma2_rn(ds, ds, __fadd2_rn(a, __ffma2_rn(t, neg, m2)));
    t = __fadd2_rn(e, m3);
    s3 += bits(t);
    s4 += bits(__fadd2_rn(__fadd2_rn(e, __ffma2_rn(t, neg, m3)), m4));
  }
};

__device__ __forceinline__ void plus(SkyPartial& v, const SkyPartial& o) {
  v.d1 += o.d1;
  v.d2 += o.d2;
  v.s1 += o.s1;
  v.s2 += o.s2;
  v.s3 += o.s3;
  v.s4 += o.s4;
  v.n += o.n;
  v.changed += o.changed;
  v.w1 += o.w1;
  v.w2 += o.w2;
}

__device__ __forceinline__ void warp_sum(SkyPartial& v) {
  for (int d = 16; d > 0; d >>= 1) {
    SkyPartial o;
    o.d1 = __shfl_down_sync(0xffffffffu, v.d1, d);
    o.d2 = __shfl_down_sync(0xffffffffu, v.d2, d);
    o.s1 = __shfl_down_sync(0xffffffffu, v.s1, d);
    o.s2 = __shfl_down_sync(0xffffffffu, v.s2, d);
    o.s3 = __shfl_down_sync(0xffffffffu, v.s3, d);
    o.s4 = __shfl_down_sync(0xffffffffu, v.s4, d);
    o.n = __shfl_down_sync(0xffffffffu, v.n, d);
    o.changed = __shfl_down_sync(0xffffffffu, v.changed, d);
    o.w1 = __shfl_down_sync(0xffffffffu, v.w1, d);
    o.w2 = __shfl_down_sync(0xffffffffu, v.w2, d);
    plus(v, o);
  }
}

// A frame in vectors of 4 from a 16-byte boundary at or before its start
// (at most 2^28 pixels).
struct SkyFrame {
  const float* xa;
  int skip;        // values before the frame's first
  int last;        // end of the frame from xa
};

// A block's sums over vectors [v0, v1) of a frame, valid in thread 0.
__device__ __forceinline__ SkyPartial sky_sums(const SkyFrame& f, int v0, int v1,
                                               const SkyState& st, SkyPartial* sh) {
  const int tid = threadIdx.x;
  const float2 sc = make_float2(st.scale, st.scale), of = make_float2(st.offset, st.offset);
  SkyPartial a{};
  int n = 0, changed = 0;
  bool any = false;
  auto keeps = [&](float x) { return x >= st.lo && x <= st.hi; };
  auto pair = [&](float x, float y, Codes& c) {
    float2 ds = __ffma2_rn(make_float2(x, y), sc, of);
    const bool kx = keeps(x), ky = keeps(y);
    n += (int)kx + (int)ky;
    changed += (int)(kx != (x >= st.plo && x <= st.phi)) + (int)(ky != (y >= st.plo && y <= st.phi));
    const bool ix = kx && fabsf(ds.x) <= 1.0f, iy = ky && fabsf(ds.y) <= 1.0f;
    any |= (kx != ix) | (ky != iy);
    ds.x = ix ? ds.x : 0.0f;
    ds.y = iy ? ds.y : 0.0f;
    c.add(ds);
  };
  // kept pixels outside the range, in FP64 (its instructions sit behind a
  // branch: predicated ones would take the FP64 pipe's time all the same)
  auto wild = [&](float x) {
    if (!keeps(x) || fabsf(fmaf(x, st.scale, st.offset)) <= 1.0f) return;
    const double d = (double)x - st.pivot;
    a.w1 += d;
    a.w2 += d * d;
  };
  constexpr int kU = 4;  // vectors in flight per thread
  const int whole0 = f.skip > 0, whole1 = f.last / 4;  // vectors without a missing value
  for (int vb = v0; vb < v1; vb += kSkyThreads * (kSkyFlush / 4)) {
    Codes c;
    uint32_t slots = 0;
    const int ve = min(v1, vb + kSkyThreads * (kSkyFlush / 4)), vw = min(ve, whole1);
    for (int v = vb + tid; v < ve; v += kSkyThreads * kU) {
      float4 q[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int w = v + u * kSkyThreads;
        if (w >= whole0 && w < vw) {
          q[u] = __ldg(reinterpret_cast<const float4*>(f.xa) + w);
        } else {
          // outside the frame: NaN, which no set keeps
          const float no = __int_as_float(0x7fc00000);
          const int e = 4 * w, last = w < ve ? f.last : 0;
          q[u].x = e >= f.skip && e < last ? __ldg(f.xa + e) : no;
          q[u].y = e + 1 >= f.skip && e + 1 < last ? __ldg(f.xa + e + 1) : no;
          q[u].z = e + 2 >= f.skip && e + 2 < last ? __ldg(f.xa + e + 2) : no;
          q[u].w = e + 3 >= f.skip && e + 3 < last ? __ldg(f.xa + e + 3) : no;
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        pair(q[u].x, q[u].y, c);
        pair(q[u].z, q[u].w, c);
      }
      if (any) {
        any = false;
#pragma unroll 1
        for (int u = 0; u < kU; ++u) {
          wild(q[0].x);
          wild(q[0].y);
          wild(q[0].z);
          wild(q[0].w);
#pragma unroll
          for (int k = 0; k < kU - 1; ++k) q[k] = q[k + 1];
        }
      }
      slots += 4 * kU;
    }
    // the codes' sums, each within +-2^30 (modulo 2^32 before the constants go)
    a.d1 += (int32_t)(c.d1 - slots * __float_as_uint(kM1));
    a.d2 += (int32_t)(c.d2 - slots * __float_as_uint(kM2));
    a.s1 += (int32_t)(c.s1 - slots * __float_as_uint(kM1));
    a.s2 += (int32_t)(c.s2 - slots * __float_as_uint(kM2));
    a.s3 += (int32_t)(c.s3 - slots * __float_as_uint(kM3));
    a.s4 += (int32_t)(c.s4 - slots * __float_as_uint(kM4));
    a.n += n;
    a.changed += changed;
    n = changed = 0;
  }
  warp_sum(a);
  if ((tid & 31) == 0) sh[tid >> 5] = a;
  __syncthreads();
  if (tid == 0)
    for (int w = 1; w < kSkyThreads / 32; ++w) plus(a, sh[w]);
  return a;
}

// v 2^e, v >= 0, rounded once.
__device__ __forceinline__ double scaled(__int128 v, int e) {
  if (v <= 0) return 0.0;
  const unsigned long long hi = (unsigned long long)(v >> 64), lo = (unsigned long long)v;
  if (hi == 0) return ldexp((double)lo, e);
  const int up = __clzll((long long)hi);
  // the first 64 bits, the last of them set if any beyond is
  const unsigned long long top = up ? hi << up | lo >> (64 - up) : hi;
  return ldexp((double)(top | (unsigned long long)((lo << up) != 0)), e + 64 - up);
}

// Mean and deviation of a kept set from its sums.  About a pivot of 0 beside a
// mean of up to 10 deviations the variance is a difference of terms 10^2
// times as large, so the sums are first moved, as the integers that they
// are, to within a step of 2^-22 of the mean: the variance is rounded twice and
// its root once, as good as a sum about the mean.  (FP64 here is one thread's,
// at the end of every pass: sums of twice FP64's length took 6 us a pass more.)
__device__ void sky_moments(const SkyPartial& a, SkyState& st) {
  const double cnt = (double)a.n;
  const long long c = (long long)rintf((float)a.d1 / (float)a.n);         // 2^-22
  const __int128 d = (__int128)a.d1 * (1 << 23) + a.d2;                   // 2^-45
  const __int128 s = ((__int128)a.s1 * (1 << 23) + a.s2) * (1 << 25) +
                     (__int128)a.s3 * (1 << 23) + a.s4;                   // 2^-70
  const double dc = (double)(long long)(d - (__int128)a.n * c * (1 << 23));
  __int128 sc = s - d * c * 16 + (__int128)a.n * (c * c) * (1 << 26);
  double m1 = dc / cnt, var;                                              // 2^-45
  if (a.w2 == 0.0) {
    sc -= __double2ll_rn(m1 * dc * 0x1p-20);
    var = scaled(sc, 2 * st.r - 70) / cnt;
    m1 = ldexp(fma(m1, 0x1p-23, (double)c), st.r - 22);
  } else {
    const double at = ldexp((double)c, st.r - 22);
    m1 = (ldexp(dc, st.r - 45) + a.w1) / cnt;
    var = (scaled(sc, 2 * st.r - 70) + (a.w2 - 2.0 * at * a.w1)) / cnt - m1 * m1;
    m1 += at;
  }
  st.mu = st.pivot + m1;
  st.sigma = sqrt(var > 0.0 ? var : 0.0);
}

// One statistic of every frame: sums over the frame's kept set; the last
// block of a frame adds up the frame's partials (fixed order) and updates its
// state.  iter: 1 (every finite pixel) .. kSkyIters.
__global__ void __launch_bounds__(kSkyThreads, 4)
    k_sky_pass(const float* __restrict__ raw, int64_t npix, int iter, SkyState* __restrict__ state,
               SkyPartial* __restrict__ partial) {
  __shared__ SkyPartial sh[kSkyThreads / 32];
  __shared__ SkyState s_st;
  // (two flags: a warp that still has to read the first must not see the second)
  __shared__ bool s_last, s_again;
  const int i = blockIdx.y, tid = threadIdx.x;
  SkyState st = state[i];
  if (st.done) return;  // frame converged (uniform per block)
  SkyFrame f;
  const float* x = raw + (int64_t)i * npix;
  f.skip = (int)((reinterpret_cast<uintptr_t>(x) >> 2) & 3);
  f.xa = x - f.skip;
  f.last = (int)npix + f.skip;
  const int nvec = (f.last + 3) / 4, blocks = gridDim.x;
  const int chunk = (nvec + blocks - 1) / blocks;
  const int v0 = min(nvec, (int)blockIdx.x * chunk);
  SkyPartial a = sky_sums(f, v0, min(nvec, v0 + chunk), st, sh);
  SkyPartial* mine = partial + (int64_t)i * kSkyBlocks;
  if (tid == 0) {
    mine[blockIdx.x] = a;
    __threadfence();
    s_last = atomicAdd(&state[i].arrived, 1u) == blocks - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (tid < 32) {
    auto load = [&](int b) {
      SkyPartial v;
      const double* src = reinterpret_cast<const double*>(mine + b);
      double* dst = reinterpret_cast<double*>(&v);
#pragma unroll
      for (int q = 0; q < (int)(sizeof(SkyPartial) / sizeof(double)); ++q) dst[q] = __ldcg(src + q);
      return v;
    };
    a = SkyPartial{};
    if (tid < blocks) a = load(tid);
    if (tid + 32 < blocks) plus(a, load(tid + 32));
    warp_sum(a);
  }
  // a set much narrower than the range it was summed with (a clip that took
  // away pixels far beyond the rest) is summed again with a range of its own,
  // by this block: rare, and the next membership depends on it
  for (int again = 0;; ++again) {
    if (tid == 0) {
      s_again = false;
      if (a.n > 0) {
        sky_moments(a, st);
        SkyState nx = st;
        set_range(nx, nx.mu, (kKappa + 0.1) * nx.sigma);
        s_again = again < 4 && ldexp(1.0, st.r) > 64.0 * st.sigma && nx.r < st.r;
        s_st = nx;
      }
    }
    __syncthreads();
    if (!s_again) break;
    st = s_st;
    a = sky_sums(f, 0, nvec, st, sh);
    __syncthreads();
  }
  if (tid != 0) return;
  st.arrived = 0;
  if (a.n == 0) {
    // nothing kept: the last statistics stay
    st = state[i];
    st.arrived = 0;
    st.done = 1;
    if (iter == 1) st.mu = st.sigma = 0.0;
  } else {
    // an unchanged set ends the clipping
    st.done = iter >= kSkyIters || (iter > 1 && a.changed == 0);
    st.plo = st.lo;
    st.phi = st.hi;
    kept_interval(st.mu, __dmul_rn(kKappa, st.sigma), &st.lo, &st.hi);
    set_range(st, st.mu, (kKappa + 0.1) * st.sigma);
  }
  state[i] = st;
}

template <typename T>
__device__ inline T to_store(float v);
template <>
__device__ inline float to_store<float>(float v) { return v; }
template <>
__device__ inline __half to_store<__half>(float v) { return __float2half_rn(v); }
template <>
__device__ inline __nv_bfloat16 to_store<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// I = (R - mu) * (1/sigma) as FP64 gives it, rounded to FP32; NaN -> 0;
// optional clip.  The FP64 pipe would take 7 times as long as the copy, so
// the value is formed in pairs of FP32 numbers (mu as three, 1/sigma as two:
// relative error below 2^-44), and where a relative change of 2^-42 would
// alter the rounded result (about one pixel in 10^5), or the range of FP32 is
// left, FP64 decides: the stored values are those of the FP64 formula.  (A
// frame whose mu or 1/sigma has no such parts, as they fall below or beyond
// FP32, has ih = NaN: no pixel of it is sure.)
// 2048^2 x 256 FP32: 1.91 ms, 4.5 TB/s (FP64 throughout: 8.65 ms).
struct NormFrame {
  double mu, inv;
  float mh, ml, mll, ih, il;
  bool zero;
};

__device__ __forceinline__ float normalize64(float r, const NormFrame& f) {
  return (float)__dmul_rn(__dsub_rn((double)r, f.mu), f.inv);
}

// The pair arithmetic; *sure: its result is that of normalize64.
__device__ __forceinline__ float normalize_pair(float r, const NormFrame& f, bool* sure) {
  // a + e = r - mh exactly; (dh, dl) = r - mu
  const float a = __fsub_rn(r, f.mh);
  const float z = __fsub_rn(a, r);
  const float e = __fsub_rn(__fsub_rn(r, __fsub_rn(a, z)), __fadd_rn(f.mh, z));
  const float dh = __fsub_rn(a, f.ml);
  const float y = __fsub_rn(dh, a);
  const float g = __fsub_rn(__fsub_rn(a, __fsub_rn(dh, y)), __fadd_rn(f.ml, y));
  const float dl = __fadd_rn(__fsub_rn(g, f.mll), e);
  const float q = __fmul_rn(dh, f.ih);
  const float c = __fmaf_rn(dl, f.ih, __fmaf_rn(dh, f.il, __fmaf_rn(dh, f.ih, -q)));
  const float tol = __fmul_rn(fabsf(q), 0x1p-42f);
  const float v = __fadd_rn(q, __fadd_rn(c, tol));
  // (dh that lost most of its bits, and results near the ends of the range)
  *sure = v == __fadd_rn(q, __fsub_rn(c, tol)) && fabsf(q) > 0x1p-80f &&
                    fabsf(q) < 0x1p100f && fabsf(dh) > fabsf(f.mh) * 0x1p-22f &&
                    fabsf(dh) > 0x1p-60f && fabsf(dh) < 0x1p100f;
  // r = mu, a masked pixel, a frame without deviation: 0
  const bool none = !(fabsf(r) <= 3.402823466e38f) || f.zero;
  *sure = *sure || none || (dh == 0.0f && dl == 0.0f && q == 0.0f);
  return none ? 0.0f : v;
}

// |v|'s bits, which order as the magnitudes do, an infinity above the finite
// ones and a NaN above both.  The run kernel's moves between running sums carry
// either to outputs that never read the pixel, so both have to reach its
// margin; in the other kernels a NaN stays with the outputs that read it, as in
// the direct gather, and counts as 0.
__device__ __forceinline__ unsigned mag(float v, bool nan) {
  const unsigned b = __float_as_uint(v) & 0x7fffffffu;
  return b > 0x7f800000u && !nan ? 0u : b;
}

// The warps' largest magnitude into *absmax.
__device__ __forceinline__ void put_max(unsigned top, unsigned* absmax) {
  const unsigned m = __reduce_max_sync(0xffffffffu, top);
  if ((threadIdx.x & 31) == 0 && m > *absmax) atomicMax(absmax, m);
}

__global__ void __launch_bounds__(256)
    k_absmax(const float* __restrict__ x, int64_t n, bool nan, unsigned* __restrict__ absmax) {
  const int64_t head = min(n, (int64_t)((16 - (reinterpret_cast<uintptr_t>(x) & 15)) & 15) / 4);
  const float4* v = reinterpret_cast<const float4*>(x + head);
  const int64_t nv = (n - head) / 4, tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned top = 0u;
  if (tid < head) top = mag(x[tid], nan);
  if (tid < n - head - 4 * nv) top = max(top, mag(x[head + 4 * nv + tid], nan));
#pragma unroll 4
  for (int64_t j = tid; j < nv; j += (int64_t)gridDim.x * blockDim.x) {
    const float4 q = __ldg(v + j);
    top = max(top, max(max(mag(q.x, nan), mag(q.y, nan)), max(mag(q.z, nan), mag(q.w, nan))));
  }
  put_max(top, absmax);
}

__global__ void k_margins(const FieldDev* __restrict__ fds, int n, int mode,
                          const unsigned* __restrict__ absmax, float* __restrict__ margin,
                          int* __restrict__ use, Counters* __restrict__ ctr) {
  const int f = threadIdx.x;
  bool ok = true;
  if (f < n) {
    const FieldDev& d = fds[f];
    const float m = margin_of(mode, __uint_as_float(absmax[f]), d.N, d.thr[d.N]);
    margin[f] = m;
    ok = margin_ok(mode, m, d.nmin, d.thr[d.nmin]);
  }
  const int all = __syncthreads_and(ok);
  if (f == 0) {
    *use = all;
    if (!all && mode == ST_BILINEAR) atomicOr(&ctr->error, ERR_MARGIN);
  }
}

template <typename T>
__global__ void __launch_bounds__(256)
    k_normalize_store(const float* __restrict__ raw, int W, int H, int normalize, float cr_clip,
                      const SkyState* __restrict__ state, T* __restrict__ cube, int pitch,
                      double* __restrict__ mu_out, double* __restrict__ sigma_out,
                      unsigned* __restrict__ absmax, bool nan) {
  const int i = blockIdx.y;
  const int64_t npix = (int64_t)W * H;
  const float* x = raw + (int64_t)i * npix;
  T* o = cube + (int64_t)i * pitch * H;
  // (one thread forms the frame's constants: FP64)
  __shared__ NormFrame s_f;
  if (normalize && threadIdx.x == 0) {
    NormFrame f;
    f.mu = state[i].mu;
    const double sg = state[i].sigma;
    f.zero = !(sg > 0.0);
    f.inv = f.zero ? 0.0 : __drcp_rn(sg);
    f.mh = (float)f.mu;
    f.ml = (float)(f.mu - (double)f.mh);
    f.mll = (float)(f.mu - (double)f.mh - (double)f.ml);
    f.ih = (float)f.inv;
    f.il = (float)(f.inv - (double)f.ih);
    // (il of a smaller ih would be subnormal and lose the bits it stands for)
    if (!(f.ih >= 0x1p-100f && f.ih <= 3.402823466e38f) ||
        f.mu - (double)f.mh - (double)f.ml != (double)f.mll)
      f.ih = __int_as_float(0x7fc00000);
    s_f = f;
    if (blockIdx.x == 0) {
      if (mu_out) mu_out[i] = f.mu;
      if (sigma_out) sigma_out[i] = sg;
    }
  }
  __syncthreads();
  const NormFrame f = s_f;
  auto clipped = [&](float v) { return cr_clip > 0.0f && fabsf(v) > cr_clip ? 0.0f : v; };
  unsigned top = 0u;
  // four pixels; the FP64 formula sits behind one branch
  auto values = [&](float4 r) {
    if (!normalize) return r;
    bool sx, sy, sz, sw;
    float4 v = make_float4(normalize_pair(r.x, f, &sx), normalize_pair(r.y, f, &sy),
                           normalize_pair(r.z, f, &sz), normalize_pair(r.w, f, &sw));
    if (!(sx && sy && sz && sw)) {
#pragma unroll 1
      for (int k = 0; k < 4; ++k) {
        const float w = sx ? v.x : normalize64(r.x, f);
        v = make_float4(v.y, v.z, v.w, w);
        r = make_float4(r.y, r.z, r.w, 0.0f);
        sx = sy;
        sy = sz;
        sz = sw;
      }
    }
    return make_float4(clipped(v.x), clipped(v.y), clipped(v.z), clipped(v.w));
  };
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  // frames on 16-byte boundaries: four pixels a thread (one load, one store)
  if (pitch == W && npix % 4 == 0 && ((reinterpret_cast<uintptr_t>(raw) & 15) | (reinterpret_cast<uintptr_t>(cube) & 15)) == 0) {
    for (int64_t j = first; j < npix / 4; j += stride) {
      const float4 r = __ldcs(reinterpret_cast<const float4*>(x) + j);
      const float4 w = values(r);
      alignas(16) T v[4] = {to_store<T>(w.x), to_store<T>(w.y), to_store<T>(w.z),
                            to_store<T>(w.w)};
      if (absmax)
#pragma unroll
        for (int k = 0; k < 4; ++k) top = max(top, mag((float)v[k], nan));
      if constexpr (sizeof(T) == 4)
        reinterpret_cast<uint4*>(o)[j] = *reinterpret_cast<const uint4*>(v);
      else
        reinterpret_cast<uint2*>(o)[j] = *reinterpret_cast<const uint2*>(v);
    }
    if (absmax) put_max(top, absmax);
    return;
  }
  // else pixels in their order whatever the rows' length, eight of a thread in
  // flight, 256 apart; the row is carried along (W = 37, 2000 x 64 frames to
  // FP16 rows of 40: 8 us; a row a block left most of its threads idle: 110)
  constexpr int kFlight = 8;
  constexpr uint32_t kRound = 256u * kFlight;
  const uint32_t n = (uint32_t)npix, w = (uint32_t)W, pad = (uint32_t)(pitch - W);
  const uint32_t hop = (gridDim.x - 1) * kRound;
  const uint32_t step_y = 256u / w, step_x = 256u - step_y * w;
  const uint32_t hop_y = hop / w, hop_x = hop - hop_y * w;
  uint32_t j = blockIdx.x * kRound + threadIdx.x, y = j / w, c = j - y * w;
  auto ahead = [&](uint32_t dy, uint32_t dx) {
    y += dy;
    c += dx;
    if (c >= w) {
      c -= w;
      ++y;
    }
  };
  auto round = [&](auto whole) {
    float r[kFlight];
#pragma unroll
    for (int k = 0; k < kFlight; ++k)
      r[k] = whole() || j + 256u * k < n ? __ldcs(x + j + 256u * k) : 0.0f;
#pragma unroll
    for (int k = 0; k < kFlight; k += 4) {
      const float4 v = values(make_float4(r[k], r[k + 1], r[k + 2], r[k + 3]));
      const float v4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t at = j + 256u * (k + q);
        if (whole() || at < n) {
          const T put = to_store<T>(v4[q]);
          if (absmax) top = max(top, mag((float)put, nan));
          o[at + y * pad] = put;
        }
        ahead(step_y, step_x);
      }
    }
    ahead(hop_y, hop_x);
  };
  for (; j + (kRound - 256u) < n; j += kRound + hop) round(std::true_type{});
  for (; j < n; j += kRound + hop) round(std::false_type{});
  if (absmax) put_max(top, absmax);
}

}  // namespace

int launch_shift_tables(const double* d_t, int N, double t_ref, double vx0, double dvx, int nvx,
                        double vy0, double dvy, int nvy, int mode, int32_t* sx, int32_t* sy,
                        float* fx, float* fy, cudaStream_t s) {
  int64_t nx = (int64_t)N * nvx, ny = (int64_t)N * nvy;
  k_shift_tables<<<(unsigned)((nx + 255) / 256), 256, 0, s>>>(d_t, N, t_ref, vx0, dvx, nvx, mode,
                                                               sx, fx);
  k_shift_tables<<<(unsigned)((ny + 255) / 256), 256, 0, s>>>(d_t, N, t_ref, vy0, dvy, nvy, mode,
                                                               sy, fy);
  return 2;
}

size_t sky_partial_doubles(int N) {
  return (size_t)N * (kSkyBlocks * sizeof(SkyPartial) + sizeof(SkyState)) / sizeof(double);
}

int launch_normalize(const float* raw, int N, int W, int H, int normalize, float cr_clip,
                     int storage, void* cube, int pitch, double* mu, double* sigma,
                     double* partial, unsigned* absmax, bool nan, cudaStream_t s) {
  const int64_t npix = (int64_t)W * H;
  int launches = 0;
  SkyPartial* parts = reinterpret_cast<SkyPartial*>(partial);
  SkyState* state = reinterpret_cast<SkyState*>(parts + (size_t)N * kSkyBlocks);
  if (normalize) {
    k_sky_guess<<<N, kSkyThreads, 0, s>>>(raw, npix, state);
    // blocks per frame: 256 pixels a thread (a block's reduction costs as much
    // as 10 pixels a thread), fewer where the frames would not fill the chip
    const int64_t want = std::max((npix + 65535) / 65536, (int64_t)((8 * 152 + N - 1) / N));
    const int64_t most = std::min((int64_t)kSkyBlocks, (npix + 4095) / 4096);
    const int blocks = (int)std::max((int64_t)1, std::min(want, most));
    for (int it = 1; it <= kSkyIters; ++it)
      k_sky_pass<<<dim3(blocks, N), kSkyThreads, 0, s>>>(raw, npix, it, state, parts);
    launches += 1 + kSkyIters;
  }
  // 16 pixels a thread, 8 where the frames would not fill the chip
  const int64_t rounds = (npix + 2047) / 2048;
  const int64_t want = std::max((rounds + 1) / 2, (int64_t)((8 * 152 + N - 1) / N));
  const int bx = (int)std::min((int64_t)4096, std::min(rounds, want));
  dim3 g(bx, N);
  switch (storage) {
    case ST_F32:
      k_normalize_store<float><<<g, 256, 0, s>>>(raw, W, H, normalize, cr_clip, state,
                                                 (float*)cube, pitch, mu, sigma, absmax, nan);
      break;
    case ST_F16:
      k_normalize_store<__half><<<g, 256, 0, s>>>(raw, W, H, normalize, cr_clip, state,
                                                  (__half*)cube, pitch, mu, sigma, absmax, nan);
      break;
    default:
      k_normalize_store<__nv_bfloat16><<<g, 256, 0, s>>>(raw, W, H, normalize, cr_clip, state,
                                                         (__nv_bfloat16*)cube, pitch, mu, sigma,
                                                         absmax, nan);
      break;
  }
  return launches + 1;
}

int launch_absmax(const float* x, int64_t n, bool nan, unsigned* absmax, cudaStream_t s) {
  const int64_t blocks = std::min((int64_t)8 * 152, (n + 4095) / 4096);
  k_absmax<<<(unsigned)std::max((int64_t)1, blocks), 256, 0, s>>>(x, n, nan, absmax);
  return 1;
}

int launch_margins(const FieldDev* fds, int n, int mode, const unsigned* absmax, float* margin,
                   int* use, Counters* ctr, cudaStream_t s) {
  k_margins<<<1, 256, 0, s>>>(fds, n, mode, absmax, margin, use, ctr);
  return 1;
}

}  // namespace st
