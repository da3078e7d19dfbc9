// k_refine.cu — differentiable refinement of candidates (forward + adjoint).
//
// Not in the paper: a continuous refinement of the grid detections of the
// synthetic-tracking search (Sec. 2.1).  For theta = (vx, vy, x0, y0, F) and a
// 64 x 64 output cutout centred on the candidate pixel:
//   S(p)   = sum_i B_i(p + v dt_i)      bilinear stack, zero outside the frame
//   g(p)   = exp(-|p - (x0, y0)|^2 / (2 s^2)),  s = FWHM / (2 sqrt(2 ln 2))
//   J      = F <g, S> - F^2 N <g, g> / 2,  SNR = <g, S> / sqrt(N <g, g>)
// and the adjoint: dJ/dF = <g,S> - F N <g,g>; dJ/dx0 = F <dg/dx0, S> -
// F^2 N <g, dg/dx0>; dJ/dvx = F sum_p g(p) sum_i dt_i dB_i/dX (the slope of
// the bilinear cell).  The samples and their derivatives are recomputed on
// every evaluation, never stored.  A frame's shift v dt_i is formed to
// FP64 accuracy (the time offset held as an FP32 pair, the product with an
// exact FMA error term) and split into its integer part and FP32 fraction.
//
// Optimisers (maximise J with F at its optimum <g,S>/(N <g,g>) each step):
// Adam on (vx, vy, x0, y0), or Gauss-Newton: J is the log-likelihood of the
// frames under the model F g(p - (x0, y0) - v dt_i), so -Hessian is replaced
// by the model's J^T J, whose entries need only template sums over the
// cutout (<g,g>, <g,Gx>, <g,Gy>, <Gx,Gx>, <Gy,Gy>, <Gx,Gy> with G = dg/dx0,
// dg/dy0) and sum dt, sum dt^2; F is profiled out by the Schur complement of
// its entry and (vx, vy, x0, y0) move by the solution of
// (Hs + damping diag(Hs)) delta = dJ/d(vx, vy, x0, y0).
//
// One CTA per candidate.  Every pixel of the cutout shares a frame's shift,
// so a frame contributes one footprint of 65 x 65 taps; a TMA ring of S
// frames stages those footprints in shared memory ahead of use (zero fill
// outside the image takes the place of bounds tests; the box x origin is
// rounded down to 16 bytes and the remainder is an index offset).  Thread t
// owns cutout column t%64 and its 16 rows (t/64)*16.., so a warp reads 32
// consecutive words of a box row, and handles its rows in pairs (k, k + 8):
// tap rows q and q + 8 are one register pair, so the differences d = a1 - a0,
// the horizontal interpolations h = a0 + fx d, their steps e = h' - h, the
// slopes and the sums S are paired FP32 operations; a frame's <g, slope> is
// added up row by row (a change of its rounding alone moves a Gauss-Newton
// path across the kinks of the bilinear stack).  A ninth warp forms a
// frame's shift when it issues the copy and leaves the fractions beside it;
// each consumer warp releases a slot by itself (a consumer that issues the
// copies paces all others: 51 ms against 48).  Reductions use a fixed-order block tree.  Every wait is
// bounded in time.
//
// What bounds it: per frame and cutout 272 shared-memory wavefronts and 58
// paired and 32 single operations a warp on the FP32 pipe, which paired FMAs of
// three distinct register pairs reach at 0.67 of its rate (measured: 85 against
// 127 for adds, in operations per clock and SM): about 400 clocks of the 600 it
// takes.  Half the
// rows copied, 3 or 5 stages or three CTAs an SM: the same time.  4096
// candidates x 300 frames x 21 evaluations: 62.5 ms with scalar operations, 50.1 (48.2 with
// the slopes' sums paired too).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <vector>

#include "st_internal.h"
#include "st_sample.cuh"
#include "st_tma.cuh"

namespace st {

namespace {

constexpr int kCut = 64;        // cutout side
constexpr int kThreads = 256;   // consumers: 8 warps
constexpr int kBlock = kThreads + 32;  // and the warp that issues the copies
constexpr int kPix = kCut * kCut / kThreads;  // 16 rows of one column per thread
constexpr int kHalf = kPix / 2;               // row pairs (k, k + 8)
constexpr int kSums = 11;
constexpr int kBoxH = kCut + 1; // footprint rows
constexpr uint64_t kWaitNs = 2000000000ull;  // wait limit: 2 s of wall-clock time

template <typename T>
constexpr int stages_for() { return sizeof(T) == 4 ? 4 : 6; }
template <typename T>
constexpr int align_elems() { return 16 / (int)sizeof(T); }
// footprint columns: 65 taps and up to 3 (7 for 16-bit types) of alignment
template <typename T>
constexpr int box_w() { return kCut + align_elems<T>(); }
template <typename T>
constexpr int box_bytes() { return ((box_w<T>() * kBoxH * (int)sizeof(T)) + 127) & ~127; }

struct RefineArgs {
  const FieldDev* fds;          // device field descriptors
  const CUtensorMap* maps;      // per field: tiled map of the cube, box kBoxW x kBoxH x 1
  const double* const* times;   // per field: device FP64 timestamps
  const double* t_ref;          // per field
  const float* theta_in;        // [n][5] (eval mode)
  const int32_t* centre_in;     // [n][2] (eval mode)
  const int32_t* field_in;      // [n]    (eval mode)
  const st_candidate* cand;     // [n]    (optimise mode)
  const double* grid;           // per field: vx0, dvx, vy0, dvy (optimise mode)
  const uint32_t* order;        // the candidates in the order they are taken (or NULL)
  int64_t n;
  float inv2s2, inv_s2;
  int steps;
  int optimizer;                // 0: Adam, 1: Gauss-Newton (optimise mode)
  float lr_pos, lr_vel;         // Adam learning rates; Gauss-Newton: lr_pos = damping
  float* J;
  float* snr;
  float* grad;                  // [n][5] or null
  st_refined* out;              // optimise mode
  int* err;                     // timeout flag
};

template <typename T>
__device__ __forceinline__ float ld_s(const T* p);
template <>
__device__ __forceinline__ float ld_s<float>(const float* p) { return *p; }
template <>
__device__ __forceinline__ float ld_s<__half>(const __half* p) { return __half2float(*p); }
template <>
__device__ __forceinline__ float ld_s<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __bfloat162float(*p);
}

// Fixed-order reduction of kSums values over the consumers; result valid in
// thread 0.  (The issuing warp meets its two barriers.)
__device__ void block_sum(float (&v)[kSums], float* sh) {
#pragma unroll
  for (int k = 0; k < kSums; ++k)
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], d);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < kSums; ++k) sh[warp * kSums + k] = v[k];
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = 0; k < kSums; ++k) {
      float s = 0.0f;
      for (int w = 0; w < kThreads / 32; ++w) s += sh[w * kSums + k];
      v[k] = s;
    }
  __syncthreads();
}

__device__ void objective(const float (&s)[kSums], int N, float F, float* J, float* snr,
                          float (&gr)[5]) {
  const float nf = (float)N;
  *J = F * s[0] - 0.5f * F * F * nf * s[1];
  *snr = s[1] > 0.0f ? s[0] / sqrtf(nf * s[1]) : 0.0f;
  gr[0] = F * s[6];
  gr[1] = F * s[7];
  gr[2] = F * s[2] - F * F * nf * s[4];
  gr[3] = F * s[3] - F * F * nf * s[5];
  gr[4] = s[0] - F * nf * s[1];
}

// A frame's shift for velocity (vx, vy): integer parts and fractions.
struct Shift {
  int ux, uy;
  float fx, fy;
};
// floor and fraction of v (dt_hi + dt_lo) without FP64 arithmetic: p = fl(v
// dt_hi) and its exact rounding error (one FMA) plus v dt_lo give the product
// as p + q to about 2^-46 relative; p - floor(p) is exact below 2^23 px, and
// the fraction is (p - floor(p)) + q rounded to FP32, moved into [0, 1).
__device__ __forceinline__ void split_shift(float v, float dt_hi, float dt_lo, int* u, float* f) {
  const float p = v * dt_hi;
  const float q = __fmaf_rn(v, dt_lo, __fmaf_rn(v, dt_hi, -p));
  float fl = floorf(p);
  float r = (p - fl) + q;
  if (r < 0.0f) {
    fl -= 1.0f;
    r += 1.0f;
  } else if (r >= 1.0f) {
    fl += 1.0f;
    r -= 1.0f;
  }
  *u = (int)fl;
  *f = r;
}
__device__ __forceinline__ Shift frame_shift(float vx, float vy, float dt_hi, float dt_lo) {
  Shift s;
  split_shift(vx, dt_hi, dt_lo, &s.ux, &s.fx);
  split_shift(vy, dt_hi, dt_lo, &s.uy, &s.fy);
  return s;
}

// Solves the 4 x 4 system A x = b by Gaussian elimination with partial
// pivoting (FP64, in place).  Returns false for a (near) singular matrix.
__device__ bool solve4(double (&A)[4][4], double (&b)[4]) {
  for (int c = 0; c < 4; ++c) {
    int piv = c;
    for (int r = c + 1; r < 4; ++r)
      if (fabs(A[r][c]) > fabs(A[piv][c])) piv = r;
    if (!(fabs(A[piv][c]) > 1e-300)) return false;
    if (piv != c) {
      for (int k = 0; k < 4; ++k) {
        const double tmp = A[c][k];
        A[c][k] = A[piv][k];
        A[piv][k] = tmp;
      }
      const double tb = b[c];
      b[c] = b[piv];
      b[piv] = tb;
    }
    for (int r = c + 1; r < 4; ++r) {
      const double f = A[r][c] / A[c][c];
      for (int k = c; k < 4; ++k) A[r][k] -= f * A[c][k];
      b[r] -= f * b[c];
    }
  }
  for (int c = 3; c >= 0; --c) {
    double v = b[c];
    for (int k = c + 1; k < 4; ++k) v -= A[c][k] * b[k];
    b[c] = v / A[c][c];
  }
  return true;
}

// One Gauss-Newton step of (vx, vy, x0, y0) (in th[0..3]) at flux F from the
// block sums s (template sums s[1] = <g,g>, s[4] = <g,Gx>, s[5] = <g,Gy>,
// s[8] = <Gx,Gx>, s[9] = <Gy,Gy>, s[10] = <Gx,Gy>), the gradient gr and the
// frames' sum dt and sum dt^2.  A singular system leaves th unchanged.
__device__ void gauss_newton_step(float* th, const float (&s)[kSums], const float (&gr)[5],
                                  float F, int N, double T1, double T2, float damping) {
  const double f = F, f2 = f * f, n = N;
  const double xx = s[8], yy = s[9], xy = s[10], gx = s[4], gy = s[5], gg = s[1];
  const double H[5][5] = {{f2 * T2 * xx, f2 * T2 * xy, f2 * T1 * xx, f2 * T1 * xy, f * T1 * gx},
                          {f2 * T2 * xy, f2 * T2 * yy, f2 * T1 * xy, f2 * T1 * yy, f * T1 * gy},
                          {f2 * T1 * xx, f2 * T1 * xy, f2 * n * xx, f2 * n * xy, f * n * gx},
                          {f2 * T1 * xy, f2 * T1 * yy, f2 * n * xy, f2 * n * yy, f * n * gy},
                          {f * T1 * gx, f * T1 * gy, f * n * gx, f * n * gy, n * gg}};
  if (!(H[4][4] > 0.0)) return;
  double A[4][4], b[4];
  for (int a = 0; a < 4; ++a) {
    for (int c = 0; c < 4; ++c) A[a][c] = H[a][c] - H[a][4] * H[4][c] / H[4][4];
    b[a] = gr[a];
  }
  for (int a = 0; a < 4; ++a) A[a][a] += (double)damping * A[a][a];
  if (!solve4(A, b)) return;
  for (int a = 0; a < 4; ++a) th[a] = (float)((double)th[a] + b[a]);
}

template <typename T, bool OPT>
__global__ void __launch_bounds__(kBlock, 2) k_refine(RefineArgs a) {
  constexpr int S = stages_for<T>();
  constexpr int kBox = box_bytes<T>();
  constexpr int kAl = align_elems<T>(), kBoxW = box_w<T>();
  extern __shared__ __align__(128) unsigned char dsm_raw[];
  __shared__ __align__(8) uint64_t full[S];
  __shared__ __align__(8) uint64_t empty[S];  // the warps that are done with a slot
  __shared__ float4 s_frame[S];  // a slot's frame: fx, fy, dt, column offset in the box
  __shared__ float sh[(kThreads / 32) * kSums];
  __shared__ float th[5];
  __shared__ double s_t12[2];   // sum dt, sum dt^2 (Gauss-Newton)
  unsigned char* ring = dsm_raw + ((128u - (smem_u32(dsm_raw) & 127u)) & 127u);
  const int64_t c = a.order ? (int64_t)a.order[blockIdx.x] : (int64_t)blockIdx.x;
  if (c >= a.n) return;
  int fi, cx, cy;
  if (OPT) {
    const st_candidate cd = a.cand[c];
    fi = cd.field;
    cx = cd.x;
    cy = cd.y;
  } else {
    fi = a.field_in[c];
    cx = a.centre_in[2 * c];
    cy = a.centre_in[2 * c + 1];
  }
  const FieldDev& fd = a.fds[fi];
  const int N = fd.N;
  // time offsets dt_i = t_i - t_ref as FP32 pairs: sdt (rounded) + sdt_lo
  float* sdt = reinterpret_cast<float*>(ring + (size_t)S * kBox);
  float* sdt_lo = sdt + N;
  const CUtensorMap* map = a.maps + fi;
  const int tid = threadIdx.x;
  const bool gn = OPT && a.optimizer == 1;
  {
    const double* t = a.times[fi];
    const double t_ref = a.t_ref[fi];
    double p1 = 0.0, p2 = 0.0;
    for (int j = tid; j < N; j += kBlock) {
      const double d = t[j] - t_ref;
      sdt[j] = (float)d;
      sdt_lo[j] = (float)(d - (double)(float)d);
      p1 += d;
      p2 += d * d;
    }
    if (gn) {
      // sum dt and sum dt^2 in FP64, fixed-order block reduction
      for (int d = 16; d > 0; d >>= 1) {
        p1 += __shfl_down_sync(0xffffffffu, p1, d);
        p2 += __shfl_down_sync(0xffffffffu, p2, d);
      }
      __shared__ double s_p[2 * (kBlock / 32)];
      if ((tid & 31) == 0) {
        s_p[2 * (tid >> 5)] = p1;
        s_p[2 * (tid >> 5) + 1] = p2;
      }
      __syncthreads();
      if (tid == 0) {
        double a1 = 0.0, a2 = 0.0;
        for (int w = 0; w < kBlock / 32; ++w) {
          a1 += s_p[2 * w];
          a2 += s_p[2 * w + 1];
        }
        s_t12[0] = a1;
        s_t12[1] = a2;
      }
    }
  }
  if (tid == 0) {
    tma_prefetch_desc(map);
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kThreads / 32);
    }
    mbar_init_fence();
    if (OPT) {
      const st_candidate cd = a.cand[c];
      const double* gr = a.grid + 4 * fi;
      th[0] = (float)(gr[0] + (cd.k % fd.nvx) * gr[1]);
      th[1] = (float)(gr[2] + (cd.k / fd.nvx) * gr[3]);
      th[2] = (float)cd.x;
      th[3] = (float)cd.y;
      th[4] = 0.0f;
    } else {
      for (int k = 0; k < 5; ++k) th[k] = a.theta_in[5 * c + k];
    }
  }
  __syncthreads();

  if (tid >= kThreads) {
    // ---- the issuing warp: frame i (sequence number q over all evaluations)
    // into ring slot q % S once every consumer warp has left the slot
    const int steps = OPT ? a.steps : 0;
    uint32_t q = 0;
    bool ok = true;
    for (int step = 0; step <= steps; ++step) {
      const float vx = th[0], vy = th[1];
      if (tid == kThreads)
        for (int i = 0; i < N && ok; ++i, ++q) {
          const int slot = (int)(q % S);
          if (q >= (uint32_t)S && !mbar_wait(&empty[slot], (q / S - 1) & 1u, kWaitNs)) {
            ok = false;  // the frames that are not issued end the consumers' waits
            break;
          }
          const Shift f = frame_shift(vx, vy, sdt[i], sdt_lo[i]);
          const int cu0 = cx - kCut / 2 + f.ux, cv0 = cy - kCut / 2 + f.uy;
          const int bx = cu0 & ~(kAl - 1);  // 16-byte aligned box origin (floor, also below 0)
          s_frame[slot] = make_float4(f.fx, f.fy, sdt[i], __int_as_float(cu0 - bx));
          mbar_arrive_expect_tx(&full[slot], (uint32_t)(kBoxW * kBoxH * sizeof(T)));
          tma_load_3d(ring + (size_t)slot * kBox, map, bx, cv0, i, &full[slot]);
        }
      ok = __syncthreads_and(ok);
      if (!ok) break;
      __syncthreads();  // (the two barriers of block_sum)
      __syncthreads();
      __syncthreads();  // the new parameters
    }
    // after a wait that gave up: the copies already issued land (bounded)
    // before exit; only the latest phase of each slot can be waited on
    if (!ok && tid == kThreads)
      for (uint32_t k = q > (uint32_t)S ? q - S : 0; k < q; ++k)
        mbar_wait(&full[k % S], (k / S) & 1u, kWaitNs);
    return;
  }

  const int col = tid % kCut;
  const int row0 = (tid / kCut) * kPix;
  const float fcol = (float)(cx - kCut / 2 + col);
  const float frow0 = (float)(cy - kCut / 2 + row0);
  float sums[kSums];
  float m[4] = {0, 0, 0, 0}, v2[4] = {0, 0, 0, 0};
  const int steps = OPT ? a.steps : 0;
  uint32_t q0 = 0;  // frames staged before this evaluation
  bool ok = true;
  for (int step = 0; step <= steps && ok; ++step) {
    const float x0 = th[2], y0 = th[3];
    float2 S2[kHalf], g2[kHalf];
    const float dx = fcol - x0;
    auto weight = [&](int k) {
      const float dy = frow0 + (float)k - y0;
      return expf(-(dx * dx + dy * dy) * a.inv2s2);
    };
#pragma unroll
    for (int k = 0; k < kHalf; ++k) {
      S2[k] = make_float2(0.0f, 0.0f);
      g2[k] = make_float2(weight(k), weight(k + kHalf));
    }
    float dvx = 0.0f, dvy = 0.0f;
    for (int i = 0; i < N; ++i) {
      const uint32_t q = q0 + i;
      const int slot = (int)(q % S);
      ok = mbar_wait(&full[slot], (q / S) & 1u, kWaitNs);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;  // (the other warps' waits run out too)
      const float4 fr = s_frame[slot];
      const T* box = reinterpret_cast<const T*>(ring + (size_t)slot * kBox) +
                     (size_t)row0 * kBoxW + __float_as_int(fr.w) + col;
      const float2 fx2 = make_float2(fr.x, fr.x), fy2 = make_float2(fr.y, fr.y);
      const float2 neg = make_float2(-1.0f, -1.0f);
      // tap rows q and q + 8 of the column and its right neighbour
      float2 hp, dp;
      // <g, slope in x> and <g, slope in y> in row order: rows 0..7 as they come,
      // then rows 8..15, whose slopes wait in registers
      float gdx = 0.0f, gdy = 0.0f, sx[kHalf], sy[kHalf];
#pragma unroll
      for (int k = 0; k <= kHalf; ++k) {
        const T* r = box + k * kBoxW;
        const T* r8 = r + kHalf * kBoxW;
        const float2 b0 = make_float2(ld_s<T>(r), ld_s<T>(r8));
        const float2 b1 = make_float2(ld_s<T>(r + 1), ld_s<T>(r8 + 1));
        const float2 d = __ffma2_rn(b0, neg, b1);   // b1 - b0, exact product
        const float2 h = __ffma2_rn(fx2, d, b0);
        if (k > 0) {
          const float2 e = __ffma2_rn(hp, neg, h);
          S2[k - 1] = __fadd2_rn(S2[k - 1], __ffma2_rn(fy2, e, hp));
          const float2 u = __ffma2_rn(fy2, __ffma2_rn(dp, neg, d), dp);  // (1-fy) dp + fy d
          gdx = __fmaf_rn(g2[k - 1].x, u.x, gdx);
          gdy = __fmaf_rn(g2[k - 1].x, e.x, gdy);
          sx[k - 1] = u.y;
          sy[k - 1] = e.y;
        }
        hp = h;
        dp = d;
      }
      __syncwarp();
      if ((tid & 31) == 0) mbar_arrive(&empty[slot]);
#pragma unroll
      for (int k = 0; k < kHalf; ++k) {
        gdx = __fmaf_rn(g2[k].y, sx[k], gdx);
        gdy = __fmaf_rn(g2[k].y, sy[k], gdy);
      }
      dvx += fr.z * gdx;
      dvy += fr.z * gdy;
    }
    ok = __syncthreads_and(ok);
    if (!ok) {
      if (tid == 0) atomicOr(a.err, 1);
      break;
    }
    q0 += (uint32_t)N;
#pragma unroll
    for (int k = 0; k < kSums; ++k) sums[k] = 0.0f;
#pragma unroll
    for (int k = 0; k < kPix; ++k) {
      const float dy = frow0 + (float)k - y0;
      const float g = k < kHalf ? g2[k % kHalf].x : g2[k % kHalf].y;
      const float Sk = k < kHalf ? S2[k % kHalf].x : S2[k % kHalf].y;
      const float gx = g * dx * a.inv_s2;
      const float gy = g * dy * a.inv_s2;
      sums[0] += g * Sk;
      sums[1] += g * g;
      sums[2] += gx * Sk;
      sums[3] += gy * Sk;
      sums[4] += g * gx;
      sums[5] += g * gy;
      sums[8] += gx * gx;
      sums[9] += gy * gy;
      sums[10] += gx * gy;
    }
    sums[6] = dvx;
    sums[7] = dvy;
    block_sum(sums, sh);
    if (tid == 0) {
      // F at its optimum <g,S>/(N <g,g>) when optimising (profile likelihood)
      if (OPT) th[4] = sums[1] > 0.0f ? sums[0] / ((float)N * sums[1]) : 0.0f;
      float J, snr, gr[5];
      objective(sums, N, th[4], &J, &snr, gr);
      if (step == steps) {
        if (a.J) a.J[c] = J;
        if (a.snr) a.snr[c] = snr;
        if (a.grad)
          for (int k = 0; k < 5; ++k) a.grad[5 * c + k] = gr[k];
        if (OPT) {
          st_refined r;
          r.vx = th[0];
          r.vy = th[1];
          r.x0 = th[2];
          r.y0 = th[3];
          r.flux = th[4];
          r.snr = snr;
          r.obj = J;
          r.field = fi;
          a.out[c] = r;
        }
      } else if (gn) {
        gauss_newton_step(th, sums, gr, th[4], N, s_t12[0], s_t12[1], a.lr_pos);
      } else {
        // Adam ascent on (vx, vy, x0, y0)
        const float b1 = 0.9f, b2 = 0.999f;
        const float c1 = 1.0f - __powf(b1, (float)(step + 1));
        const float c2 = 1.0f - __powf(b2, (float)(step + 1));
        for (int k = 0; k < 4; ++k) {
          m[k] = b1 * m[k] + (1.0f - b1) * gr[k];
          v2[k] = b2 * v2[k] + (1.0f - b2) * gr[k] * gr[k];
          const float lr = k < 2 ? a.lr_vel : a.lr_pos;
          th[k] += lr * (m[k] / c1) / (sqrtf(v2[k] / c2) + 1e-12f);
        }
      }
    }
    __syncthreads();
  }
}

// Key of a candidate for the order by place: field, band of 32 rows, column.
__global__ void k_refine_keys(const st_candidate* __restrict__ cand, int64_t n, int64_t n_pow2,
                              uint64_t* __restrict__ keys, uint32_t* __restrict__ idx) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_pow2) return;
  uint64_t key = ~0ull;
  if (i < n) {
    const st_candidate c = cand[i];
    key = (uint64_t)(uint32_t)c.field << 48 | (uint64_t)((uint32_t)c.y >> 5 & 0xfffu) << 24 |
          ((uint32_t)c.x & 0xffffffu);
  }
  keys[i] = key;
  idx[i] = i < n ? (uint32_t)i : 0xffffffffu;
}

template <typename T, bool OPT>
void set_smem_attr() {
  static bool done = false;
  if (!done) {
    cudaFuncSetAttribute((const void*)k_refine<T, OPT>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    done = true;
  }
}

}  // namespace

int refine_max_frames() { return 8192; }

int launch_refine(const FieldDev* h_fds, int n_fields, const FieldDev* fds, CUtensorMap* d_maps,
                  const double* const* times, const double* t_ref, const double* grid,
                  int storage, bool optimise, const float* theta, const int32_t* centre,
                  const int32_t* field, const st_candidate* cand, int64_t n, int steps,
                  int optimizer, float fwhm, float lr_pos, float lr_vel, float* J, float* snr,
                  float* grad, st_refined* out, int* err, uint64_t* keys, uint32_t* idx,
                  int64_t sort_cap, cudaStream_t s) {
  if (n <= 0) return 0;
  // tensor maps of the fields' cubes (box: the footprint of one frame)
  std::vector<CUtensorMap> maps(n_fields);
  int max_n = 0;
  for (int f = 0; f < n_fields; ++f) {
    // (rows of the caller's frames, not of a padded copy)
    if ((int64_t)h_fds[f].W * (h_fds[f].storage == ST_F32 ? 4 : 2) % 16 != 0) return -1;
    if (!encode_tile_map(&maps[f], h_fds[f],
                         h_fds[f].storage == ST_F32 ? box_w<float>() : box_w<__half>(), kBoxH)) return -1;
    max_n = h_fds[f].N > max_n ? h_fds[f].N : max_n;
  }
  if (max_n > refine_max_frames()) return -1;
  if (cudaMemcpyAsync(d_maps, maps.data(), sizeof(CUtensorMap) * n_fields,
                      cudaMemcpyHostToDevice, s) != cudaSuccess)
    return -1;
  RefineArgs a{};
  a.fds = fds;
  a.maps = d_maps;
  a.times = times;
  a.t_ref = t_ref;
  a.theta_in = theta;
  a.centre_in = centre;
  a.field_in = field;
  a.cand = cand;
  a.grid = grid;
  a.n = n;
  // More candidates than run at once, taken in the order of their places: CTAs
  // that run together share frame footprints in L2 (4096 candidates x 300
  // frames x 21 evaluations: 57.3 -> 51.0 ms; the sort takes 30 us).
  int launches = 1;
  int64_t pow2 = 1;
  while (pow2 < n) pow2 <<= 1;
  if (cand && n > 304 && n * max_n * (steps + 1) > (1 << 20) && pow2 <= sort_cap) {
    k_refine_keys<<<(unsigned)((pow2 + 255) / 256), 256, 0, s>>>(cand, n, pow2, keys, idx);
    launches += 1 + launch_sort(keys, idx, pow2, s);
    a.order = idx;
  }
  const double sg = fwhm / (2.0 * 1.1774100225154747);  // 2 sqrt(2 ln 2)
  a.inv2s2 = (float)(1.0 / (2.0 * sg * sg));
  a.inv_s2 = (float)(1.0 / (sg * sg));
  a.steps = steps;
  a.optimizer = optimizer;
  a.lr_pos = lr_pos;
  a.lr_vel = lr_vel;
  a.J = J;
  a.snr = snr;
  a.grad = grad;
  a.out = out;
  a.err = err;
  const size_t dt_bytes = 2 * sizeof(float) * (size_t)max_n;
#define ST_REF(T, O)                                                                         \
  do {                                                                                       \
    set_smem_attr<T, O>();                                                                   \
    const size_t smem = (size_t)stages_for<T>() * box_bytes<T>() + dt_bytes + 128;           \
    k_refine<T, O><<<(unsigned)n, kBlock, smem, s>>>(a);                                   \
  } while (0)
  if (storage == ST_F32) {
    if (optimise) ST_REF(float, true); else ST_REF(float, false);
  } else if (storage == ST_F16) {
    if (optimise) ST_REF(__half, true); else ST_REF(__half, false);
  } else {
    if (optimise) ST_REF(__nv_bfloat16, true); else ST_REF(__nv_bfloat16, false);
  }
#undef ST_REF
  return launches;
}

}  // namespace st
