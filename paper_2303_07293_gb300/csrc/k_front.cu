// k_front.cu — the pre-tracking front end of Sec. 2.1 on the device.
//
// * Median star removal: for a group of frames, the per-pixel median over the
//   group (finite values only; NaN marks a masked pixel; an even count takes
//   (a + b) * 0.5 of the two middle values) is subtracted from every frame,
//   removing the stationary high-S/N sources before the shift-and-stack.
// * Frame sums: every n consecutive frames summed in frame order with one
//   FP32 accumulator (a trailing partial group is dropped), for slow movers.
// * 2 x 2 binning: ((p00 + p01) + p10) + p11 per block (flux kept), for fast
//   movers.
//
// All three are HBM-bound streams.  The median kernels give each thread one
// pixel, so a warp reads 32 consecutive pixels of a frame per load
// (coalesced).  Up to 64 frames a sorting network per group size selects the
// median (k_median_select.cu); longer groups bisect its value
// (k_median_long).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "st_internal.h"

namespace st {

namespace {

// ---- median over more than 64 frames
//
// A block takes 32 consecutive pixels: their columns are copied to shared
// memory asynchronously (the cube is read once; rows of 36 words, so that 8
// frames x 4 pixels lie in different banks), and 8 threads a pixel hold a
// share of its samples as integer keys that order like the floats.  The k-th
// smallest key is found by bisection on its value: a step counts the keys at
// or below the middle of the bracket (each thread its own, added up over the
// 8), until the count singles the key out (about log2 of the range over the
// spacing at the median: 10 steps for noise) or the bracket is one value.  No
// step moves data or branches on it.  Masked samples are the highest key and
// never counted.
// Frames that all start on 16 bytes are moved 16 bytes a lane, in and out, as
// 4-byte pieces kept too few bytes in flight.
// What bounds it: the counting, about 12 steps x N x 2 instructions a pixel,
// against 8 N bytes.  1024^2 x 200: 0.498 ms, 3.4 TB/s (4-byte pieces 0.645;
// quickselect in shared memory, one warp a block: 6.5 ms).
constexpr int kMedPix = 32, kMedShare = 8, kMedPitch = 36;

__device__ __forceinline__ int32_t med_key(float x) {
  const int32_t b = __float_as_int(x);
  return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float med_value(int32_t k) {
  return __int_as_float(k ^ ((k >> 31) & 0x7fffffff));
}
// over the 8 lanes of a pixel
__device__ __forceinline__ int sum8(int v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v + __shfl_xor_sync(0xffffffffu, v, 4);
}
__device__ __forceinline__ int min8(int v) {
  v = min(v, __shfl_xor_sync(0xffffffffu, v, 1));
  v = min(v, __shfl_xor_sync(0xffffffffu, v, 2));
  return min(v, __shfl_xor_sync(0xffffffffu, v, 4));
}
__device__ __forceinline__ int max8(int v) { return ~min8(~v); }

// K: keys a thread holds (8 K >= N).  in and out may be the same cube: a block
// has its pixels' whole columns in shared memory before it writes any of them.
template <int K>
__global__ void __launch_bounds__(kMedPix * kMedShare)
    k_median_long(const float* in, int N, int64_t P, float* out, float* __restrict__ median,
                  const bool vec) {
  extern __shared__ __align__(16) float sm[];  // [N][kMedPitch] samples in frame order, [32] medians
  float* med_sh = sm + (size_t)N * kMedPitch;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t p0 = (int64_t)blockIdx.x * kMedPix;
  // (a pixel past the end reads zeros)
  const int row4 = tid / 8, off4 = tid % 8 * 4;  // 16-byte pieces: 8 lanes a frame
  const bool ok4 = p0 + off4 < P;
  if (vec) {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(sm + off4);
    const float* src = ok4 ? in + p0 + off4 : in;
    for (int i = row4; i < N; i += kMedPix)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                       dst + (uint32_t)(i * kMedPitch * 4)),
                   "l"(src + (int64_t)i * P), "r"(ok4 ? 16 : 0)
                   : "memory");
  } else {
    const bool ok = p0 + lane < P;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(sm + lane);
    for (int i = warp; i < N; i += kMedShare) {
      const float* src = ok ? in + (int64_t)i * P + p0 + lane : in;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                       dst + (uint32_t)(i * kMedPitch * 4)),
                   "l"(src), "r"(ok ? 4 : 0)
                   : "memory");
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // lane = 8 pixel + share, 4 pixels a warp
  const int px = 4 * warp + (lane >> 3), share = lane & 7;
  int32_t key[K];
  int n = 0;
  int32_t lo = INT32_MAX, hi = INT32_MIN;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = k * kMedShare + share;
    const float x = i < N ? sm[i * kMedPitch + px] : INFINITY;
    const bool fin = isfinite(x);
    key[k] = fin ? med_key(x) : INT32_MAX;
    n += fin;
    lo = min(lo, key[k]);
    hi = max(hi, fin ? key[k] : INT32_MIN);
  }
  n = sum8(n);
  lo = min8(lo);
  hi = max8(hi);
  // the key of rank k1 lies in (below, hi]: fewer than k1 + 1 keys are at most
  // `below`, and k1 + 1 or more at most hi
  const int k1 = (n - 1) / 2;
  int32_t below = lo - (n > 0);
  bool above = false;  // it is the smallest key above hi (else the largest up to hi)
  bool done = n <= 0;
  while (!__all_sync(0xffffffffu, done)) {
    const int32_t mid = (int32_t)(((int64_t)below + hi) >> 1);
    int c = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) c += key[k] <= mid;
    c = sum8(c);
    if (!done) {
      above = c == k1;
      if (c >= k1) hi = mid;
      else below = mid;
      // (keys that are equal leave a bracket of one value)
      done = above || c == k1 + 1 || (int64_t)hi - below == 1;
    }
  }
  int32_t under = INT32_MIN, over = INT32_MAX;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    under = max(under, key[k] <= hi ? key[k] : INT32_MIN);
    over = min(over, key[k] > hi ? key[k] : INT32_MAX);
  }
  under = max8(under);
  over = min8(over);
  const int32_t a = above ? over : under;
  // the next order statistic: the same value again, or the smallest above it
  int at_most = 0;
  int32_t next = INT32_MAX;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    at_most += key[k] <= a;
    next = min(next, key[k] > a ? key[k] : INT32_MAX);
  }
  at_most = sum8(at_most);
  next = min8(next);
  float med = __int_as_float(0x7fc00000);  // NaN: no finite sample
  if (n > 0) {
    med = med_value(a);
    if (!(n & 1)) med = __fmul_rn(__fadd_rn(med, at_most >= k1 + 2 ? med : med_value(next)), 0.5f);
  }
  if (share == 0) med_sh[px] = med;
  __syncthreads();
  const int64_t p = p0 + lane;
  if (median && warp == 0 && p < P) median[p] = med_sh[lane];
  if (vec) {
    if (!ok4) return;
    const float4 m = *reinterpret_cast<const float4*>(med_sh + off4);
    for (int i = row4; i < N; i += kMedPix) {
      const float4 v = *reinterpret_cast<const float4*>(sm + i * kMedPitch + off4);
      __stcs(reinterpret_cast<float4*>(out + (int64_t)i * P + p0 + off4),
             make_float4(__fsub_rn(v.x, m.x), __fsub_rn(v.y, m.y), __fsub_rn(v.z, m.z),
                         __fsub_rn(v.w, m.w)));
    }
    return;
  }
  if (p >= P) return;
  med = med_sh[lane];
  for (int i = warp; i < N; i += kMedShare)
    out[(int64_t)i * P + p] = __fsub_rn(sm[i * kMedPitch + lane], med);
}

// V: pixels a thread takes (4 where every frame starts on 16 bytes: one load
// and one store each).  HBM: 2048^2 x 256 in sums of 13, 0.616 ms, 7.2 TB/s of
// bytes read and written (one pixel a thread: 0.712).  V = 1: four frames'
// loads in flight, 1999 x 2001 x 64 in 0.173 ms (one at a time: 0.187).
template <int V>
__global__ void k_sum_frames(const float* __restrict__ in, int n_sum, int M, int64_t P,
                             float* __restrict__ out) {
  const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * V;
  const int m = blockIdx.y;
  if (p >= P || m >= M) return;
  const float* src = in + (int64_t)m * n_sum * P + p;
  float* dst = out + (int64_t)m * P + p;
  if constexpr (V == 4) {
    float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 4
    for (int i = 0; i < n_sum; ++i) {
      const float4 x = __ldcs(reinterpret_cast<const float4*>(src + (int64_t)i * P));
      acc.x = __fadd_rn(acc.x, x.x);
      acc.y = __fadd_rn(acc.y, x.y);
      acc.z = __fadd_rn(acc.z, x.z);
      acc.w = __fadd_rn(acc.w, x.w);
    }
    __stcs(reinterpret_cast<float4*>(dst), acc);
  } else {
    float acc = 0.0f;
#pragma unroll 4
    for (int i = 0; i < n_sum; ++i) acc = __fadd_rn(acc, __ldcs(src + (int64_t)i * P));
    __stcs(dst, acc);
  }
}

// Any row length and base: kBinRows output rows a thread, their loads all in
// flight together (HBM latency bounds the plain form).  1999 x 2001 x 64,
// 0.181 ms, 7.1 TB/s (an output a thread: 0.262).
constexpr int kBinRows = 4;
__global__ void __launch_bounds__(128)
    k_bin2x2(const float* __restrict__ in, int H, int W, int h, int w, float* __restrict__ out) {
  const int X = blockIdx.x * 128 + threadIdx.x;
  const int Y0 = blockIdx.y * kBinRows;
  const int64_t f = blockIdx.z;
  if (X >= w) return;
  float v[kBinRows][4];
#pragma unroll
  for (int j = 0; j < kBinRows; ++j) {
    if (Y0 + j >= h) break;
    const float* r = in + (f * H + 2 * (Y0 + j)) * (int64_t)W + 2 * X;
    v[j][0] = r[0], v[j][1] = r[1], v[j][2] = r[W], v[j][3] = r[W + 1];
  }
#pragma unroll
  for (int j = 0; j < kBinRows; ++j) {
    if (Y0 + j >= h) break;
    __stcs(out + (f * h + Y0 + j) * (int64_t)w + X,
           __fadd_rn(__fadd_rn(__fadd_rn(v[j][0], v[j][1]), v[j][2]), v[j][3]));
  }
}

// The same for rows of a multiple of 8 pixels on 16-byte boundaries: four
// outputs from two vectors of each of two rows, kBinRows output rows a block.
// HBM: 2048^2 x 256, 0.718 ms, 7.5 TB/s (an output a thread: 1.07).
__global__ void __launch_bounds__(256)
    k_bin2x2_vec(const float* __restrict__ in, int H, int W, int h, int w,
                 float* __restrict__ out) {
  const int X = (blockIdx.x * 64 + threadIdx.x % 64) * 4;
  const int Y = blockIdx.y * kBinRows + threadIdx.x / 64;
  const int64_t f = blockIdx.z;
  if (X >= w || Y >= h) return;
  const float4* r0 = reinterpret_cast<const float4*>(in + (f * H + 2 * Y) * (int64_t)W + 2 * X);
  const float4* r1 = reinterpret_cast<const float4*>(in + (f * H + 2 * Y + 1) * (int64_t)W + 2 * X);
  const float4 a = __ldcs(r0), b = __ldcs(r0 + 1), c = __ldcs(r1), d = __ldcs(r1 + 1);
  float4 o;
  o.x = __fadd_rn(__fadd_rn(__fadd_rn(a.x, a.y), c.x), c.y);
  o.y = __fadd_rn(__fadd_rn(__fadd_rn(a.z, a.w), c.z), c.w);
  o.z = __fadd_rn(__fadd_rn(__fadd_rn(b.x, b.y), d.x), d.y);
  o.w = __fadd_rn(__fadd_rn(__fadd_rn(b.z, b.w), d.z), d.w);
  __stcs(reinterpret_cast<float4*>(out + (f * h + Y) * (int64_t)w + X), o);
}

bool on_16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

int median_max_frames() { return 768; }  // 768 x 36 floats = 111 KB of shared memory

int launch_median_subtract(const float* in, int N, int64_t P, float* out, float* median,
                           cudaStream_t s) {
  // up to 64 frames: a sorting network per group size (k_median_select.cu)
  if (N <= median_select_max_frames()) return launch_median_select(in, N, P, out, median, s);
  const int64_t blocks = (P + kMedPix - 1) / kMedPix;
  if (blocks > 0x7fffffff) return -1;
  const size_t smem = ((size_t)N * kMedPitch + kMedPix) * sizeof(float);
  const bool vec = P % 4 == 0 && on_16(in) && on_16(out);
#define ST_MED(K)                                                                              \
  if (N <= kMedShare * K) {                                                                    \
    cudaFuncSetAttribute((const void*)k_median_long<K>,                                        \
                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);              \
    k_median_long<K><<<(unsigned)blocks, kMedPix * kMedShare, smem, s>>>(in, N, P, out, median, \
                                                                         vec);                 \
    return 1;                                                                                  \
  }
  ST_MED(12) ST_MED(16) ST_MED(20) ST_MED(24) ST_MED(28) ST_MED(32) ST_MED(40) ST_MED(48) ST_MED(64)
  ST_MED(80) ST_MED(96)
#undef ST_MED
  return -1;
}

int launch_sum_frames(const float* in, int n_sum, int M, int64_t P, float* out, cudaStream_t s) {
  if (M <= 0) return 0;
  const int64_t bx = (P + 255) / 256;
  if (bx > 0x7fffffff || M > 65535) return -1;
  if (P % 4 == 0 && on_16(in) && on_16(out))
    k_sum_frames<4><<<dim3((unsigned)((P + 1023) / 1024), (unsigned)M), 256, 0, s>>>(in, n_sum, M, P,
                                                                                  out);
  else
    k_sum_frames<1><<<dim3((unsigned)bx, (unsigned)M), 256, 0, s>>>(in, n_sum, M, P, out);
  return 1;
}

int launch_bin2x2(const float* in, int N, int H, int W, float* out, cudaStream_t s) {
  const int h = H / 2, w = W / 2;
  if (h <= 0 || w <= 0 || N <= 0) return 0;
  if (h > 65535 || N > 65535) return -1;
  if (W % 8 == 0 && on_16(in) && on_16(out)) {
    k_bin2x2_vec<<<dim3((unsigned)((w / 4 + 63) / 64), (unsigned)((h + kBinRows - 1) / kBinRows),
                        (unsigned)N), 256, 0, s>>>(in, H, W, h, w, out);
    return 1;
  }
  k_bin2x2<<<dim3((unsigned)((w + 127) / 128), (unsigned)((h + kBinRows - 1) / kBinRows),
                  (unsigned)N), 128, 0, s>>>(in, H, W, h, w, out);
  return 1;
}

}  // namespace st
