// k_median_select.cu — median star removal (Sec. 2.1) for groups of at most
// 64 frames, one kernel per group size.
//
// The per-pixel median over the group's finite samples (NaN marks a masked
// pixel; an even count takes (a + b) * 0.5 of the two middle values; no
// finite sample gives NaN) is subtracted from every frame of the group.
//
// A block of 128 threads takes 128 consecutive pixels: their columns of N
// frames are copied into shared memory asynchronously, so the cube is read
// from global memory once and the subtraction takes its inputs from shared
// memory.  Each thread sorts its column in registers with Batcher's odd-even
// merge network, whose every index is a compile-time constant: comparators
// with positions past N, and those that do not feed the three middle outputs
// k1 - 1, k1, k1 + 1 (k1 = (N - 1) / 2), vanish at compile time (N = 50: 613
// minima and maxima; 783 of the bitonic network).
//
// HBM bounds it: the cube in and out once.  Where frames start on 16 bytes a
// warp moves a frame's 128 pixels with one 16-byte piece a lane, four frames
// at a time, in and out; else each thread moves its own pixel's values.  2048^2
// x 50: 248 us, 6.8 TB/s (4-byte pieces 365; with integer keys and the bitonic
// network 372); 1777^2 x 64, frames off 16 bytes: 329 us (403).
//
// Masked samples do not change those positions: of a pixel's N - n masked
// samples, half (rounded down) become -inf and the rest +inf, so the n finite values sit in the middle of the sorted column and
// their one or two middle values fall on k1 - 1 .. k1 + 1:
//   n, N of equal parity: k1 (N odd) or k1, k1 + 1 (N even);
//   n even, N odd: k1 - 1, k1;   n odd, N even: k1.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <array>
#include <utility>

#include "st_internal.h"

namespace st {

namespace {

constexpr int kSelThreads = 128, kSelWarps = kSelThreads / 32;

// Stage (p, k) of Batcher's odd-even merge network for M values over v[0..N),
// ascending, then the following stages.  (Every comparator puts the smaller
// value first, so values past N, all at the top, would never move.)  The
// minimum and maximum instructions order -0 below +0, as the sorted list does,
// and there is no NaN among the keys.
template <int N, int M, int p, int k>
__device__ __forceinline__ void odd_even_merge(float (&v)[N]) {
#pragma unroll
  for (int i = k % p; i + k < N; ++i) {
    if ((i - k % p) % (2 * k) < k && i / (2 * p) == (i + k) / (2 * p)) {
      const float a = v[i], b = v[i + k];
      v[i] = fminf(a, b);
      v[i + k] = fmaxf(a, b);
    }
  }
  if constexpr (k > 1) {
    odd_even_merge<N, M, p, k / 2>(v);
  } else if constexpr (2 * p < M) {
    odd_even_merge<N, M, 2 * p, 2 * p>(v);
  }
}

constexpr int pow2_at_least(int n) {
  int m = 1;
  while (m < n) m *= 2;
  return m;
}

template <int N>
__global__ void __launch_bounds__(kSelThreads, 4)
    k_median_select(const float* in, int64_t P, float* out, float* __restrict__ median,
                    const bool vec) {
  constexpr int M = pow2_at_least(N < 2 ? 2 : N);
  __shared__ __align__(16) float col[N][kSelThreads];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t p0 = (int64_t)blockIdx.x * kSelThreads, p = p0 + tid;
  const int64_t p4 = p0 + 4 * lane;  // the lane's pixels in a row of 16-byte pieces
  const bool ok = p < P;
  // the columns of the block's pixels (a pixel past the end reads zeros)
  if (vec) {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&col[0][4 * lane]);
    const float* src = p4 < P ? in + p4 : in;
#pragma unroll
    for (int j = 0; j < (N + kSelWarps - 1) / kSelWarps; ++j) {
      const int i = j * kSelWarps + warp;
      if (i < N)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                         dst + (uint32_t)(i * kSelThreads * 4)),
                     "l"(src + (int64_t)i * P), "r"(p4 < P ? 16 : 0)
                     : "memory");
    }
  } else {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&col[0][tid]);
    const float* src = ok ? in + p : in;
#pragma unroll
    for (int i = 0; i < N; ++i)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                       dst + (uint32_t)(i * kSelThreads * 4)),
                   "l"(src + (int64_t)i * P), "r"(ok ? 4 : 0)
                   : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // masked samples take +inf and -inf alternately (the first +inf): sign and
  // number in one word
  float key[N];
  uint32_t masked = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float x = col[i][tid];
    const bool fin = fabsf(x) < INFINITY;
    key[i] = fin ? x : __uint_as_float((masked & 0x80000000u) | 0x7f800000u);
    masked += fin ? 0u : 0x80000001u;
  }
  odd_even_merge<N, M, 1, 1>(key);
  constexpr int k1 = (N - 1) / 2;
  const int n = N - (int)(masked & 0x7fffffffu);
  float med = __int_as_float(0x7fc00000);  // NaN: no finite sample
  if (n > 0) {
    const float lo = key[k1 > 0 ? k1 - 1 : 0], mid = key[k1];
    const float hi = key[k1 + 1 < N ? k1 + 1 : k1];
    if ((n & 1) && (((N ^ n) & 1) == 0 || (N & 1) == 0)) {
      med = mid;                                            // one middle value at k1
    } else if ((N & 1) == 0) {
      med = __fmul_rn(__fadd_rn(mid, hi), 0.5f);            // N, n even
    } else {
      med = __fmul_rn(__fadd_rn(lo, mid), 0.5f);            // N odd, n even
    }
  }
  if (median && ok) median[p] = med;
  if (vec) {
    __shared__ __align__(16) float meds[kSelThreads];
    meds[tid] = med;
    __syncthreads();
    const float4 m = *reinterpret_cast<const float4*>(&meds[4 * lane]);
    if (p4 >= P) return;
#pragma unroll
    for (int j = 0; j < (N + kSelWarps - 1) / kSelWarps; ++j) {
      const int i = j * kSelWarps + warp;
      if (i >= N) break;
      float4 v = *reinterpret_cast<const float4*>(&col[i][4 * lane]);
      v = make_float4(__fsub_rn(v.x, m.x), __fsub_rn(v.y, m.y), __fsub_rn(v.z, m.z),
                      __fsub_rn(v.w, m.w));
      __stcs(reinterpret_cast<float4*>(out + (int64_t)i * P + p4), v);
    }
    return;
  }
  if (!ok) return;
#pragma unroll
  for (int i = 0; i < N; ++i) __stcs(out + (int64_t)i * P + p, __fsub_rn(col[i][tid], med));
}

using SelectFn = void (*)(const float*, int64_t, float*, float*, bool);

template <int... I>
constexpr auto select_table(std::integer_sequence<int, I...>) {
  return std::array<SelectFn, sizeof...(I)>{{k_median_select<I + 1>...}};
}

}  // namespace

int median_select_max_frames() { return 64; }

int launch_median_select(const float* in, int N, int64_t P, float* out, float* median,
                         cudaStream_t s) {
  static const auto table = select_table(std::make_integer_sequence<int, 64>{});
  if (N < 1 || N > 64) return -1;
  const int64_t blocks = (P + kSelThreads - 1) / kSelThreads;
  if (blocks > 0x7fffffff) return -1;
  // frames that all start on 16 bytes are moved 16 bytes at a time
  const bool vec =
      P % 4 == 0 && ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
  table[N - 1]<<<(unsigned)blocks, kSelThreads, 0, s>>>(in, P, out, median, vec);
  return 1;
}

}  // namespace st
