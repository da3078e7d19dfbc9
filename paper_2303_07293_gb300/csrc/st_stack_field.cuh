// st_stack_field.cuh — what the register-window stack kernels share: a
// field's descriptor, staircase patterns, coverage counts, work items.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "st_internal.h"

namespace st {

// One field of a launch: geometry, per-frame tile tables and thresholds.
struct FastField {
  int W, H, N, nvx, nvy, nA, nB, nmin, field;
  const int4* xt;   // [N][nA]: box x offset, packed 4-bit column offsets, min shift, max shift
  const int4* yt;   // [N][nB]: min shift, max shift, pattern id, 0
  const unsigned char* pat;  // [N][nB] staircase pattern ids
  const int32_t* sx;
  const int32_t* sy;
  const float* fx;   // bilinear: FP32 fractions [N][nvx], [N][nvy]
  const float* fy;
  const float4* fxt;  // bilinear: [N][nA][2] x-fractions of a velocity tile's 8 x-velocities
  const float4* fyt;  // bilinear: [N][nB] y-fractions of its 4 y-velocities
  const float* thr;
  // coverage prefix tables: for velocity a, covx[a * cov_len + s - cov_xmin[a]]
  // = number of frames with sx(i, a) <= s (likewise y)
  const int* covx;
  const int* covy;
  const int* cov_xmin;
  const int* cov_xmax;
  const int* cov_ymin;
  const int* cov_ymax;
  int cov_len;
  // tables of the run kernel (k_stack_runs.cu)
  int nG, nT;           // groups of 4 x-velocities, tiles of at most 4 groups
  const uint32_t* xg;   // [N][nG] shift and steps of a group
  const int2* ord;      // [nB][N] frames by pattern
};

constexpr int kMaxFields = 256;
constexpr int kMB = 4;           // y-velocities per block (staircase group)
constexpr int kTX = 32;          // pixel tile width
constexpr int kPatterns = 15;
constexpr int kSuper = 4;        // pixel tiles per super-tile side (L2 locality)
constexpr uint64_t kStackWaitNs = 2000000000ull;  // wait limit: 2 s of wall-clock time
constexpr unsigned kProducerSleepNs = 128;  // producer back-off between polls

// Storage types: TMA element type, conversion.
template <typename T>
struct StoreType;
template <>
struct StoreType<float> {
  static constexpr CUtensorMapDataType kTma = CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  __device__ static float f(float v) { return v; }
};
template <>
struct StoreType<__half> {
  static constexpr CUtensorMapDataType kTma = CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  __device__ static float f(__half v) { return __half2float(v); }
};
template <>
struct StoreType<__nv_bfloat16> {
  static constexpr CUtensorMapDataType kTma = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  __device__ static float f(__nv_bfloat16 v) { return __bfloat162float(v); }
};

// Pattern id -> row offsets of the 4 y-velocities (min offset 0).
// ids 0..7: non-decreasing, steps (id&1, id>>1&1, id>>2&1);
// ids 8..14: non-increasing, steps of t = id - 7 read from the other end.
__host__ __device__ constexpr int pat_off(int id, int j) {
  if (id < 8) {
    int s1 = id & 1, s2 = (id >> 1) & 1, s3 = (id >> 2) & 1;
    return j == 0 ? 0 : j == 1 ? s1 : j == 2 ? s1 + s2 : s1 + s2 + s3;
  }
  int t = id - 7;
  int t1 = t & 1, t2 = (t >> 1) & 1, t3 = (t >> 2) & 1;
  return j == 0 ? t1 + t2 + t3 : j == 1 ? t2 + t3 : j == 2 ? t3 : 0;
}

// Number of frames whose shift s satisfies lo <= s <= hi, from a prefix table.
__device__ __forceinline__ int count_shifts(const int* pre, int smin, int smax, int N, int lo,
                                            int hi) {
  auto upto = [&](int s) { return s < smin ? 0 : s >= smax ? N : __ldg(pre + (s - smin)); };
  return hi < lo ? 0 : upto(hi) - upto(lo - 1);
}

// Acquire a tensor map written to global memory before the launch for the
// TMA unit (tensor-map proxy).
__device__ __forceinline__ void tmap_acquire(const CUtensorMap* m) {
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"((uint64_t)m)
               : "memory");
}

// Run tables and kernel (k_stack_runs.cu) of a field; see there.
struct RunPlan {
  uint32_t* xg = nullptr;
  int2* ord = nullptr;
  int* bad = nullptr;    // device: [0] a group's steps exceed 1, [1] largest box offset
  int* h_bad = nullptr;  // pinned copy
  CUtensorMap tmap;
  CUtensorMap* d_map = nullptr;
  const void* encoded_for = nullptr;
  int nG = 0, nT = 0;
  bool fits = false;
};
RunPlan* run_plan_build(const FieldDev& fd, int nB);
void run_plan_free(RunPlan* rp);
// Queues the tables' kernels and the copy of their maxima (no synchronisation);
// run_finish reads the maxima once the stream has been synchronised.
void run_prepare(const FieldDev& fd, const unsigned char* pat, const int4* yt, int nB,
                 RunPlan* rp, cudaStream_t s);
void run_finish(const FieldDev& fd, RunPlan* rp);
int run_box_w(int storage);
int run_box_h();

struct RunArgs {
  const FastField* ff[kMaxFields];      // the launch's fields, longest first (device)
  const CUtensorMap* maps[kMaxFields];  // their cubes' tiled maps (global memory)
  float margin[kMaxFields];             // how far below the threshold a sum is still kept
  const float* d_margin;                // by field of the plan, in device memory (or NULL)
  const int* d_use;                     // 0: leave the work to the next launch (or NULL)
  int n_fields;
  int64_t n_items;
  unsigned long long* work;             // next item to take (zero at launch)
  Pending* pend;
  int64_t cap;
  Counters* ctr;
};
int64_t run_items(const FastField& ff);
int launch_runs(const RunArgs& a, int storage, int sms, cudaStream_t s);

}  // namespace st
