// k_finish.cu — local-maximum test of the above-threshold points, candidate
// records, and the deterministic (field, k, y, x) ordering.
//
// Sec. 2.1 returns detections with pixel coordinates, motion and S/N.  The
// local-maximum rule (8 neighbours inside the frame with n_cov >= n_min;
// strictly greater than earlier neighbours in raster order, greater or equal
// to later ones) needs neighbour stack values that the stack kernels never
// store: they are recomputed here by the same ordered FP32 sum, so they are
// bit-identical to the values the stack kernel formed.
#include <algorithm>

#include "st_internal.h"
#include "st_sample.cuh"

namespace st {

namespace {

// Sums and coverage of the three pixels x - 1, x, x + 1 of a row, each in
// frame order.  (y may lie outside the frame: every sample that does reads 0.)
template <typename T, int MODE>
__device__ void stack_three(const FieldDev& fd, int x, int y, int a, int b, float (&S)[3],
                            int (&C)[3]) {
  const T* cube = (const T*)fd.cube;
  const int64_t P = (int64_t)fd.pitch * fd.H;
  const int W = fd.W, H = fd.H, pitch = fd.pitch, N = fd.N;
  const int32_t* sx = fd.sx + a;
  const int32_t* sy = fd.sy + b;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    S[q] = 0.0f;
    C[q] = 0;
  }
#pragma unroll 4
  for (int i = 0; i < N; ++i) {
    const T* fr = cube + (int64_t)i * P;
    const int u = x + __ldg(sx + (int64_t)i * fd.nvx);
    const int w = y + __ldg(sy + (int64_t)i * fd.nvy);
    if (MODE == ST_NEAREST) {
      const bool row = w >= 0 && w < H;
      const T* r = fr + (int64_t)(row ? w : 0) * pitch;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int uq = u + q - 1;
        const bool in = row && uq >= 0 && uq < W;
        S[q] = __fadd_rn(S[q], in ? load_px<T>(r + uq) : 0.0f);
        C[q] += in;
      }
    } else {
      const float fx = __ldg(fd.fx + (int64_t)i * fd.nvx + a);
      const float fy = __ldg(fd.fy + (int64_t)i * fd.nvy + b);
      const BW wt = bilinear_weights(fx, fy);
      float t0[4], t1[4];  // taps of the row and of the one below
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        t0[q] = tap<T>(fr, pitch, W, H, u + q - 1, w);
        t1[q] = tap<T>(fr, pitch, W, H, u + q - 1, w + 1);
      }
      const bool row = bilinear_inside(w, fy, H);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        S[q] = bilinear_acc(S[q], wt, t0[q], t0[q + 1], t1[q], t1[q + 1]);
        C[q] += row && bilinear_inside(u + q - 1, fx, W);
      }
    }
  }
}

template <int MODE>
__device__ void stack_any(const FieldDev& fd, int x, int y, int a, int b, float (&S)[3],
                          int (&C)[3]) {
  if (fd.storage == ST_F32) stack_three<float, MODE>(fd, x, y, a, b, S, C);
  else if (fd.storage == ST_F16) stack_three<__half, MODE>(fd, x, y, a, b, S, C);
  else stack_three<__nv_bfloat16, MODE>(fd, x, y, a, b, S, C);
}

// 4 lanes per pending point, of which three sum a row of three pixels each
// (the row above, its own, the row below): the two shifts of a frame, which
// are as many loads as a pixel's, serve three pixels, and the point's own sum
// comes with its row.  2048^2 x 256, 101^2 velocities, 1 M points:
// 8.2 ms (a neighbour a lane, the point itself after them: 22.1).
// The grid is sized for the chip, not for the list's capacity (131 072 blocks
// that found nothing to do took 76 us of a small search).
constexpr int kResolveThreads = 256;
template <int MODE>
__global__ void __launch_bounds__(kResolveThreads)
    k_resolve(const FieldDev* __restrict__ fds, const Pending* __restrict__ pend,
              const Counters* __restrict__ ctr_in, int64_t pend_cap,
              st_candidate* __restrict__ cand, uint64_t* __restrict__ keys,
              uint32_t* __restrict__ idx, int64_t cand_cap, Counters* __restrict__ ctr) {
  const int64_t n = (int64_t)min((unsigned long long)pend_cap, ctr_in->n_pending);
  const int lane = threadIdx.x & 31, part = threadIdx.x & 3;
  constexpr int kPoints = kResolveThreads / 4;
  for (int64_t p0 = (int64_t)blockIdx.x * kPoints; p0 < n; p0 += (int64_t)gridDim.x * kPoints) {
    const int64_t p = p0 + (threadIdx.x >> 2);
    const bool have = p < n;
    Pending r{};
    float S[3] = {0.0f, 0.0f, 0.0f};
    int C[3] = {0, 0, 0};
    int nmin = 0, W = 0, H = 0;
    if (have) {
      r = pend[p];
      const FieldDev& fd = fds[r.field];
      nmin = fd.nmin;
      W = fd.W;
      H = fd.H;
      const int y = r.y + part - 1;
      if (part < 3 && y >= 0 && y < H)
        stack_any<MODE>(fd, r.x, y, r.k % fd.nvx, r.k / fd.nvx, S, C);
    }
    // the point's own sum and coverage (recorded, or formed here)
    float Sc = __shfl_sync(0xffffffffu, S[1], (lane & ~3) + 1);
    int Cc = __shfl_sync(0xffffffffu, C[1], (lane & ~3) + 1);
    if (r.n_cov >= 0) {
      Sc = r.S;
      Cc = r.n_cov;
    }
    const bool center_ok = have && Cc >= nmin && Sc >= __ldg(fds[r.field].thr + Cc);
    // a neighbour inside the frame and covered blocks the point: earlier in
    // raster order unless the point is greater, later unless it is at least equal
    bool blocks = false;
    const int y = r.y + part - 1;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int x = r.x + q - 1;
      const bool other = part < 3 && !(part == 1 && q == 1);
      const bool in = x >= 0 && x < W && y >= 0 && y < H && C[q] >= nmin;
      const bool earlier = part == 0 || (part == 1 && q == 0);
      blocks |= have && other && in && (earlier ? !(Sc > S[q]) : !(Sc >= S[q]));
    }
    const unsigned bal = __ballot_sync(0xffffffffu, blocks);
    const bool is_cand = center_ok && part == 0 && ((bal >> (lane & ~3)) & 15u) == 0u;
    const unsigned m = __ballot_sync(0xffffffffu, is_cand);
    if (m == 0u) continue;
    const int leader = __ffs(m) - 1;
    unsigned long long base = 0;
    if (lane == leader) base = atomicAdd(&ctr->n_cand, (unsigned long long)__popc(m));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (is_cand) {
      const unsigned long long pos = base + __popc(m & ((1u << lane) - 1u));
      if (pos < (unsigned long long)cand_cap) {
        const FieldDev& fd = fds[r.field];
        st_candidate c;
        c.x = r.x;
        c.y = r.y;
        c.k = r.k;
        c.field = r.field;
        c.stack = Sc;
        c.snr = __fmul_rn(Sc, __ldg(fd.rsq + Cc));
        c.n_cov = Cc;
        cand[pos] = c;
        keys[pos] = cand_key(r.field, r.k, r.y, r.x);
        idx[pos] = (uint32_t)pos;
      } else {
        atomicOr(&ctr->error, ERR_CAND_OVERFLOW);
      }
    }
  }
}

__global__ void k_pad_keys(uint64_t* keys, uint32_t* idx, int64_t n_pow2,
                           const Counters* __restrict__ ctr) {
  int64_t n = (int64_t)ctr->n_cand;
  int64_t i = n + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n_pow2) {
    keys[i] = ~0ull;
    idx[i] = 0xffffffffu;
  }
}

__device__ __forceinline__ void cswap(uint64_t* keys, uint32_t* idx, int64_t i, int64_t l,
                                      bool asc) {
  uint64_t a = keys[i], b = keys[l];
  if ((a > b) == asc) {
    keys[i] = b;
    keys[l] = a;
    uint32_t t = idx[i];
    idx[i] = idx[l];
    idx[l] = t;
  }
}

__global__ void k_bitonic_global(uint64_t* keys, uint32_t* idx, int64_t n, int64_t j, int64_t k) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int64_t l = i ^ j;
  if (l > i) cswap(keys, idx, i, l, (i & k) == 0);
}

constexpr int kLocal = 2048;  // elements per shared-memory tile

// All steps j < kLocal of stage k (k may be <= kLocal: then all stages up to k).
__global__ void __launch_bounds__(kLocal / 2)
    k_bitonic_local(uint64_t* keys, uint32_t* idx, int64_t n, int64_t k_from, int64_t k_to,
                    int64_t j_from) {
  __shared__ uint64_t sk[kLocal];
  __shared__ uint32_t si[kLocal];
  int64_t base = (int64_t)blockIdx.x * kLocal;
  for (int t = threadIdx.x; t < kLocal; t += blockDim.x) {
    sk[t] = base + t < n ? keys[base + t] : ~0ull;
    si[t] = base + t < n ? idx[base + t] : 0xffffffffu;
  }
  __syncthreads();
  for (int64_t k = k_from; k <= k_to; k <<= 1) {
    for (int64_t j = (k == k_from ? j_from : k >> 1); j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < kLocal; t += blockDim.x) {
        int l = t ^ (int)j;
        if (l > t) {
          bool asc = ((base + t) & k) == 0;
          uint64_t a = sk[t], b = sk[l];
          if ((a > b) == asc) {
            sk[t] = b;
            sk[l] = a;
            uint32_t q = si[t];
            si[t] = si[l];
            si[l] = q;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int t = threadIdx.x; t < kLocal; t += blockDim.x)
    if (base + t < n) {
      keys[base + t] = sk[t];
      idx[base + t] = si[t];
    }
}

// The sort and gather of a short list (at most kLocal candidates; a longer one
// is left alone) in one block, the padding in shared memory only.
__global__ void __launch_bounds__(kLocal / 2)
    k_sort_short(const uint64_t* __restrict__ keys, const Counters* __restrict__ ctr,
                 const st_candidate* __restrict__ cand, st_candidate* __restrict__ out,
                 int64_t capacity) {
  __shared__ uint64_t sk[kLocal];
  __shared__ uint16_t si[kLocal];
  if (ctr->n_cand == 0 || ctr->n_cand > kLocal || ctr->error != 0u) return;
  const int n = (int)ctr->n_cand;
  int m = 2;
  while (m < n) m <<= 1;
  for (int t = threadIdx.x; t < m; t += blockDim.x) {
    sk[t] = t < n ? keys[t] : ~0ull;
    si[t] = (uint16_t)t;
  }
  __syncthreads();
  for (int k = 2; k <= m; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < m; t += blockDim.x) {
        const int l = t ^ j;
        if (l > t) {
          const uint64_t a = sk[t], b = sk[l];
          if ((a > b) == ((t & k) == 0)) {
            sk[t] = b;
            sk[l] = a;
            const uint16_t q = si[t];
            si[t] = si[l];
            si[l] = q;
          }
        }
      }
      __syncthreads();
    }
  const int g = (int)min((int64_t)n, capacity);
  for (int t = threadIdx.x; t < g; t += blockDim.x) out[t] = cand[si[t]];
}

__global__ void k_gather(const uint32_t* __restrict__ idx, const Counters* __restrict__ ctr,
                         const st_candidate* __restrict__ cand, st_candidate* __restrict__ out,
                         int64_t capacity) {
  int64_t n = min((int64_t)ctr->n_cand, capacity);
  int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n) out[r] = cand[idx[r]];
}

}  // namespace

int launch_resolve(const FieldDev* fds_dev, int n_fields, int mode, const Pending* pend,
                   const Counters* ctr, int64_t pend_cap, st_candidate* cand, uint64_t* keys,
                   uint32_t* idx, int64_t cand_cap, Counters* ctr_out, cudaStream_t s) {
  (void)n_fields;
  const int64_t blocks = std::min((int64_t)8 * 152, (pend_cap + kResolveThreads / 4 - 1) /
                                                        (kResolveThreads / 4));
  if (mode == ST_NEAREST)
    k_resolve<ST_NEAREST><<<(unsigned)blocks, kResolveThreads, 0, s>>>(
        fds_dev, pend, ctr, pend_cap, cand, keys, idx, cand_cap, ctr_out);
  else
    k_resolve<ST_BILINEAR><<<(unsigned)blocks, kResolveThreads, 0, s>>>(
        fds_dev, pend, ctr, pend_cap, cand, keys, idx, cand_cap, ctr_out);
  return 1;
}

int launch_pad_keys(uint64_t* keys, uint32_t* idx, int64_t n_pow2, const Counters* ctr,
                    cudaStream_t s) {
  k_pad_keys<<<(unsigned)((n_pow2 + 255) / 256), 256, 0, s>>>(keys, idx, n_pow2, ctr);
  return 1;
}

int64_t sort_short_max() { return kLocal; }
int launch_sort_short(const uint64_t* keys, const Counters* ctr, const st_candidate* cand,
                      st_candidate* out, int64_t capacity, cudaStream_t s) {
  k_sort_short<<<1, kLocal / 2, 0, s>>>(keys, ctr, cand, out, capacity);
  return 1;
}

int launch_sort(uint64_t* keys, uint32_t* idx, int64_t n, cudaStream_t s) {
  // n is a power of two >= the live count; padding keys sort last.
  int launches = 0;
  if (n >= 2) {
    int64_t tiles = (n + kLocal - 1) / kLocal;
    int64_t kmax_local = n < kLocal ? n : kLocal;
    k_bitonic_local<<<(unsigned)tiles, kLocal / 2, 0, s>>>(keys, idx, n, 2, kmax_local, 1);
    ++launches;
    for (int64_t k = 2 * kLocal; k <= n; k <<= 1) {
      for (int64_t j = k >> 1; j >= kLocal; j >>= 1) {
        k_bitonic_global<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(keys, idx, n, j, k);
        ++launches;
      }
      k_bitonic_local<<<(unsigned)tiles, kLocal / 2, 0, s>>>(keys, idx, n, k, k, kLocal / 2);
      ++launches;
    }
  }
  return launches;
}

int launch_sort_gather(uint64_t* keys, uint32_t* idx, int64_t n, const Counters* ctr,
                       const st_candidate* cand, st_candidate* out, int64_t capacity,
                       cudaStream_t s) {
  int launches = launch_sort(keys, idx, n, s);
  if (capacity > 0) {
    int64_t g = (n < capacity ? n : capacity);
    if (g < 1) g = 1;
    k_gather<<<(unsigned)((g + 255) / 256), 256, 0, s>>>(idx, ctr, cand, out, capacity);
    ++launches;
  }
  return launches;
}

}  // namespace st
