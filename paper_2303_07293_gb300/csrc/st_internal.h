// st_internal.h — internal types of the synthetic-tracking library (device +
// host).  Not part of the C ABI.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/st.h"

namespace st {

// Above-threshold point waiting for the local-maximum test (24 bytes).
struct Pending {
  int32_t x, y, k, field;
  float S;
  int32_t n_cov;
};

// Counters shared by the kernels of one search, in device memory.
struct Counters {
  unsigned long long n_pending;   // points written (or attempted) to the pending list
  unsigned long long n_cand;      // candidates after the local-maximum test
  unsigned int error;             // bit flags, ERR_*
  unsigned int runs;              // 1: the run kernel did the stacking
  unsigned long long work_next;   // persistent-kernel work counter
  unsigned long long n_sure;      // pending points that reach the threshold for certain
                                  // (bilinear window kernel; a lower bound)
};

// ERR_MARGIN: the bilinear window kernel left the work (its margin is too wide)
enum : unsigned { ERR_PENDING_OVERFLOW = 1u, ERR_CAND_OVERFLOW = 2u, ERR_TIMEOUT = 4u,
                  ERR_MARGIN = 8u };

// Everything a kernel needs to read one field.  Plain data, passed by value.
struct FieldDev {
  const void* cube;      // storage cube [N][H][pitch] of `storage` type
  int32_t pitch;         // elements from one row to the next (>= W)
  int32_t storage;       // st_dtype
  int32_t W, H, N;
  int32_t nvx, nvy;
  int32_t nmin;
  int32_t field;
  const int32_t* sx;     // [N][nvx] integer shift (nearest: rounded; bilinear: floor)
  const int32_t* sy;     // [N][nvy]
  const float* fx;       // [N][nvx] bilinear fraction
  const float* fy;       // [N][nvy]
  const float* thr;      // [N+1] thr[n] = (float)(tau*sqrt(n))
  const float* rsq;      // [N+1] (float)(1/sqrt(n))
};

// Key of a candidate: (field, k, y, x) packed into 64 bits, increasing in
// the output order.
__host__ __device__ inline uint64_t cand_key(int field, int k, int y, int x) {
  return ((uint64_t)(uint32_t)field << 56) | ((uint64_t)(uint32_t)k << 30) |
         ((uint64_t)(uint32_t)y << 15) | (uint64_t)(uint32_t)x;
}

// Sets the message returned by st_last_error() on this thread.
void set_last_error(const char* msg);

// ---- kernel launchers (each returns the number of kernels it launched) ----

int launch_shift_tables(const double* d_t, int N, double t_ref, double vx0, double dvx,
                        int nvx, double vy0, double dvy, int nvy, int mode, int32_t* sx,
                        int32_t* sy, float* fx, float* fy, cudaStream_t s);

// Sky statistics (FP64, deterministic) and normalisation/conversion.
//   partial: workspace of sky_partial_doubles(N) doubles.
size_t sky_partial_doubles(int N);
//   cube: rows of W values, pitch values apart.  absmax, nan: as launch_absmax,
//   of the stored values, if absmax is not NULL.
int launch_normalize(const float* raw, int N, int W, int H, int normalize, float cr_clip,
                     int storage, void* cube, int pitch, double* mu, double* sigma,
                     double* partial, unsigned* absmax, bool nan, cudaStream_t s);
// Largest |x| of n values as FP32 bits, into *absmax (which the caller zeroes).
// nan: a NaN counts as larger than any (else not at all).
int launch_absmax(const float* x, int64_t n, bool nan, unsigned* absmax, cudaStream_t s);

// Bound of the difference between the FP32 sum of N values of at most
// `largest` in frame order and the run kernel's: an addition errs by at most
// u = 2^-24 times its result.  Frame order: u largest (1 + 2 + .. + N).  Runs:
// the running sums err as much (an output takes each frame from one of them,
// and what two terms share of an earlier error cancels), and their terms, up
// to 11 of at most N largest each, are added up in steps of at most 3 N
// largest.  thr: the largest threshold, whose difference with the margin is
// rounded too.
__host__ __device__ inline float run_margin(float largest, int N, float thr) {
  const float n = (float)N;
  return 1.02f * 0x1p-24f * (largest * n * (n + 40.0f) + 4.0f * thr);
}
// Bound of the difference between the bilinear window kernel's sum (the
// sample as two horizontal interpolations, weighted 1 - fy and fy) and the
// direct gather's (four taps, each weighted by a rounded product): with taps
// of at most `largest`, the weights and interpolations of a frame err by at
// most 2 u and 3.5 u times that, and the two and four multiply-adds by u times
// the sum so far, i largest after i frames: u largest N (3 N + 8.5).  (The
// last term: roundings below the normal range.)
__host__ __device__ inline float bilinear_margin(float largest, int N, float thr) {
  const float n = (float)N;
  return 1.02f * 0x1p-24f * (largest * n * (3.0f * n + 9.0f) + 4.0f * thr) + n * 0x1p-146f;
}
// Whether the margin is at most `share` of the noise of the least covered
// points over the threshold: it then adds about share times as many points as
// lie above the threshold for small shares, e^share times for larger ones.
// (False for a margin that an infinite or NaN value made.)
__host__ __device__ inline bool margin_ok(float margin, int nmin, float thr_nmin, float share) {
  const float root = sqrtf((float)(nmin > 1 ? nmin : 1));
  const float tau = thr_nmin / root;
  return margin * (tau > 1.0f ? tau : 1.0f) <= share * root;
}
// Shares up to which the kernels that need a margin run: the run kernel's
// stand-in costs twice its time, the bilinear window kernel's (the direct
// gather) ten times, and twenty times the points above a threshold of 5 are
// still few.
constexpr float kRunShare = 0.1f, kBilinearShare = 3.0f;
__host__ __device__ inline float margin_of(int mode, float largest, int N, float thr) {
  return mode == ST_BILINEAR ? bilinear_margin(largest, N, thr) : run_margin(largest, N, thr);
}
__host__ __device__ inline bool margin_ok(int mode, float margin, int nmin, float thr_nmin) {
  return margin_ok(margin, nmin, thr_nmin, mode == ST_BILINEAR ? kBilinearShare : kRunShare);
}
// The margins of the n fields, and whether all are small enough, from the
// largest values (bilinear sampling: else ERR_MARGIN, too).
int launch_margins(const FieldDev* fds, int n, int mode, const unsigned* absmax, float* margin,
                   int* use, Counters* ctr, cudaStream_t s);

// Generic stack kernels over velocity indices [k0, k0+nk): threshold ->
// pending list; optional dump of S and n_cov for the listed velocities.
int launch_stack_generic(const FieldDev& fd, int mode, int k0, int nk, const int32_t* dump_k,
                         float* dump_S, int32_t* dump_C, Pending* pend, int64_t pend_cap,
                         Counters* ctr, cudaStream_t s);

// Register-window stack kernel (nearest or bilinear sampling); returns -1 when
// the field's geometry does not fit the kernel (caller falls back).
struct FastPlan;
int fast_plan_size_bytes();
int fast_num_variants();
int fast_num_variants_for(const FastPlan* fp, int storage);
int fast_get_variant(const FastPlan* fp);
int fast_autotune(const FieldDev& fd, FastPlan* fp, int64_t items, Pending* pend,
                  int64_t pend_cap, Counters* ctr, cudaStream_t s);
// A hash (FNV-1a) of the names of the variants for a storage type and sampling.
uint32_t fast_list_mark(int storage, int mode);
const char* fast_variant_name(const FastPlan* fp, int storage);
void fast_set_variant(FastPlan* fp, int v);
// Whether the field can use the fast kernel at all (row pitch a multiple of
// 16 bytes for the tensor map).
bool fast_eligible(const FieldDev& fd, int mode);
// Builds the per-frame tile tables for the current shift tables; *fits tells
// whether the motion spans fit the kernel.  Synchronises the stream.
int fast_prepare(const FieldDev& fd, FastPlan* fp, cudaStream_t s, bool* fits);
bool fast_plan_build(const FieldDev& fd, int mode, FastPlan** out);
void fast_plan_free(FastPlan* fp);
int launch_stack_fast(const FieldDev& fd, const FastPlan* fp, int k0, int nk,
                      const int32_t* dump_k, float* dump_S, int32_t* dump_C, Pending* pend,
                      int64_t pend_cap, Counters* ctr, cudaStream_t s);
// One persistent launch over n prepared, fitting fields (same storage and
// sampling; the variant of fps[0]), items taken longest field first.
// Encodes and uploads the tensor maps a launch over these fields needs (so the
// launch itself copies nothing); *restaged tells whether any map changed.
// plain: for a launch without a RunCtl.
bool fast_stage(const FieldDev* fds, FastPlan* const* fps, int n, bool plain, cudaStream_t s,
                bool* restaged);
// Without `rc` the default variant is the frame-order kernel of 8-row tiles.
// With it the default follows the field's sizes, and the run kernel may do the
// work (k_stack_runs.cu): it keeps points
// down to a margin below the threshold, given per field (margin, or d_margin in
// device memory); with d_use it runs only if *d_use is not 0, else the
// variant that stands in for it does (both are launched).  Bilinear sampling:
// the window kernel keeps such a margin, and does nothing where *d_use is 0.
struct RunCtl {
  bool runs;              // the run kernel may do the work
  const float* margin;    // host, [n] in the order of fds (NULL: 0)
  const float* d_margin;  // device, by field of the plan
  const int* d_use;
};
bool fast_runs_chosen(const FieldDev* fds, FastPlan* const* fps, int n);
// Whether a launch without a RunCtl runs another variant than one with it did
// (runs: the run kernel).
bool fast_plain_differs(const FieldDev* fds, FastPlan* const* fps, int n, bool runs);
// Notes which of the two a launch with d_use ran (for the variant's name).
void fast_note_ran(const FieldDev* fds, FastPlan* const* fps, int n, bool runs);
int launch_stack_fast_multi(const FieldDev* fds, FastPlan* const* fps, int n, float* dump_S,
                            int32_t* dump_C, Pending* pend, int64_t pend_cap, Counters* ctr,
                            const RunCtl* rc, cudaStream_t s);

// Local-maximum test of the pending points -> candidate list (unsorted) and keys.
int launch_resolve(const FieldDev* fds_dev, int n_fields, int mode, const Pending* pend,
                   const Counters* ctr, int64_t pend_cap, st_candidate* cand,
                   uint64_t* keys, uint32_t* idx, int64_t cand_cap, Counters* ctr_out,
                   cudaStream_t s);

// Sorts keys/idx (n_pow2 entries, padded with ~0) and gathers the first
// `capacity` records into out.
int launch_sort_gather(uint64_t* keys, uint32_t* idx, int64_t n_pow2, const Counters* ctr,
                       const st_candidate* cand, st_candidate* out, int64_t capacity,
                       cudaStream_t s);
// The same for at most sort_short_max() candidates, whose number the kernel
// reads itself (others, and lists with an error, are left alone).
int64_t sort_short_max();
int launch_sort_short(const uint64_t* keys, const Counters* ctr, const st_candidate* cand,
                      st_candidate* out, int64_t capacity, cudaStream_t s);
// The sort alone (idx carried along).
int launch_sort(uint64_t* keys, uint32_t* idx, int64_t n_pow2, cudaStream_t s);
int launch_pad_keys(uint64_t* keys, uint32_t* idx, int64_t n_pow2, const Counters* ctr,
                    cudaStream_t s);

// Refinement: optimise == false evaluates J, SNR and (optionally) dJ/dtheta at
// the given theta; optimise == true runs `steps` Adam steps from each
// candidate's grid velocity and pixel, with F at its optimum, and writes the
// refined records.
// Refinement (forward + adjoint, optional Adam steps) of n candidates; h_fds
// are the host copies of the n_fields device descriptors fds (their cubes are
// mapped for TMA into d_maps, n_fields entries).  Returns -1 if a field cannot
// be mapped or has more than refine_max_frames() frames.  keys, idx: sort_cap
// entries of scratch for the order of the candidates.
int refine_max_frames();
int launch_refine(const FieldDev* h_fds, int n_fields, const FieldDev* fds, CUtensorMap* d_maps,
                  const double* const* times, const double* t_ref, const double* grid,
                  int storage, bool optimise, const float* theta, const int32_t* centre,
                  const int32_t* field, const st_candidate* cand, int64_t n, int steps,
                  int optimizer, float fwhm, float lr_pos, float lr_vel, float* J, float* snr,
                  float* grad, st_refined* out, int* err, uint64_t* keys, uint32_t* idx,
                  int64_t sort_cap, cudaStream_t s);

// Tracks: links the sorted candidates [n] into components (workspace of
// link_workspace_bytes(n, velocities) bytes; velocities: of all fields, their
// descriptors in fds); writes up to cap tracks, *n_tracks = all (h_count:
// pinned scratch).  Synchronises s.  Returns launches or -1.
int64_t link_workspace_bytes(int64_t n, int64_t velocities);
int launch_link_tracks(const st_candidate* c, int64_t n, const FieldDev* fds, int n_fields,
                       int64_t velocities, const double* grid, int r_xy, int r_v, void* ws,
                       st_track* out, int64_t cap, int* h_count, int64_t* n_tracks,
                       cudaStream_t s);

// Front end (Sec. 2.1): median star removal over a group of N frames (N <=
// median_max_frames()), sums of every n_sum frames into M outputs, 2 x 2
// binning.  Each returns the number of launches or -1 if the sizes exceed
// the launch limits.
int median_max_frames();
int median_select_max_frames();
int launch_median_select(const float* in, int N, int64_t P, float* out, float* median,
                         cudaStream_t s);
int launch_median_subtract(const float* in, int N, int64_t P, float* out, float* median,
                           cudaStream_t s);
int launch_sum_frames(const float* in, int n_sum, int M, int64_t P, float* out, cudaStream_t s);
int launch_bin2x2(const float* in, int N, int H, int W, float* out, cudaStream_t s);

// Tiled TMA map of a field's cube [N][H][W] (storage type) with a box of
// box_w x box_h x 1 elements, zero fill outside.  False if it cannot be built.
bool encode_tile_map(CUtensorMap* map, const FieldDev& fd, int box_w, int box_h);

}  // namespace st
