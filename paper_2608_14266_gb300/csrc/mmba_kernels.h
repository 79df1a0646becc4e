// Host-side declarations of the library's kernel launchers (internal).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "mmba_internal.cuh"

namespace mmba {

constexpr int kVoxelThreads = 128;
constexpr int kScanThreads = 128;      // FP64 scan pass: threads per scan
constexpr int kScanMixedThreads = 32;  // mixed scan pass: one warp per scan (long pipelined loops, no block barrier)
constexpr int kDecideThreads = 256;  // one block; FP64 sums are 1/64 rate, so few warps and few adds
constexpr int kSolveThreads = 64;  // small blocks spread the scans over every SM

__host__ __device__ inline int64_t voxel_pass_blocks(int64_t n_voxels) { return (n_voxels + kVoxelThreads - 1) / kVoxelThreads; }
// FP64 voxel pass: the threads that share a voxel's observations, whose partial
// sums are added up in a fixed order.  More of them (fewer voxels per block of
// kVoxelThreads) spread a small problem over more of the FP64 pipes; the price
// is the eigenproblem's warp, which then holds fewer voxels.  Measured (us per
// pass, 8-40 observations per voxel, event-timed; 16 / 8 / 4 threads, and one
// before):
//     200 voxels   32 /  37 /  47   (118)      9,728   85 /  66 /  64   (121)
//   2,432          37 /  38 /  49   (121)     19,456  149 / 116 /  97   (129)
//   4,864          47 /  43 /  49   (120)     50,000  344 / 245 / 206   (258)
// One thread where voxels are many and short, so that most of four would be idle
// (us, four and one): 300,000 voxels of 1-2 observations 328 / 248, of 3-4 402 /
// 315, 200,000 of 5-8 328 / 293, 50,000 of 3-4 89 / 70, of 6-8 105 / 94; 100,000 of
// 10-12 225 / 221.
constexpr int64_t kShortVoxels = 50000, kShortObs = 10;
__host__ __device__ inline int voxel_pass_f64_rows(int64_t n_voxels, int64_t n_obs) {
  if (n_voxels <= 6144) return n_voxels <= 2432 ? 16 : 8;
  return n_voxels >= kShortVoxels && n_obs <= kShortObs * n_voxels ? 1 : 4;
}
// partial sums of the cost: one for every so many voxels
__host__ __device__ inline int voxel_pass_f64_width(int rows) { return rows == 1 ? 32 : kVoxelThreads / rows; }
__host__ __device__ inline int64_t voxel_pass_f64_parts(int64_t n_voxels, int64_t n_obs) {
  const int v = voxel_pass_f64_width(voxel_pass_f64_rows(n_voxels, n_obs));
  return (n_voxels + v - 1) / v;
}
// Blocks of a problem's own launch: a part to a block, or, with one thread to a
// voxel, kVoxelThreads voxels.
inline int64_t voxel_pass_f64_blocks(int64_t n_voxels, int64_t n_obs) {
  return voxel_pass_f64_rows(n_voxels, n_obs) == 1 ? voxel_pass_blocks(n_voxels)
                                                   : voxel_pass_f64_parts(n_voxels, n_obs);
}
// Whether a batch of n_voxels in all (its groups run beside each other) gives a
// voxel to one thread, which then forms the partial sums of 4, 8 or 16 in turn:
// where it fills the GPU.  Us a pass, a slice of 32 voxels to a block / so: 60 jobs of
// 2,000 voxels of 2-3 observations 290 / 154, of 20-30 570 / 514; 128 jobs of 500
// voxels 215 / 178; but 16 jobs of 100 43 / 64.  (From kShortVoxels on, so that a
// job which alone has one thread to a voxel has it in every batch.)
inline bool batch_voxels_whole(int64_t n_voxels) { return n_voxels >= kShortVoxels; }
// Lanes per scan in the solve kernel, for a launch of n_scans scans in all (a
// handle's, or a batch group's): 8 while the GPU has few warps to each of its
// 608 SM sub-partitions, else 1; the results have the same bits.  Both sides,
// launch included: 500 scans 18.5 us with one lane and 12.4 with eight, 4000
// scans 19.6 and 16.3, 6000 scans 20.5 and 18.4, 10,000 scans 21.7 and 31.6.
constexpr int64_t kLaneSolveScans = 6144;
__host__ __device__ inline int solve_lanes(int64_t n_scans) { return n_scans <= kLaneSolveScans ? 8 : 1; }
inline int64_t solve_blocks(int64_t n_scans, int lanes) {
  const int per = kSolveThreads / lanes;
  return (n_scans + per - 1) / per;
}
// the solve's partial sums of the predicted reduction: one for every kPredScans scans
constexpr int kPredScans = 8;
__host__ __device__ inline int64_t pred_parts(int64_t n_scans) { return (n_scans + kPredScans - 1) / kPredScans; }

// Which FP64 kernels of an iteration may start under the tail of the one before
// (launch_dependent).  A block that starts early takes the first place that
// comes free, so a grid that does not fill the chip ends up on the few SMs that
// drained first and shares their FP64 pipes, with the others idle; started
// after the drain it is spread over all SMs.  So early only
//   the solve       of at most 16 scans an SM, two blocks (and the scan pass
//                   before it spends 0.5 ns a scan on it, see grid_order),
//   the voxel pass  of at most 5/3 blocks an SM (with 282 blocks the scan pass
//                   behind it loses, with 250 it does not), and in a batch,
//                   whose groups run beside each other, where the scan pass
//                   fills the chip,
//   the scan pass   where it and the voxel pass before it are just under four
//                   blocks an SM (both then have room on every SM; with 600
//                   blocks 52 us instead of 55, with 613 95 instead of 85),
//                   or with a grid that fills the chip (three resident blocks)
//                   and is not so large that the wait itself costs more
//                   (grid_order: 2 us at 4,000 scans).
// Measured, us an iteration with none / all / these early: 20 scans and 200
// voxels 45.8 / 40.5 / 40.2; 20 and 5,500 139 / 204 / 137; 20 and 20,000 382 /
// 923 / 382; 100 and 20,000 142 / 253 / 138; 1,000 and 50,000 474 / 470 / 470;
// 10,000 and 300,000 1,155 / 1,158 / 1,151.
constexpr int64_t kSMs = 152;
inline bool early_solve(int64_t n_scans) { return n_scans <= 16 * kSMs; }
inline bool early_voxel_pass_f64(int64_t blocks) { return 3 * blocks <= 5 * kSMs; }
inline bool early_scan_pass_f64(int64_t blocks, int64_t voxel_blocks) {
  return blocks + voxel_blocks <= 4 * kSMs - 8 || (blocks >= 3 * kSMs && blocks <= 28 * kSMs);
}

// Launch of an iteration kernel; with dependent = true it may start while the
// kernel before it in the stream drains (see grid_wait in mmba_internal.cuh).
template <typename... P, typename... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), int64_t blocks, int threads, cudaStream_t stream,
                                    bool dependent, A&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = stream;
  cfg.attrs = &at;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Launch of a set-up kernel (a load's, or the preprocessing's) that may start
// while the one before it drains, as launch_dependent's.  The kernel calls
// grid_wait() first and grid_launch_next() after it, so when a kernel starts
// all but the one before it have finished; pointers to what that one writes
// are plain, not __restrict__, so that no load through them moves above the
// wait.  A set-up is a chain of thirty to ninety small kernels with 2 us
// between two: a load of 20 scans 308 -> 246 us, of 500 scans 445 -> 392 us, of
// the city (15M clusters) 4209 -> 4119 us; 65,000 points preprocessed in 675 us
// instead of 758.  (Only launches of at most 1216 blocks so: 404 us at 500
// scans, 4150 us at the city.)
template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream,
                                  A&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// ---- batched launches over a job group (one launch per kind for the group's jobs) ----
cudaError_t launch_batch_solve(const JobGroup& T, int64_t n_blocks, cudaStream_t stream);
cudaError_t launch_batch_voxel_pass_f64(const JobGroup& T, int64_t n_blocks, int use_trial, cudaStream_t stream);
cudaError_t launch_batch_scan_pass_f64(const JobGroup& T, int64_t n_blocks, cudaStream_t stream);
// min_blocks in {4, 6, 8} (register cap of the batch voxel pass), pf = L2
// prefetch distance in slot rows (0 = none); neither changes the results
cudaError_t launch_batch_voxel_pass_mixed(const JobGroup& T, int64_t n_blocks, int use_trial, cudaStream_t stream,
                                          int min_blocks = 6, int pf = 2);
cudaError_t launch_batch_scan_pass_mixed(const JobGroup& T, int64_t n_blocks, cudaStream_t stream);

// ---- iteration (FP64) ----
// dependent = true: an iteration's launch, which may overlap the tail of the
// kernel before it (launch_dependent); next_early = true: the launch after it is
// one.
// decide_mode: 0 = LM decision in the launch's last block (an iteration's
// trial pass), 1 = only install the summed cost (evaluation at the current
// poses), -1 = no decision (planes for output)
cudaError_t launch_voxel_pass_f64(const DevLayout& L, const double* poses2, double* planes2, double* full_out,
                                  double* cost_part, const double* pred_part, DevState* st, int use_trial,
                                  int decide_mode, cudaStream_t stream, bool dependent = false);
cudaError_t launch_scan_pass_f64(const DevLayout& L, const double* poses2, const double* planes2, double* gH,
                                 const DevState* st, int force, cudaStream_t stream, bool dependent = false,
                                 bool next_early = false);
// sref/stab2 non-null: also write the trial FP32 scan table (mixed precision)
// voxel-sharded solve: this handle's summed trial cost into *out (device);
// the LM decision from the total trial cost over all shards
cudaError_t launch_shard_cost(const double* cost_part, int64_t n_cost, double* out, cudaStream_t stream);
cudaError_t launch_shard_decide(const DevLayout& L, const double* pred_part, DevState* st, double trial_total,
                                cudaStream_t stream);
cudaError_t launch_solve_f64(const DevLayout& L, double* poses2, const double* gH, double* pred_part, DevState* st,
                             const double* sref, float* stab2, cudaStream_t stream, bool dependent = false);
cudaError_t launch_decide(const double* cost_part, int64_t n_cost, const double* pred_part, int64_t n_pred,
                          DevState* st, int mode, cudaStream_t stream);

// ---- layout build / primitives ----
// Stable LSD radix sort of (key, value) pairs on the low `bits` bits of the
// keys (n < 2^32).  Buffers of n entries each and scratch of
// radix_scratch_count(n) int64 are supplied by the caller; the sorted pairs end
// in *keys and *vals, which each pass (radix_passes) exchanges with *tmp_keys
// and *tmp_vals.  With positions = true the values are the positions 0 .. n - 1
// and *vals need not be filled.
int64_t radix_scratch_count(int64_t n);
// passes of a sort, one a digit: none for one element, which stays where it is
inline int radix_passes(int64_t n, int bits) { return n <= 1 || bits <= 0 ? 0 : (bits + 7) / 8; }
// wait = false: a tile does not wait for the counts of the tiles before it but
// counts their keys itself, as it does when a wait runs out (a check's sort).
cudaError_t radix_sort_pairs(uint32_t** keys, uint32_t** vals, uint32_t** tmp_keys, uint32_t** tmp_vals, int64_t n,
                             int bits, bool positions, int64_t* scratch, cudaStream_t stream, int64_t* launches,
                             bool wait = true);
// The same for 64-bit keys (bits up to 64).
cudaError_t radix_sort_pairs64(uint64_t** keys, uint32_t** vals, uint64_t** tmp_keys, uint32_t** tmp_vals, int64_t n,
                               int bits, bool positions, int64_t* scratch, cudaStream_t stream, int64_t* launches,
                               bool wait = true);
// The library's stream-ordered memory pool of a device (freed memory stays
// mapped for reuse); NULL if it cannot be created.
cudaMemPool_t library_pool(int device);

// Exclusive prefix sum of n int64 values in place; scratch of scan_scratch_count(n).
int64_t scan_scratch_count(int64_t n);
cudaError_t exclusive_scan_i64(int64_t* data, int64_t n, int64_t* scratch, cudaStream_t stream, int64_t* launches);

struct LoadInput {
  int32_t n_scans;
  int64_t n_voxels;
  int64_t n_obs;
  const int64_t* voxel_off;  // device
  const int32_t* obs_scan;   // device
  const double* agg;         // device, n_obs x 10 (AoS)
  int32_t agg_form;          // 0 raw sums, 1 centred
  const double* poses;       // device, n_scans x 12
};

// validation results (first violating index per check, or -1)
struct ValidateResult {
  long long first_bad_offset;
  long long first_empty_voxel;
  long long first_bad_scan;
  long long first_bad_count;
  long long first_nonfinite_agg;
  long long first_bad_pose;
  long long n_obs_seen;
  long long max_len;
};
// What the validation of a load's inputs writes besides its result: the inputs'
// copies in the handle (each may be null), and the poses' translations in FP32.
struct InputCopies {
  int64_t* voxel_off;
  int32_t* obs_scan;
  double* poses;
  float4* t32;
};
// the result's start values, and those of the spatial order's bounding box (8 words)
cudaError_t launch_load_init(ValidateResult* d_res, uint32_t* box, cudaStream_t stream, int64_t* launches);
// offsets, scan ids and poses
cudaError_t launch_validate(const LoadInput& in, const InputCopies& to, ValidateResult* d_res, cudaStream_t stream,
                            int64_t* launches);
// clusters [o0, o1) of agg; dst non-null: also copied there, at the same places
cudaError_t launch_validate_agg(const double* agg, int64_t o0, int64_t o1, double* dst, ValidateResult* d_res,
                                cudaStream_t stream, int64_t* launches);

// Build the device layout; buffers are allocated through the given allocators
// as sizes become known.
struct Allocator {
  void* (*fn)(void* self, size_t bytes);
  void* self;
};
// Device arrays of one allocation, each on a 256-byte boundary: a load needs
// some forty arrays, and an allocation is a call into the driver.
class ArrayGroup {
 public:
  template <typename T>
  void add(T** p, size_t count) {
    items_.push_back({(void**)(void*)p, total_});
    total_ += (sizeof(T) * (count ? count : 1) + 255) & ~(size_t)255;
  }
  bool empty() const { return items_.empty(); }
  bool allocate(Allocator a) {
    char* base = (char*)a.fn(a.self, total_);
    for (auto& it : items_) *it.p = base ? base + it.at : nullptr;
    return base != nullptr;
  }

 private:
  struct Item {
    void** p;
    size_t at;
  };
  std::vector<Item> items_;
  size_t total_ = 0;
};
struct LayoutBuffers {
  int64_t* slice_off;
  int32_t* vlen;
  int32_t* vperm;
  double* ve;
  int32_t* ve_scan;
  int64_t* scan_off;
  int32_t* scans_by_len;  // scans by decreasing observation count, ties by index
  double* se;
  int32_t* se_vox;
  int64_t n_elems;  // at least the slots of all slices
  int64_t n_slices;
  int64_t max_len;  // observations of the longest voxel (rows of the longest slice)
  // kept only when the FP64 copies are not built (mixed precision)
  int32_t* vrank;        // input voxel -> sorted position
  int2* place;           // observation -> (sorted voxel position, row)
  double* vscale;        // input voxel -> 2 / N_i
  uint32_t* scan_order;  // scan-major position -> observation
  // kept only by a load with defer_scale: vstart[p] = observations of the
  // voxels before sorted position p (p = 0 .. n_voxels)
  int64_t* vstart;
};
// `keep` allocates the buffers of *out, `temp` the build's temporaries (the
// caller frees those after the stream has drained).
// With fill_f64 the FP64 cluster copies are filled; without, only the index
// structures are built and the maps above are kept for the FP32 copies (se_vox
// is left for the mixed path's scan-major copy to fill).  t32: the poses'
// translations in FP32 (launch_validate); box: launch_load_init.
// With defer_scale the clusters are not read (vscale is left for
// launch_vscale, voxel range by voxel range, as the clusters arrive).
cudaError_t build_layout(const LoadInput& in, const float4* t32, uint32_t* box, int max_len, bool fill_f64,
                         bool defer_scale, Allocator keep, Allocator temp, LayoutBuffers* out, cudaStream_t stream,
                         int64_t* launches);
cudaError_t launch_vscale(const LoadInput& in, int64_t v0, int64_t v1, double* vscale, cudaStream_t stream,
                          int64_t* launches);
// A load that copies its clusters in chunks of observations [o[k], o[k + 1])
// (o[0] = 0, o[n] = n_obs, at most kMaxCopyChunks chunks) groups the
// scan-major positions by chunk: (*out_q)[o[k] .. o[k + 1]) holds, ascending,
// the positions q whose observation order[q] lies in chunk k (order is a
// permutation of 0 .. n_obs - 1).  *out_q and temporaries come from temp.
constexpr int kMaxCopyChunks = 20;  // chunks halving in size: up to 2^20 - 1 windows, more than 2^31 voxels
struct ChunkBounds {
  int64_t o[kMaxCopyChunks + 1];
  int n;
};
cudaError_t group_by_chunk(const uint32_t* order, int64_t n_obs, const ChunkBounds& cb, const uint32_t** out_q,
                           Allocator temp, cudaStream_t stream, int64_t* launches);

// ---- mixed precision ----
cudaError_t launch_voxel_pass_mixed(const DevLayout& L, const DevMixed& X, double* full_out, double* cost_part,
                                    const double* pred_part, DevState* st, int use_trial, int decide_mode,
                                    cudaStream_t stream, bool dependent = false);
cudaError_t launch_scan_pass_mixed(const DevLayout& L, const DevMixed& X, const double* poses2, double* gH,
                                   DevState* st, int force, cudaStream_t stream, bool next_early = false);
cudaError_t launch_scan_table(int32_t n_scans, const double* poses2, const double* sref, float* stab2, int buf,
                              cudaStream_t stream);
// Build (or rebuild) the FP32 copies, frames, anchors and reference poses at
// the poses of buffer 0 of poses2.
struct MixedBuffers {
  float4* ve32;
  float4* vstate;
  float* se32;
  float4* vanchor;
  double* sref;
  float* stab2;
  float4* planes32_2;
  int32_t* se_vox;  // the layout's, filled with the scan-major copy
};
cudaError_t build_mixed(const LoadInput& in, const LayoutBuffers& lb, const double* poses2, MixedBuffers& mb,
                        cudaStream_t stream, int64_t* launches);
// The same in stages, for a load that overlaps the clusters' copy: begin
// (reference poses); input voxels [v0, v1) with their observations [o0, o1)
// (frames and anchors, the slots staged voxel by voxel in the sorted voxel
// order, 3 float4 per observation at lb.vstart, and the observations'
// scan-major entries; their clusters on the device); place (every staged slot
// to its slice, padding zero); end (the scan table; with scan_filled false
// also the scan-major copy from the placed slots).  scan_major fills the
// scan-major entries at positions qlist[i0 .. i1) (positions i0 .. i1 when
// qlist is null: chunk_q of group_by_chunk lists a chunk's), from the staged
// slots when staging is non-null, else from the placed ones.
cudaError_t build_mixed_begin(const LoadInput& in, const double* poses2, MixedBuffers& mb, cudaStream_t stream,
                              int64_t* launches);
cudaError_t build_mixed_voxels(const LoadInput& in, const LayoutBuffers& lb, const double* poses2, MixedBuffers& mb,
                               int64_t v0, int64_t v1, int64_t o0, int64_t o1, float4* staging,
                               const uint32_t* chunk_q, cudaStream_t stream, int64_t* launches);
cudaError_t build_mixed_place(const LoadInput& in, const LayoutBuffers& lb, MixedBuffers& mb, const float4* staging,
                              cudaStream_t stream, int64_t* launches);
cudaError_t build_mixed_scan_major(const LoadInput& in, const LayoutBuffers& lb, MixedBuffers& mb,
                                   const float4* staging, const uint32_t* qlist, int64_t i0, int64_t i1,
                                   cudaStream_t stream, int64_t* launches);
cudaError_t build_mixed_end(const LoadInput& in, const LayoutBuffers& lb, const double* poses2, MixedBuffers& mb,
                            cudaStream_t stream, int64_t* launches, bool scan_filled = false);

// bounded-wait check: out[0] = 1 if an mbarrier wait that cannot complete gave up
cudaError_t launch_wait_probe(int limit, int32_t* out, cudaStream_t stream);

// points -> centred clusters
cudaError_t launch_aggregate_points(int64_t n_obs, const int64_t* point_off, const double* points, double* agg_out,
                                    cudaStream_t stream);

}  // namespace mmba
