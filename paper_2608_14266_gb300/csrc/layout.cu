// Device-side layout build (the index mappers of Algorithm 1) and the
// primitives it uses: a stable LSD radix sort of (key, value) pairs, an
// exclusive scan, input validation and point-cluster formation (Eq. 2).
// Everything here runs once per load; none of it is on the per-iteration path.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <utility>

#include "block_order.cuh"
#include "fixed_sums.cuh"
#include "mmba_internal.cuh"
#include "mmba_kernels.h"

namespace mmba {

#define RETURN_IF(err)                   \
  do {                                   \
    cudaError_t e_ = (err);              \
    if (e_ != cudaSuccess) return e_;    \
  } while (0)

// ============================================================================
// Exclusive scan of int64: (1) each tile's sum; (2) each tile scanned behind the
// sum of the tiles before it, which its block adds up itself while there are
// few (their recursive scan beyond).  Bound by DRAM: two reads and a write (a
// scan of every tile and a pass that adds the prefixes back wrote twice).  A
// warp takes 256 consecutive elements, two to a lane, so its accesses are whole
// lines (120M points: all prefix sums of a call 360 -> 200 us).
// ============================================================================
constexpr int kScanBlock = 512;
constexpr int kScanRounds = 4;  // of 64 elements a warp
constexpr int64_t kScanTile = (int64_t)kScanBlock * 2 * kScanRounds;
constexpr int64_t kScanOwnTiles = 4096;  // tiles whose sums a block adds up itself

// elements i, i + 1 (0 past the end)
__device__ __forceinline__ longlong2 scan_load(const int64_t* data, int64_t i, int64_t n, bool pair) {
  if (pair && i + 1 < n) return *reinterpret_cast<const longlong2*>(data + i);
  return make_longlong2(i < n ? data[i] : 0, i + 1 < n ? data[i + 1] : 0);
}

// the block's total of v, in every thread
__device__ __forceinline__ int64_t scan_block_total(int64_t v, int64_t* warp_tot) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) warp_tot[threadIdx.x >> 5] = v;
  __syncthreads();
  int64_t t = 0;
#pragma unroll
  for (int k = 0; k < kScanBlock / 32; ++k) t += warp_tot[k];
  __syncthreads();
  return t;
}

__global__ void __launch_bounds__(kScanBlock) scan_sums_kernel(const int64_t* data, int64_t n, int64_t* tile_sums) {
  grid_wait();
  grid_launch_next();
  __shared__ int64_t warp_tot[kScanBlock / 32];
  const bool pair = reinterpret_cast<uintptr_t>(data) % 16 == 0;
  const int64_t i0 = (int64_t)blockIdx.x * kScanTile + 2 * threadIdx.x;
  longlong2 v[kScanRounds];
#pragma unroll
  for (int r = 0; r < kScanRounds; ++r) v[r] = scan_load(data, i0 + r * (2 * kScanBlock), n, pair);
  int64_t t = 0;
#pragma unroll
  for (int r = 0; r < kScanRounds; ++r) t += v[r].x + v[r].y;
  t = scan_block_total(t, warp_tot);
  if (threadIdx.x == 0) tile_sums[blockIdx.x] = t;
}

// before: the tiles' sums (scanned = false) or their exclusive scan; null with one tile
__global__ void __launch_bounds__(kScanBlock) scan_tiles_kernel(int64_t* data, int64_t n, const int64_t* before,
                                                                bool scanned) {
  grid_wait();
  grid_launch_next();
  __shared__ int64_t warp_tot[kScanBlock / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const bool pair = reinterpret_cast<uintptr_t>(data) % 16 == 0;
  const int64_t i0 = (int64_t)blockIdx.x * kScanTile + w * (64 * kScanRounds) + 2 * lane;
  longlong2 v[kScanRounds];
#pragma unroll
  for (int r = 0; r < kScanRounds; ++r) v[r] = scan_load(data, i0 + 64 * r, n, pair);
  int64_t pre = 0;
  if (before) {
    if (scanned) {
      pre = before[blockIdx.x];
    } else {
      for (int64_t k = threadIdx.x; k < blockIdx.x; k += kScanBlock) pre += before[k];
      pre = scan_block_total(pre, warp_tot);
    }
  }
  // the warp's running sums, round by round
  int64_t run = 0, start[kScanRounds];
#pragma unroll
  for (int r = 0; r < kScanRounds; ++r) {
    const int64_t x = v[r].x + v[r].y;
    int64_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    start[r] = run + incl - x;
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) warp_tot[w] = run;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kScanBlock / 32; ++k) pre += k < w ? warp_tot[k] : 0;
#pragma unroll
  for (int r = 0; r < kScanRounds; ++r) {
    const int64_t i = i0 + 64 * r;
    const int64_t x = pre + start[r], y = x + v[r].x;
    if (pair && i + 1 < n) {
      *reinterpret_cast<longlong2*>(data + i) = make_longlong2(x, y);
    } else {
      if (i < n) data[i] = x;
      if (i + 1 < n) data[i + 1] = y;
    }
  }
}

int64_t scan_scratch_count(int64_t n) {
  int64_t total = 0;
  while (n > kScanTile) {
    n = (n + kScanTile - 1) / kScanTile;
    total += n + 1;
  }
  return total + 1;
}

cudaError_t exclusive_scan_i64(int64_t* data, int64_t n, int64_t* scratch, cudaStream_t stream, int64_t* launches) {
  if (n <= 0) return cudaSuccess;
  const int64_t tiles = (n + kScanTile - 1) / kScanTile;
  if (tiles == 1) {
    launch_chained(scan_tiles_kernel, 1, kScanBlock, 0, stream, data, n, nullptr, false);
    ++*launches;
    return cudaGetLastError();
  }
  int64_t* sums = scratch;
  launch_chained(scan_sums_kernel, (unsigned)tiles, kScanBlock, 0, stream, data, n, sums);
  ++*launches;
  RETURN_IF(cudaGetLastError());
  const bool scanned = tiles > kScanOwnTiles;
  if (scanned) RETURN_IF(exclusive_scan_i64(sums, tiles, scratch + tiles + 1, stream, launches));
  launch_chained(scan_tiles_kernel, (unsigned)tiles, kScanBlock, 0, stream, data, n, sums, scanned);
  ++*launches;
  return cudaGetLastError();
}

// ============================================================================
// Stable LSD radix sort, 8-bit digits, one kernel per digit.
//  (1) the keys are read once and every digit's histogram taken;
//  (2) per digit, each tile loads its elements (all loads issued up front);
//      each warp ranks its 512 consecutive elements in order with match masks
//      and warp-private digit counters (stable, deterministic, no block
//      barrier); per-digit prefix sums over the warps and the digits place the
//      tile digit-sorted in shared memory, and every digit's run goes to its
//      global place with consecutive threads on consecutive addresses
//      (full-sector writes).
// A run's global place is the digit's start (a 256-entry scan of the
// histogram, by every block) plus the counts of that digit in the tiles
// before, which come from the tiles themselves: each publishes its counts in
// one 64-bit word a digit, walks back over the words of the tiles before it
// until it meets one that holds a running total, and publishes its own running
// total (single-pass prefix sum with decoupled look-back; Merrill & Garland,
// NVIDIA technical report NVR-2016-002).  Tiles are numbered in the order the
// blocks start, so a tile waits only for tiles whose blocks are running and
// publish before they wait; a wait that lasts kLookLimit polls all the same
// ends with the tile counting the keys before it itself (ba_check_sort has it do
// so at once).
//
// Bound at large sizes: instruction issue (57% active) and the look-back's
// waits.  Against a histogram kernel and a prefix sum of one to three kernels
// per digit: 120M 32-bit keys in 3 digits with their packing 2.81 -> 2.54 ms
// (the result in either buffer saves a copy after an odd number); 7.9M 36-bit
// keys 0.70 -> 0.45 ms; a problem of 25,000 voxels loads in 22 launches fewer
// (618 -> 575 us).
// ============================================================================
constexpr int kRadixBlock = 256;
constexpr int kRadixItems = 16;  // chunks per tile
constexpr int64_t kRadixTile = (int64_t)kRadixBlock * kRadixItems;
constexpr int kRadixWarps = kRadixBlock / 32;
constexpr int kRadixPasses = 8;      // digits of a 64-bit key
constexpr int kLookLimit = 1 << 20;  // polls of one word
constexpr int kLookAhead = 4;        // words of a look-back in flight
constexpr int64_t kCountBlocks = 4 * kSMs;

// a tile's word for one digit: the pass it belongs to, whether it is the
// running total (tiles up to this one) or the tile's own count, and the value
// (below 2^32); zero before the first pass
__device__ __forceinline__ uint64_t look_word(int pass, bool total, uint32_t v) {
  return ((uint64_t)(2 * pass + 2 + (total ? 1 : 0)) << 32) | v;
}
__device__ __forceinline__ uint64_t look_load(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void look_store(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// histograms of the first `passes` digits: hist[256 pass + digit]
template <typename K>
__global__ void __launch_bounds__(kRadixBlock) radix_count_kernel(const K* keys, int64_t n, int passes,
                                                                  uint32_t* hist) {
  grid_wait();
  grid_launch_next();
  __shared__ uint32_t cnt[kRadixPasses * 256];
  for (int k = threadIdx.x; k < passes * 256; k += kRadixBlock) cnt[k] = 0;
  __syncthreads();
  for (int64_t base = (int64_t)blockIdx.x * kRadixTile; base < n; base += (int64_t)gridDim.x * kRadixTile) {
    // every key of the thread loaded before the first count
    K key[kRadixItems];
#pragma unroll
    for (int c = 0; c < kRadixItems; ++c) {
      const int64_t i = base + (int64_t)c * kRadixBlock + threadIdx.x;
      key[c] = i < n ? keys[i] : (K)0;
    }
#pragma unroll
    for (int c = 0; c < kRadixItems; ++c)
      if (base + (int64_t)c * kRadixBlock + threadIdx.x < n)
        for (int p = 0; p < passes; ++p) atomicAdd(&cnt[256 * p + ((unsigned)(key[c] >> (8 * p)) & 255u)], 1u);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < passes * 256; k += kRadixBlock)
    if (cnt[k]) atomicAdd(hist + k, cnt[k]);
}

template <typename K>
constexpr size_t radix_scatter_smem() {
  return (size_t)kRadixTile * (sizeof(K) + sizeof(uint32_t));
}

// exclusive prefix sum of one value per thread of the block (256 threads)
__device__ __forceinline__ uint32_t block_exclusive(uint32_t v, uint32_t* wsum) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) wsum[w] = incl;
  __syncthreads();
  uint32_t pre = 0;
  for (int k = 0; k < w; ++k) pre += wsum[k];
  return pre + incl - v;
}

// One tile of a digit's pass.  kFull: the tile holds kRadixTile elements.
// vals_in null: the values are the positions 0 .. n - 1.
struct RadixShared {
  uint32_t gstart[256];       // global start of this tile's run of each digit
  uint32_t lstart[256];       // tile-local start of each digit
  int wc[kRadixWarps][256];   // per warp: count, then start, of each digit
  uint32_t wsum[2][kRadixWarps];
};

template <typename K, bool kFull, bool kWait>
__device__ __forceinline__ void radix_tile(const K* __restrict__ keys_in, const uint32_t* __restrict__ vals_in,
                                           K* __restrict__ keys_out, uint32_t* __restrict__ vals_out, int64_t n,
                                           int64_t tile, int pass, uint32_t total, uint64_t* look, K* skey,
                                           uint32_t* sval, RadixShared& sh) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int shift = 8 * pass;
  const int64_t base = tile * kRadixTile;
  const int tile_n = kFull ? (int)kRadixTile : (int)(n - base);
  // warp w owns the tile's elements [w * 512, (w + 1) * 512), 32 per round
  const int li0 = w * (32 * kRadixItems) + lane;
  K key[kRadixItems];
  uint32_t val[kRadixItems];
#pragma unroll
  for (int j = 0; j < kRadixItems; ++j) {
    const int li = li0 + j * 32;
    key[j] = kFull || li < tile_n ? keys_in[base + li] : (K)0;
    val[j] = kFull || li < tile_n ? (vals_in ? vals_in[base + li] : (uint32_t)(base + li)) : 0u;
  }
  // 256 for lanes past the end
  auto digit = [&](int j) {
    return kFull || li0 + j * 32 < tile_n ? (unsigned)(key[j] >> shift) & 255u : 256u;
  };
  // rank within the warp, in element order (rounds, then lanes)
  uint32_t rk[kRadixItems / 2];  // two ranks (below 512) each
#pragma unroll
  for (int j = 0; j < kRadixItems; ++j) {
    const unsigned d = digit(j);
    const unsigned same = __match_any_sync(0xffffffffu, d);
    const int first = kFull || d < 256u ? sh.wc[w][d] : 0;
    const uint32_t r = (uint32_t)(first + __popc(same & ((1u << lane) - 1u)));
    rk[j / 2] = j & 1 ? rk[j / 2] | (r << 16) : r;
    __syncwarp();
    if ((kFull || d < 256u) && lane == __ffs(same) - 1) sh.wc[w][d] = first + __popc(same);
    __syncwarp();
  }
  __syncthreads();
  // per digit (thread tid = digit): warps' starts within the digit, tile total
  uint32_t run = 0;
#pragma unroll
  for (int k = 0; k < kRadixWarps; ++k) {
    const int x = sh.wc[k][tid];
    sh.wc[k][tid] = (int)run;
    run += (uint32_t)x;
  }
  look_store(look + 256 * tile + tid, look_word(pass, tile == 0, run));
  sh.lstart[tid] = block_exclusive(run, sh.wsum[0]);
  const uint32_t digit0 = block_exclusive(total, sh.wsum[1]);  // the digit's global start
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kRadixItems; ++j) {
    const unsigned d = digit(j);
    if (kFull || d < 256u) {
      const int p = (int)sh.lstart[d] + sh.wc[w][d] + (int)((rk[j / 2] >> (16 * (j & 1))) & 0xffffu);
      skey[p] = key[j];
      sval[p] = val[j];
    }
  }
  // the digit's elements in the tiles before
  uint32_t before = 0;
  bool gave_up = false;
  bool done = tile == 0;
  for (int64_t t = tile - 1; !done && !gave_up; t -= kLookAhead) {
    // the words of several tiles on their way at once (a word's load is most of a step)
    uint64_t v[kLookAhead];
#pragma unroll
    for (int k = 0; k < kLookAhead; ++k) v[k] = t - k >= 0 ? look_load(look + 256 * (t - k) + tid) : 0;
#pragma unroll
    for (int k = 0; k < kLookAhead; ++k) {
      if (done || gave_up || t - k < 0) continue;
      for (int it = 0; (uint32_t)(v[k] >> 32) < (uint32_t)(2 * pass + 2) && it < (kWait ? kLookLimit : 0); ++it)
        v[k] = look_load(look + 256 * (t - k) + tid);
      const uint32_t tag = (uint32_t)(v[k] >> 32);
      gave_up = tag < (uint32_t)(2 * pass + 2);
      before += (uint32_t)v[k];
      done = tag == (uint32_t)(2 * pass + 3);
    }
  }
  if (__syncthreads_or(gave_up)) {  // count them here
    sh.lstart[tid] = 0;
    __syncthreads();
    for (int64_t i = tid; i < base; i += kRadixBlock)
      atomicAdd(&sh.lstart[(unsigned)(keys_in[i] >> shift) & 255u], 1u);
    __syncthreads();
    before = sh.lstart[tid];
    __syncthreads();
    sh.lstart[tid] = block_exclusive(run, sh.wsum[0]);
  }
  if (tile > 0) look_store(look + 256 * tile + tid, look_word(pass, true, before + run));
  // (less the local start, so that an element's place is gstart + its place in the tile)
  sh.gstart[tid] = digit0 + before - sh.lstart[tid];
  __syncthreads();
#pragma unroll 4
  for (int p = tid; p < tile_n; p += kRadixBlock) {
    const K k = skey[p];
    const uint32_t dst = sh.gstart[(unsigned)(k >> shift) & 255u] + (uint32_t)p;
    keys_out[dst] = k;
    vals_out[dst] = sval[p];
  }
}

// kBlocks: resident blocks per SM that the registers are held to
template <typename K, int kBlocks, bool kWait>
__global__ void __launch_bounds__(kRadixBlock, kBlocks)
    radix_scatter_kernel(const K* keys_in, const uint32_t* vals_in,
                         K* keys_out, uint32_t* vals_out, int64_t n, int pass,
                         const uint32_t* hist, uint32_t* ticket, uint64_t* look) {
  grid_wait();
  grid_launch_next();
  extern __shared__ __align__(16) unsigned char radix_smem[];
  K* skey = reinterpret_cast<K*>(radix_smem);
  uint32_t* sval = reinterpret_cast<uint32_t*>(radix_smem + sizeof(K) * kRadixTile);
  __shared__ RadixShared sh;
  __shared__ uint32_t s_tile;
  const int tid = threadIdx.x;
  if (tid == 0) s_tile = atomicAdd(ticket + pass, 1u);
#pragma unroll
  for (int k = 0; k < kRadixWarps; ++k) sh.wc[k][tid] = 0;
  const uint32_t total = hist[256 * pass + tid];
  __syncthreads();
  const int64_t tile = s_tile;
  if ((tile + 1) * kRadixTile <= n)
    radix_tile<K, true, kWait>(keys_in, vals_in, keys_out, vals_out, n, tile, pass, total, look, skey, sval, sh);
  else
    radix_tile<K, false, kWait>(keys_in, vals_in, keys_out, vals_out, n, tile, pass, total, look, skey, sval, sh);
}

__global__ void positions_kernel(int64_t n, uint32_t* v) {
  grid_wait();
  grid_launch_next();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) v[i] = (uint32_t)i;
}

// scratch: the tiles' words, the histograms and the tile counters
int64_t radix_scratch_count(int64_t n) {
  const int64_t tiles = (n + kRadixTile - 1) / kRadixTile;
  return 256 * (tiles > 0 ? tiles : 1) + kRadixPasses * 128 + kRadixPasses;
}

template <typename K>
static cudaError_t radix_sort_pairs_t(K** keys, uint32_t** vals, K** tmp_keys, uint32_t** tmp_vals, int64_t n, int bits,
                                      bool positions, int64_t* scratch, cudaStream_t stream, int64_t* launches,
                                      bool wait) {
  const int passes = radix_passes(n, bits);
  if (passes == 0) {
    if (!positions || n <= 0) return cudaSuccess;
    launch_chained(positions_kernel, (unsigned)((n + 255) / 256), 256, 0, stream, n, *vals);
    ++*launches;
    return cudaGetLastError();
  }
  const int64_t tiles = (n + kRadixTile - 1) / kRadixTile;
  uint64_t* look = (uint64_t*)scratch;
  uint32_t* hist = (uint32_t*)(look + 256 * tiles);
  uint32_t* ticket = hist + kRadixPasses * 256;
  // two resident blocks (no spilled registers) while that is one wave, else more
  // in flight: 65,000 points 758 -> 732 us a call with two, 120M 2.59 -> 2.83 ms
  const auto scatter = !wait                ? radix_scatter_kernel<K, 2, false>
                       : tiles <= 2 * kSMs ? radix_scatter_kernel<K, 2, true>
                                           : radix_scatter_kernel<K, sizeof(K) == 4 ? 4 : 3, true>;
  RETURN_IF(cudaFuncSetAttribute(scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)radix_scatter_smem<K>()));
  RETURN_IF(cudaMemsetAsync(scratch, 0, sizeof(int64_t) * (size_t)radix_scratch_count(n), stream));
  launch_chained(radix_count_kernel<K>, (unsigned)(tiles < kCountBlocks ? tiles : kCountBlocks), kRadixBlock, 0, stream,
                 *keys, n, passes, hist);
  ++*launches;
  RETURN_IF(cudaGetLastError());
  for (int p = 0; p < passes; ++p) {
    launch_chained(scatter, (unsigned)tiles, kRadixBlock, radix_scatter_smem<K>(), stream, *keys,
                   p == 0 && positions ? nullptr : *vals, *tmp_keys, *tmp_vals, n, p, hist, ticket, look);
    ++*launches;
    RETURN_IF(cudaGetLastError());
    std::swap(*keys, *tmp_keys);
    std::swap(*vals, *tmp_vals);
  }
  return cudaSuccess;
}

cudaError_t radix_sort_pairs(uint32_t** keys, uint32_t** vals, uint32_t** tmp_keys, uint32_t** tmp_vals, int64_t n,
                             int bits, bool positions, int64_t* scratch, cudaStream_t stream, int64_t* launches,
                             bool wait) {
  return radix_sort_pairs_t<uint32_t>(keys, vals, tmp_keys, tmp_vals, n, bits, positions, scratch, stream, launches,
                                      wait);
}

cudaError_t radix_sort_pairs64(uint64_t** keys, uint32_t** vals, uint64_t** tmp_keys, uint32_t** tmp_vals, int64_t n,
                               int bits, bool positions, int64_t* scratch, cudaStream_t stream, int64_t* launches,
                               bool wait) {
  return radix_sort_pairs_t<uint64_t>(keys, vals, tmp_keys, tmp_vals, n, bits, positions, scratch, stream, launches,
                                      wait);
}

// ============================================================================
// Validation: the first violating index of each check (atomicMin, so the
// result does not depend on scheduling).
// ============================================================================
__device__ inline void amin(long long* p, long long v) { atomicMin(p, v); }

constexpr int kValidateThreads = 256;

__global__ void load_init_kernel(ValidateResult* r, uint32_t* box) {
  grid_launch_next();
  const int k = threadIdx.x;
  if (k < 6) box[k] = k < 3 ? 0xffffffffu : 0u;  // minima, maxima
  if (k == 0) {
    r->first_bad_offset = r->first_empty_voxel = r->first_bad_scan = r->first_bad_count = r->first_nonfinite_agg =
        r->first_bad_pose = LLONG_MAX;
    r->n_obs_seen = 0;
    r->max_len = 0;
  }
}

cudaError_t launch_load_init(ValidateResult* d_res, uint32_t* box, cudaStream_t stream, int64_t* launches) {
  load_init_kernel<<<1, 32, 0, stream>>>(d_res, box);
  ++*launches;
  return cudaGetLastError();
}

// offsets and voxel lengths, scan ids, and poses (their translations also into
// t32 in FP32, for the spatial order), a range of blocks each, and their copies
// where asked for.  Every thread of a voxel block reaches the warp reduction.
__global__ void __launch_bounds__(kValidateThreads) validate_kernel(LoadInput in, int64_t voxel_blocks,
                                                                    int64_t scan_blocks, InputCopies to,
                                                                    ValidateResult* r) {
  grid_wait();
  grid_launch_next();
  int64_t blk = blockIdx.x;
  if (blk < voxel_blocks) {
    const int64_t i = blk * kValidateThreads + threadIdx.x;
    int len = 0;  // the voxel's observation count (capped at 2^31 - 1), 0 if none or invalid
    if (i <= in.n_voxels) {
      const int64_t a = in.voxel_off[i];
      if (to.voxel_off) to.voxel_off[i] = a;
      if (i == 0 && a != 0) amin(&r->first_bad_offset, 0);
      if (i == in.n_voxels) {
        if (a != in.n_obs) amin(&r->first_bad_offset, i);
      } else {
        const int64_t b = in.voxel_off[i + 1];
        if (b < a || a < 0 || b > in.n_obs) amin(&r->first_bad_offset, i);
        else if (b == a) amin(&r->first_empty_voxel, i);
        else len = (int)(b - a > 0x7fffffff ? 0x7fffffff : b - a);
      }
    }
    // one atomic per warp (one per voxel serialises on the single word)
    const int wmax = __reduce_max_sync(0xffffffffu, len);
    if ((threadIdx.x & 31) == 0 && wmax > 0) atomicMax(&r->max_len, (long long)wmax);
    return;
  }
  blk -= voxel_blocks;
  if (blk < scan_blocks) {
    const int64_t o = blk * kValidateThreads + threadIdx.x;
    if (o < in.n_obs) {
      const int32_t j = in.obs_scan[o];
      if (to.obs_scan) to.obs_scan[o] = j;
      if (j < 0 || j >= in.n_scans) amin(&r->first_bad_scan, o);
    }
    return;
  }
  const int64_t j = (blk - scan_blocks) * kValidateThreads + threadIdx.x;
  if (j >= in.n_scans) return;
  double P[12];
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    P[k] = in.poses[12 * j + k];
    if (to.poses) to.poses[12 * j + k] = P[k];
    ok = ok && isfinite(P[k]);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const double d = P[3 * a] * P[3 * b] + P[3 * a + 1] * P[3 * b + 1] + P[3 * a + 2] * P[3 * b + 2];
      if (fabs(d - (a == b ? 1.0 : 0.0)) > 1e-6) ok = false;
    }
  if (ok) {  // proper rotation: det = +1
    const double det = P[0] * (P[4] * P[8] - P[5] * P[7]) - P[1] * (P[3] * P[8] - P[5] * P[6]) +
                       P[2] * (P[3] * P[7] - P[4] * P[6]);
    if (det < 0.0) ok = false;
  }
  if (!ok) amin(&r->first_bad_pose, j);
  to.t32[j] = make_float4(f64_to_f32(P[9]), f64_to_f32(P[10]), f64_to_f32(P[11]), 0.f);
}

// Clusters [o0, o1): finite, and at least one point; with dst given also copied
// there (the handle's own clusters).  Threads take consecutive pairs of values
// (kPair: where both arrays are 16-byte aligned) or single values, so that the
// rows of 80 bytes are read as one stream.  Bound by DRAM: 15M clusters copied
// and validated in 435 us; a row per thread was 318 us behind a copy of 360 us.
template <bool kPair>
__global__ void __launch_bounds__(kValidateThreads) validate_agg_kernel(const double* agg, int64_t o0,
                                                                        int64_t o1, double* dst,
                                                                        ValidateResult* r) {
  grid_wait();
  grid_launch_next();
  constexpr int kUnits = 4;  // loads in flight
  constexpr int64_t kRow = kPair ? 5 : 10;
  const int64_t e1 = kRow * o1;
  const int64_t first = kRow * o0 + (int64_t)blockIdx.x * (kValidateThreads * kUnits) + threadIdx.x;
  double2 v[kUnits];
#pragma unroll
  for (int k = 0; k < kUnits; ++k) {
    const int64_t e = first + k * kValidateThreads;
    v[k] = make_double2(1.0, 1.0);
    if (e < e1) {
      if (kPair)
        v[k] = reinterpret_cast<const double2*>(agg)[e];
      else
        v[k].x = v[k].y = agg[e];
    }
  }
#pragma unroll
  for (int k = 0; k < kUnits; ++k) {
    const int64_t e = first + k * kValidateThreads;
    if (e >= e1) break;
    if (dst) {
      if (kPair)
        reinterpret_cast<double2*>(dst)[e] = v[k];
      else
        dst[e] = v[k].x;
    }
    const bool fin = isfinite(v[k].x) && isfinite(v[k].y);
    const bool count = e % kRow == kRow - 1;  // holds N
    if (!fin) amin(&r->first_nonfinite_agg, e / kRow);
    if (count && !(v[k].y >= 1.0)) amin(&r->first_bad_count, e / kRow);
  }
}

cudaError_t launch_validate(const LoadInput& in, const InputCopies& to, ValidateResult* d_res, cudaStream_t stream,
                            int64_t* launches) {
  auto blocks = [](int64_t n) { return (n + kValidateThreads - 1) / kValidateThreads; };
  const int64_t nv = blocks(in.n_voxels + 1), no = blocks(in.n_obs), ns = blocks(in.n_scans);
  launch_chained(validate_kernel, (unsigned)(nv + no + ns), kValidateThreads, 0, stream, in, nv, no, to, d_res);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_validate_agg(const double* agg, int64_t o0, int64_t o1, double* dst, ValidateResult* d_res,
                                cudaStream_t stream, int64_t* launches) {
  if (o1 <= o0) return cudaSuccess;
  // pairs where every row starts on 16 bytes
  const bool pair = (reinterpret_cast<uintptr_t>(agg) | reinterpret_cast<uintptr_t>(dst)) % 16 == 0;
  const int64_t units = (pair ? 5 : 10) * (o1 - o0), per = 4 * kValidateThreads;
  const unsigned nb = (unsigned)((units + per - 1) / per);
  if (pair)
    launch_chained(validate_agg_kernel<true>, nb, kValidateThreads, 0, stream, agg, o0, o1, dst, d_res);
  else
    launch_chained(validate_agg_kernel<false>, nb, kValidateThreads, 0, stream, agg, o0, o1, dst, d_res);
  ++*launches;
  return cudaGetLastError();
}

// ============================================================================
// Layout build
// ============================================================================

// Input cluster -> centred (S, m, N).  Raw sums: m = v / N and
// S_ab = fma(-v_a, m_b, P_ab).
// (the row in 128-bit loads where its address allows: a thread with a row of its
// own is bound by the requests to L1)
__device__ inline void to_centred(const double* in, int form, double out[10]) {
  double a[10];
  if (reinterpret_cast<uintptr_t>(in) % 16 == 0) {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const double2 v = reinterpret_cast<const double2*>(in)[k];
      a[2 * k] = v.x;
      a[2 * k + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 10; ++k) a[k] = in[k];
  }
  if (form == 1) {
#pragma unroll
    for (int k = 0; k < 10; ++k) out[k] = a[k];
    return;
  }
  const double n = a[9];
  const double mx = a[6] / n, my = a[7] / n, mz = a[8] / n;
  out[0] = fma(-a[6], mx, a[0]);
  out[1] = fma(-a[6], my, a[1]);
  out[2] = fma(-a[6], mz, a[2]);
  out[3] = fma(-a[7], my, a[3]);
  out[4] = fma(-a[7], mz, a[4]);
  out[5] = fma(-a[8], mz, a[5]);
  out[6] = mx;
  out[7] = my;
  out[8] = mz;
  out[9] = n;
}

// ---- spatial order of the voxels ----
// Mean translation of the scans observing each voxel (FP32, from the table of
// the validation, summed in the voxel's observation order), and the bounding box of those means as
// order-preserving unsigned encodings of the floats (min and max are exact,
// so the box does not depend on the order of the atomics).
__device__ __forceinline__ uint32_t float_order_key(float f) {
  const uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float float_from_order_key(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__global__ void observer_mean_kernel(const int64_t* off, const int32_t* obs_scan,
                                     const float4* t32, int64_t n_voxels, float4* mean,
                                     uint32_t* box) {
  grid_wait();
  grid_launch_next();
  __shared__ uint32_t sbox[6];
  if (threadIdx.x < 6) sbox[threadIdx.x] = threadIdx.x < 3 ? 0xffffffffu : 0u;
  __syncthreads();
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n_voxels) {
    const int64_t a0 = off[v], a1 = off[v + 1];
    float x = 0.f, y = 0.f, z = 0.f;
    for (int64_t o = a0; o < a1; ++o) {
      const float4 t = t32[obs_scan[o]];
      x += t.x;
      y += t.y;
      z += t.z;
    }
    const float inv = 1.0f / (float)(a1 - a0);
    const float m[3] = {x * inv, y * inv, z * inv};
    mean[v] = make_float4(m[0], m[1], m[2], 0.f);
    for (int c = 0; c < 3; ++c) {
      atomicMin(&sbox[c], float_order_key(m[c]));
      atomicMax(&sbox[3 + c], float_order_key(m[c]));
    }
  }
  __syncthreads();
  if (threadIdx.x < 3) atomicMin(&box[threadIdx.x], sbox[threadIdx.x]);
  else if (threadIdx.x < 6) atomicMax(&box[threadIdx.x], sbox[threadIdx.x]);
}

// 10 bits of each coordinate spread to every third bit
__device__ __forceinline__ uint32_t spread3(uint32_t v) {
  v &= 0x3ffu;
  v = (v | (v << 16)) & 0x030000ffu;
  v = (v | (v << 8)) & 0x0300f00fu;
  v = (v | (v << 4)) & 0x030c30c3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

__global__ void morton_keys_kernel(const float4* mean, int64_t n_voxels, const uint32_t* box,
                                   uint32_t* keys) {
  grid_wait();
  grid_launch_next();
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n_voxels) return;
  const float4 m = mean[v];
  const float mc[3] = {m.x, m.y, m.z};
  uint32_t code = 0;
  for (int c = 0; c < 3; ++c) {
    const float lo = float_from_order_key(box[c]), hi = float_from_order_key(box[3 + c]);
    uint32_t q = 0;
    if (hi > lo) {
      const float t = (mc[c] - lo) / (hi - lo) * 1023.0f;
      q = t <= 0.f ? 0u : t >= 1023.f ? 1023u : (uint32_t)t;
    }
    code |= spread3(q) << c;
  }
  keys[v] = code;
}

// after the spatial sort (vals[r] = voxel of spatial rank r): window of the
// rank, then length descending
__global__ void window_keys_kernel(const int64_t* off, const uint32_t* vals,
                                   int64_t n_voxels, int max_len, int len_bits, uint32_t* keys) {
  grid_wait();
  grid_launch_next();
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n_voxels) return;
  const uint32_t v = vals[r];
  const int64_t len = off[v + 1] - off[v];
  keys[r] = ((uint32_t)(r / kWindow) << len_bits) | (uint32_t)(max_len - len);
}

__global__ void slice_len_kernel(const int64_t* off, const uint32_t* vperm, int64_t n_voxels, int64_t n_slices,
                                 int64_t* slice_off, int32_t* vlen, int32_t* vperm_out, int32_t* vrank) {
  grid_wait();
  grid_launch_next();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n_voxels) {
    const uint32_t v = vperm[p];
    const int32_t len = (int32_t)(off[v + 1] - off[v]);
    vlen[p] = len;
    vperm_out[p] = (int32_t)v;
    vrank[v] = (int32_t)p;
    if ((p & 31) == 0) slice_off[p >> 5] = (int64_t)kSlice * len;  // first voxel is the longest of its slice
  }
  if (p == 0) slice_off[n_slices] = 0;
}

// FP64 slots: thread (p, blockIdx.y) fills rows blockIdx.y, blockIdx.y + gridDim.y
// .. of the voxel at sorted position p.  Bound by the factorisation's FP64
// divisions; a thread for all rows of a voxel left most of the chip idle (50,000
// voxels, 1.2M clusters 380 us; a thread per row 165 us).
__global__ void fill_sell_kernel(LoadInput in, const int32_t* vperm, const int32_t* vlen, const int64_t* slice_off,
                                 int64_t n_voxels, double* ve, int32_t* ve_scan, int64_t n_elems) {
  grid_wait();
  grid_launch_next();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t s = p >> 5;
  if (s * kSlice >= n_voxels) return;
  const int lane = (int)(p & 31);
  const int64_t base = slice_off[s] + lane;
  const int64_t rows = (slice_off[s + 1] - slice_off[s]) / kSlice;
  const bool real = p < n_voxels;
  const int32_t len = real ? vlen[p] : 0;
  const int64_t o0 = real ? in.voxel_off[vperm[p]] : 0;
  for (int64_t k = blockIdx.y; k < rows; k += gridDim.y) {
    const int64_t e = base + k * kSlice;
    double c[10], f[10];
    uint32_t scan = 0;
    if (k < len) {
      to_centred(in.agg + 10 * (o0 + k), in.agg_form, c);
      // the scatter as its pivoted LDL^T, the mean permuted alike
      const uint32_t code = ldlt3_pivoted(c, f);
      int p0, p1, p2;
      perm_decode(code, p0, p1, p2);
      f[6] = c[6 + p0];
      f[7] = c[6 + p1];
      f[8] = c[6 + p2];
      f[9] = c[9];
      scan = (uint32_t)in.obs_scan[o0 + k] | (code << kPermShift);
    } else {
#pragma unroll
      for (int q = 0; q < 10; ++q) f[q] = 0.0;
    }
#pragma unroll
    for (int q = 0; q < 10; ++q) ve[q * n_elems + e] = f[q];
    ve_scan[e] = (int32_t)scan;
  }
}

// The voxel of every observation of voxels [v0, v1) (unless obs_vox is null), and
// each voxel's 2 / N_i (unless vscale is null), kVoxelLanes threads to a voxel:
// a voxel's rows are then read together (15M clusters 268 us as a thread per
// voxel, 184 us).
constexpr int kVoxelLanes = 8;
__global__ void __launch_bounds__(256) obs_voxel_kernel(LoadInput in, int64_t v0, int64_t v1, int32_t* obs_vox,
                                                        double* vscale) {
  grid_wait();
  grid_launch_next();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t v = v0 + t / kVoxelLanes;
  const int sub = (int)(t % kVoxelLanes);
  if (v >= v1) return;  // whole groups leave together
  const unsigned mask = ((1u << kVoxelLanes) - 1u) << (threadIdx.x & 31 & ~(kVoxelLanes - 1));
  double n = 0.0;
  const int64_t b = in.voxel_off[v + 1];
  for (int64_t o = in.voxel_off[v] + sub; o < b; o += kVoxelLanes) {
    if (obs_vox) obs_vox[o] = (int32_t)v;
    if (vscale) n += in.agg[10 * o + 9];
  }
  if (!vscale) return;
#pragma unroll
  for (int o = 1; o < kVoxelLanes; o <<= 1) n += __shfl_xor_sync(mask, n, o);
  if (sub == 0) vscale[v] = 2.0 / n;
}

// observations listed by sorted voxel position (pbase[p] = observations of
// the voxels before position p), keyed by scan for the stable sort that makes
// the scan-major copy: inside a scan, observations follow the voxel order, so
// the scan pass gathers the plane records of nearby voxels
// (and, unless place is null, each observation's sorted voxel position and row)
__global__ void scan_keys_kernel(LoadInput in, const int32_t* obs_vox, const int32_t* vrank, const int64_t* pbase,
                                 uint32_t* keys, uint32_t* vals, int2* place) {
  grid_wait();
  grid_launch_next();
  const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= in.n_obs) return;
  const int32_t v = obs_vox[o];
  const int32_t p = vrank[v];
  const int32_t row = (int32_t)(o - in.voxel_off[v]);
  const int64_t q = pbase[p] + row;
  keys[q] = (uint32_t)in.obs_scan[o];
  vals[q] = (uint32_t)o;
  if (place) place[o] = make_int2(p, row);
}

// scan_off[j] = the first scan-major position of scan j (n at the end), from
// the scan ids sorted ascending: position q starts every scan after its
// predecessor's id up to its own (scans with no observation included), so
// each entry is written once
__global__ void scan_off_kernel(const uint32_t* keys, int64_t n, int32_t n_scans, int64_t* scan_off) {
  grid_wait();
  grid_launch_next();
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q > n) return;
  const int64_t lo = q == 0 ? 0 : (int64_t)keys[q - 1] + 1;
  const int64_t hi = q == n ? (int64_t)n_scans : (int64_t)keys[q];
  for (int64_t j = lo; j <= hi; ++j) scan_off[j] = q;
}

__global__ void vlen_i64_kernel(const int32_t* vlen, int64_t n_voxels, int64_t* out) {
  grid_wait();
  grid_launch_next();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n_voxels) out[p] = vlen[p];
  if (p == 0) out[n_voxels] = 0;
}

__global__ void fill_scan_major_kernel(LoadInput in, const uint32_t* order, const int32_t* obs_vox,
                                       const double* vscale, const int32_t* vrank, double* se, int32_t* se_vox) {
  grid_wait();
  grid_launch_next();
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= in.n_obs) return;
  const int64_t o = order[q];
  const int32_t v = obs_vox[o];
  se_vox[q] = vrank[v];
  double c[10];
  to_centred(in.agg + 10 * o, in.agg_form, c);
  const double k = vscale[v];
#pragma unroll
  for (int a = 0; a < 6; ++a) c[a] *= k;
  c[9] *= k;
  const int64_t n = in.n_obs;
#pragma unroll
  for (int a = 0; a < 10; ++a) se[a * n + q] = c[a];
}

// chunk index of each scan-major position's observation (its place among
// the chunk bounds), keyed for a stable one-digit partition
__global__ void chunk_keys_kernel(const uint32_t* order, int64_t n, ChunkBounds cb, uint32_t* keys) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  const int64_t o = order[q];
  uint32_t c = 0;
  for (int k = 1; k < cb.n; ++k) c += o >= cb.o[k] ? 1u : 0u;
  keys[q] = c;
}

static int bit_width(uint64_t x) {
  int b = 0;
  while (x) {
    ++b;
    x >>= 1;
  }
  return b;
}

static cudaError_t launch_obs_voxel(const LoadInput& in, int64_t v0, int64_t v1, int32_t* obs_vox, double* vscale,
                                    cudaStream_t stream, int64_t* launches) {
  if (v1 <= v0) return cudaSuccess;
  launch_chained(obs_voxel_kernel, (unsigned)(((v1 - v0) * kVoxelLanes + 255) / 256), 256, 0, stream, in, v0, v1,
                 obs_vox, vscale);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_vscale(const LoadInput& in, int64_t v0, int64_t v1, double* vscale, cudaStream_t stream,
                          int64_t* launches) {
  return launch_obs_voxel(in, v0, v1, nullptr, vscale, stream, launches);
}

cudaError_t group_by_chunk(const uint32_t* order, int64_t n_obs, const ChunkBounds& cb, const uint32_t** out_q,
                           Allocator temp, cudaStream_t stream, int64_t* launches) {
  if (n_obs <= 0) return cudaSuccess;
  if (cb.n < 1 || cb.n > kMaxCopyChunks) return cudaErrorInvalidValue;
  uint32_t* keys = (uint32_t*)temp.fn(temp.self, sizeof(uint32_t) * n_obs);
  uint32_t* vals = (uint32_t*)temp.fn(temp.self, sizeof(uint32_t) * n_obs);
  uint32_t* tk = (uint32_t*)temp.fn(temp.self, sizeof(uint32_t) * n_obs);
  uint32_t* tv = (uint32_t*)temp.fn(temp.self, sizeof(uint32_t) * n_obs);
  int64_t* scratch = (int64_t*)temp.fn(temp.self, sizeof(int64_t) * radix_scratch_count(n_obs));
  if (!keys || !vals || !tk || !tv || !scratch) return cudaErrorMemoryAllocation;
  chunk_keys_kernel<<<(unsigned)((n_obs + 255) / 256), 256, 0, stream>>>(order, n_obs, cb, keys);
  ++*launches;
  RETURN_IF(cudaGetLastError());
  RETURN_IF(radix_sort_pairs(&keys, &vals, &tk, &tv, n_obs, bit_width((uint64_t)(cb.n - 1)), true, scratch, stream,
                             launches));
  *out_q = vals;
  return cudaSuccess;
}

// Scans by decreasing observation count, ties by index.  Up to kRankScans, eight
// lanes count the scans before one (1000 scans: 5 us, a thread per scan in one
// block 30 us); beyond, the general sort of n_obs - count.
constexpr int kRankScans = 1024, kRankThreads = 256, kRankLanes = 8;
__global__ void __launch_bounds__(kRankThreads) scan_rank_kernel(const int64_t* scan_off, int n, int32_t* order) {
  grid_wait();
  grid_launch_next();
  __shared__ __align__(16) uint32_t len[kRankScans];
  for (int i = threadIdx.x; i < (n + 3) / 4 * 4; i += kRankThreads)
    len[i] = i < n ? (uint32_t)(scan_off[i + 1] - scan_off[i]) : 0u;
  __syncthreads();
  const int t = blockIdx.x * kRankThreads + threadIdx.x, j = t / kRankLanes;
  const uint32_t mine = len[j < n ? j : 0];
  int rank = 0;  // the padding's 0 is longer than none, and after all
  for (int i = 4 * (t % kRankLanes); i < n; i += 4 * kRankLanes) {
    const uint4 v = *reinterpret_cast<const uint4*>(len + i);
    rank += (v.x > mine || (v.x == mine && i < j)) + (v.y > mine || (v.y == mine && i + 1 < j)) +
            (v.z > mine || (v.z == mine && i + 2 < j)) + (v.w > mine || (v.w == mine && i + 3 < j));
  }
#pragma unroll
  for (int o = kRankLanes / 2; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
  if (j < n && t % kRankLanes == 0) order[rank] = j;
}

__global__ void scan_len_keys_kernel(const int64_t* scan_off, int32_t n_scans, int64_t n_obs, uint32_t* keys) {
  grid_wait();
  grid_launch_next();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n_scans) keys[j] = (uint32_t)(n_obs - (scan_off[j + 1] - scan_off[j]));
}

cudaError_t build_layout(const LoadInput& in, const float4* t32, uint32_t* box, int max_len, bool fill_f64,
                         bool defer_scale, Allocator keep, Allocator temp, LayoutBuffers* out, cudaStream_t stream,
                         int64_t* launches) {
  const int64_t nv = in.n_voxels, no = in.n_obs;
  const int64_t n_slices = (nv + kSlice - 1) / kSlice, n_windows = (nv + kWindow - 1) / kWindow;
  const int64_t nsort = std::max(std::max(nv, no), (int64_t)in.n_scans);
  const int scan_bits = bit_width((uint64_t)(in.n_scans - 1));
  // Slots of all slices.  Within a window the lengths decrease, so each slice's
  // padding is at most 32 x (its longest - the next slice's longest) and a
  // window's at most 32 x max_len: where that bound keeps the slots within the
  // estimate's share (an eighth more than the observations) it stands for their
  // number, and the host need not wait for the prefix sum; else the sum is read.
  const int64_t elem_bound = (no + n_windows * kSlice * (int64_t)max_len + kSlice - 1) / kSlice * kSlice;
  const bool bounded = elem_bound <= no + no / 8 + 64;
  uint32_t *keys, *vals, *tk, *tv;
  int64_t *scratch, *pscratch, *pbase;
  int32_t *vrank, *obs_vox;
  int2* place = nullptr;
  double* vscale;
  uint32_t* order = nullptr;
  float4* mean;
  {
    ArrayGroup t, k;
    // the maps are kept when the FP32 copies will be rebuilt later, the
    // prefixes by a load that stages its slots (they are staged in this order)
    ArrayGroup& maps = fill_f64 ? t : k;
    t.add(&keys, nsort);
    t.add(&vals, nsort);
    t.add(&tk, nsort);
    t.add(&tv, nsort);
    t.add(&scratch, radix_scratch_count(nsort) + scan_scratch_count(n_slices + no + 2));
    t.add(&pscratch, scan_scratch_count(nv + 1));
    t.add(&obs_vox, no);
    t.add(&mean, nv);
    maps.add(&vrank, nv);
    maps.add(&vscale, nv);
    (defer_scale ? k : t).add(&pbase, nv + 1);
    if (!fill_f64) {
      k.add(&place, no);
      k.add(&order, no);
    }
    k.add(&out->slice_off, n_slices + 1);
    k.add(&out->vlen, nv);
    k.add(&out->vperm, nv);
    k.add(&out->scan_off, in.n_scans + 1);
    k.add(&out->scans_by_len, in.n_scans);
    if (fill_f64) k.add(&out->se, 10 * no);
    // + 4 entries: the staged mixed scan pass copies whole 16-byte groups
    k.add(&out->se_vox, no + 4);
    if (fill_f64 && bounded) {
      k.add(&out->ve, 10 * elem_bound);
      k.add(&out->ve_scan, elem_bound);
    }
    if (!t.allocate(temp) || !k.allocate(keep)) return cudaErrorMemoryAllocation;
  }
  out->vrank = vrank;
  out->place = place;
  out->vscale = vscale;
  out->scan_order = order;

  // ---- voxel order: spatial windows, length-descending inside each ----
  const int len_bits = bit_width((uint64_t)max_len);
  const int win_bits = bit_width((uint64_t)((nv - 1) / kWindow));
  if (len_bits + win_bits > 32) return cudaErrorInvalidValue;
  {
    const unsigned nb = (unsigned)((nv + 255) / 256);
    launch_chained(observer_mean_kernel, nb, 256, 0, stream, in.voxel_off, in.obs_scan, t32, nv, mean, box);
    launch_chained(morton_keys_kernel, nb, 256, 0, stream, mean, nv, box, keys);
    *launches += 2;
    RETURN_IF(cudaGetLastError());
    RETURN_IF(radix_sort_pairs(&keys, &vals, &tk, &tv, nv, 30, true, scratch, stream, launches));
    launch_chained(window_keys_kernel, nb, 256, 0, stream, in.voxel_off, vals, nv, max_len, len_bits, keys);
    ++*launches;
    RETURN_IF(cudaGetLastError());
  }
  RETURN_IF(radix_sort_pairs(&keys, &vals, &tk, &tv, nv, len_bits + win_bits, false, scratch, stream, launches));
  launch_chained(slice_len_kernel, (unsigned)((nv + 255) / 256), 256, 0, stream, in.voxel_off, vals, nv, n_slices,
                                                                     out->slice_off, out->vlen, out->vperm, vrank);
  ++*launches;
  RETURN_IF(cudaGetLastError());
  RETURN_IF(exclusive_scan_i64(out->slice_off, n_slices + 1, scratch, stream, launches));
  int64_t n_elems = elem_bound;
  if (!bounded) {
    RETURN_IF(cudaMemcpyAsync(&n_elems, out->slice_off + n_slices, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
    RETURN_IF(cudaStreamSynchronize(stream));
  }
  out->n_elems = n_elems;
  out->n_slices = n_slices;
  out->max_len = max_len;
  // the FP64 slice copy (the mixed path builds its own FP32 slots)
  if (fill_f64) {
    if (!bounded) {
      ArrayGroup k;
      k.add(&out->ve, 10 * n_elems);
      k.add(&out->ve_scan, n_elems);
      if (!k.allocate(keep)) return cudaErrorMemoryAllocation;
    }
    // rows over blockIdx.y: enough for voxels of four times the mean length, the
    // rest of a longer one in further turns
    const unsigned row_blocks = (unsigned)std::min<int64_t>(std::min<int64_t>(max_len, 4 * (no / nv) + 4), 65535);
    launch_chained(fill_sell_kernel, dim3((unsigned)((n_slices * kSlice + 255) / 256), row_blocks), 256, 0, stream, in,
                   out->vperm, out->vlen, out->slice_off, nv, out->ve, out->ve_scan, n_elems);
    ++*launches;
    RETURN_IF(cudaGetLastError());
  }

  // ---- scan-major copy ----
  RETURN_IF(launch_obs_voxel(in, 0, nv, obs_vox, defer_scale ? nullptr : vscale, stream, launches));
  {
    launch_chained(vlen_i64_kernel, (unsigned)((nv + 255) / 256), 256, 0, stream, out->vlen, nv, pbase);
    ++*launches;
    RETURN_IF(cudaGetLastError());
    RETURN_IF(exclusive_scan_i64(pbase, nv + 1, pscratch, stream, launches));
    out->vstart = defer_scale ? pbase : nullptr;
    // the order, where it is kept, lands in its own buffer: the sort ends in the
    // buffer it starts from after an even number of passes, else in the other
    if (order) (radix_passes(no, scan_bits) % 2 == 0 ? vals : tv) = order;
    launch_chained(scan_keys_kernel, (unsigned)((no + 255) / 256), 256, 0, stream, in, obs_vox, vrank, pbase, keys,
                   vals, place);
    ++*launches;
    RETURN_IF(cudaGetLastError());
  }
  RETURN_IF(radix_sort_pairs(&keys, &vals, &tk, &tv, no, scan_bits, false, scratch, stream, launches));
  launch_chained(scan_off_kernel, (unsigned)((no + 1 + 255) / 256), 256, 0, stream, keys, no, in.n_scans,
                 out->scan_off);
  ++*launches;
  RETURN_IF(cudaGetLastError());
  if (fill_f64) {  // the mixed path fills its own copy, se_vox included
    launch_chained(fill_scan_major_kernel, (unsigned)((no + 255) / 256), 256, 0, stream, in, vals, obs_vox, vscale,
                   vrank, out->se, out->se_vox);
    ++*launches;
    RETURN_IF(cudaGetLastError());
  }
  // ---- scan-pass block order, so the longest scans start first ----
  if (in.n_scans <= kRankScans) {
    launch_chained(scan_rank_kernel, (unsigned)(((int64_t)in.n_scans * kRankLanes + kRankThreads - 1) / kRankThreads),
                   kRankThreads, 0, stream, out->scan_off, in.n_scans, out->scans_by_len);
    ++*launches;
    return cudaGetLastError();
  }
  const int len_digits = bit_width((uint64_t)no);
  uint32_t* by_len = (uint32_t*)out->scans_by_len;
  uint32_t* other = tv;  // free: the scan-major order is in vals
  launch_chained(scan_len_keys_kernel, (unsigned)((in.n_scans + 255) / 256), 256, 0, stream, out->scan_off, in.n_scans,
                 no, keys);
  ++*launches;
  RETURN_IF(cudaGetLastError());
  if (radix_passes(in.n_scans, len_digits) % 2 != 0) std::swap(by_len, other);
  RETURN_IF(radix_sort_pairs(&keys, &by_len, &tk, &other, in.n_scans, len_digits, true, scratch, stream, launches));
  return cudaSuccess;
}

// ============================================================================
// Point clusters (Eq. 2) in centred form: two lanes per observation (sixteen
// observations per warp; the pair reads neighbouring points, so a sector's
// three coordinates come from one fetch), one pass over the points as sums
// shifted by the observation's first point p0: with d = p - p0,
//   m = p0 + (sum d) / N,   S = sum d d^T - (sum d)(sum d)^T / N,
// algebraically the mean and the scatter about it (Eq. 2 fixes the sums, not
// their order).
//
// The sums are exact integer sums in fixed point.  An observation's scale is
// 2^-F with F = 1076 - E0, E0 the largest biased binary exponent of p0's
// coordinates: half the last bit of p0's largest coordinate.  Every coordinate
// of that size or larger (up to 2^9 times) is an exact integer multiple of
// 2^-F, and smaller ones are rounded to it (an error below half the last bit
// of p0's largest coordinate, the resolution of FP64 arithmetic on these
// points).  d, sum d and sum d d^T are then 64- and 128-bit integer sums with
// no rounding at all, on the integer pipe; GB300's FP64 pipe (1/64 of FP32)
// only forms m and S once per observation.  An observation whose points do not
// fit (a coordinate over 2^9 times p0's largest, a spread over 2^56 steps,
// more than 2^14 points, a first point at the origin, or a scale outside
// 2^-400 .. 2^400) takes the same shifted sums in FP64.
//
// Points within 2^54 steps of the first (two metres at one metre's range, 128
// m at 100 m) take d split at 27 bits into two 32-bit halves, each product of
// halves in a 64-bit sum of its own, one multiply-add each: 21 a point instead
// of six 128-bit multiply-adds.  The bounds: both halves are below 2^27 in
// size, a pair of cross products is below 2^55, and 254 of those below 2^63,
// the lanes' sums added; longer observations are joined 254 points at a time.
//
// A block takes 256 observations (128 in a small call) in order of their lengths,
// so that the sixteen of a warp are about as long (a warp runs as long as its
// longest), and each
// lane has its next two points on their way while it sums one.
//
// Bound: instruction issue (0.56 a cycle; ~176 instructions a point, ~1,400 a
// warp for the sixteen records) and the loads' latency at 16 warps an SM.
// Measured, before (128-bit sums, observations in input order) and now:
// 0.6M observations of 1-64 points 576 -> 265 us, 1M of 32 454 -> 386 us, 0.2M of
// 100 319 -> 222 us, 3M of 1-8 614 -> 586 us, 60,000 of 200-400 645 -> 267 us.
constexpr int kAggLanes = 2;

// the shifted sums in FP64 (observations the fixed point does not fit)
__device__ void aggregate_f64(int64_t a, int64_t b, int sub, unsigned mask, const double* __restrict__ pts,
                              double* __restrict__ r) {
  const double p0x = pts[3 * a], p0y = pts[3 * a + 1], p0z = pts[3 * a + 2];
  double sx = 0.0, sy = 0.0, sz = 0.0;
  double c00 = 0.0, c01 = 0.0, c02 = 0.0, c11 = 0.0, c12 = 0.0, c22 = 0.0;
  for (int64_t k = a + sub; k < b; k += kAggLanes) {
    const double x = pts[3 * k] - p0x, y = pts[3 * k + 1] - p0y, z = pts[3 * k + 2] - p0z;
    sx += x;
    sy += y;
    sz += z;
    c00 = fma(x, x, c00);
    c01 = fma(x, y, c01);
    c02 = fma(x, z, c02);
    c11 = fma(y, y, c11);
    c12 = fma(y, z, c12);
    c22 = fma(z, z, c22);
  }
  double* sums[9] = {&sx, &sy, &sz, &c00, &c01, &c02, &c11, &c12, &c22};
#pragma unroll
  for (int o = 1; o < kAggLanes; o <<= 1)
#pragma unroll
    for (int q = 0; q < 9; ++q) *sums[q] += __shfl_xor_sync(mask, *sums[q], o);
  const double n = (double)(b - a);
  const double rn = 1.0 / n;
  const double dx = sx * rn, dy = sy * rn, dz = sz * rn;
  if (sub == 0) {
    r[0] = fma(-sx, dx, c00);
    r[1] = fma(-sx, dy, c01);
    r[2] = fma(-sx, dz, c02);
    r[3] = fma(-sy, dy, c11);
    r[4] = fma(-sy, dz, c12);
  } else if (sub == 1) {
    r[5] = fma(-sz, dz, c22);
    r[6] = p0x + dx;
    r[7] = p0y + dy;
    r[8] = p0z + dz;
    r[9] = n;
  }
}

// one observation by a pair of lanes (sub = 0, 1; mask = the pair's lanes;
// totals: five values of this thread's, kOrderBlock apart)
__device__ __forceinline__ void aggregate_one(int64_t a, int64_t b, int sub, unsigned mask,
                                              const double* __restrict__ pts, double* __restrict__ r,
                                              __int128* totals) {
  if (b <= a) {
    for (int k = sub; k < 10; k += kAggLanes) r[k] = 0.0;
    return;
  }
  const double p0x = pts[3 * a], p0y = pts[3 * a + 1], p0z = pts[3 * a + 2];
  int E0 = (__double2hiint(p0x) >> 20) & 0x7ff;
  E0 = max(E0, (__double2hiint(p0y) >> 20) & 0x7ff);
  E0 = max(E0, (__double2hiint(p0z) >> 20) & 0x7ff);
  const int F = 1076 - E0;
  bool fits = E0 != 0 && F >= -400 && F <= 400 && b - a <= (1 << 14);
  const long long X0x = fix_round(p0x, F, fits), X0y = fix_round(p0y, F, fits), X0z = fix_round(p0z, F, fits);
  // lane 0 ends with S xx, xy, xz, yy in u[0 .. 3], lane 1 with S yz, zz and
  // sum d in u[0 .. 4], all exact
  __int128 u[5] = {0, 0, 0, 0, 0};
  bool ok = fits;
#pragma unroll 1
  for (int64_t a1 = a; ok && a1 < b; a1 += kHalfPoints) {
    HalfSums h;
    h.clear();
    const double* q = pts + 3 * (a1 + sub);
    const int n1 = (int)(b - a1 < kHalfPoints ? b - a1 : kHalfPoints);
    const int cnt = (n1 - sub + kAggLanes - 1) / kAggLanes;  // points of this lane
    const int sh = 1075 - F;
    int emax = -2048;
    unsigned wide = 0;
    auto add = [&](double x, double y, double z) {
      const long long dx = fix_offset(x, sh, X0x, emax, wide);
      const long long dy = fix_offset(y, sh, X0y, emax, wide);
      const long long dz = fix_offset(z, sh, X0z, emax, wide);
      h.add(dx, dy, dz);
    };
    double ax = p0x, ay = p0y, az = p0z, bx = p0x, by = p0y, bz = p0z;
    if (cnt > 0) {
      ax = q[0];
      ay = q[1];
      az = q[2];
    }
    if (cnt > 1) {
      bx = q[3 * kAggLanes];
      by = q[3 * kAggLanes + 1];
      bz = q[3 * kAggLanes + 2];
    }
    for (int k = 0; k < cnt; k += 2) {
      q += 6 * kAggLanes;
      {
        const double x = ax, y = ay, z = az;
        if (k + 2 < cnt) {
          ax = q[0];
          ay = q[1];
          az = q[2];
        }
        add(x, y, z);
      }
      if (k + 1 < cnt) {
        const double x = bx, y = by, z = bz;
        if (k + 3 < cnt) {
          bx = q[3 * kAggLanes];
          by = q[3 * kAggLanes + 1];
          bz = q[3 * kAggLanes + 2];
        }
        add(x, y, z);
      }
    }
    // every coordinate within 2^9 of p0's largest, every offset below 2^54
    ok = __all_sync(mask, emax <= 9 && (wide >> 22) == 0u);
    // lane 0 takes the pair's first 12 sums, lane 1 the other 9
    long long w[12];
    const bool up = sub != 0;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const long long hi = k < 9 ? h.v[k + 12 < 21 ? k + 12 : 20] : 0;
      w[k] = (up ? hi : h.v[k]) + __shfl_xor_sync(mask, up ? h.v[k] : hi, 1);
    }
    u[0] = join_halves(w[0], w[1], up ? 27 : 28, w[2]);  // yz or xx
    u[1] = join_halves(w[3], w[4], up ? 28 : 27, w[5]);  // zz or xy
    u[2] = up ? (__int128)w[6] : join_halves(w[6], w[7], 27, w[8]);
    u[3] = up ? (__int128)w[7] : join_halves(w[9], w[10], 28, w[11]);
    u[4] = w[8];  // (lane 1)
    if (b - a > kHalfPoints) {  // the sums so far wait in shared memory, not in registers
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        if (a1 > a) u[k] += totals[k * kOrderBlock];
        totals[k * kOrderBlock] = u[k];
      }
    }
  }
  if (!ok) {  // wide observations: 128-bit sums, or FP64
    ok = fits;
    constexpr long long kMaxD = 1ll << 56;
    __int128 t[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t k = a + sub; k < b && ok; k += kAggLanes) {
      const long long dx = fix_round(pts[3 * k], F, ok) - X0x;
      const long long dy = fix_round(pts[3 * k + 1], F, ok) - X0y;
      const long long dz = fix_round(pts[3 * k + 2], F, ok) - X0z;
      ok = ok && dx > -kMaxD && dx < kMaxD && dy > -kMaxD && dy < kMaxD && dz > -kMaxD && dz < kMaxD;
      t[0] += (__int128)dx * dx;
      t[1] += (__int128)dx * dy;
      t[2] += (__int128)dx * dz;
      t[3] += (__int128)dy * dy;
      t[4] += (__int128)dy * dz;
      t[5] += (__int128)dz * dz;
      t[6] += dx;
      t[7] += dy;
      t[8] += dz;
    }
    if (!__all_sync(mask, ok)) {
      aggregate_f64(a, b, sub, mask, pts, r);
      return;
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) t[q] += shfl_xor_i128(mask, t[q], 1);
#pragma unroll
    for (int q = 0; q < 5; ++q) u[q] = sub == 0 ? t[q] : t[4 + q];
  }
  // S = C - s_a d_b and m = p0 + d from the exact sums, one instruction
  // sequence with operands chosen per lane (an FP64 warp instruction costs the
  // same whatever the number of lanes on each side of a branch)
  const bool up = sub != 0;
  const int e2 = up ? -F : -2 * F;
  double c[5] = {i128_scaled(u[0], -2 * F), i128_scaled(u[1], -2 * F), i128_scaled(u[2], e2), i128_scaled(u[3], e2), 0.0};
  // sum d is below 2^56 2^14: slot 4 of lane 1 may need 128 bits
  const int lane0 = threadIdx.x & 30;
  if (up) c[4] = i128_scaled(u[4], -F);
  const double sx = __shfl_sync(mask, c[2], lane0 + 1), sy = __shfl_sync(mask, c[3], lane0 + 1),
               sz = __shfl_sync(mask, c[4], lane0 + 1);
  // p0 in whole steps: x by lane 0, y by lane 1, then z
  const double xy = i64_scaled(up ? X0y : X0x, -F), mx0 = __shfl_sync(mask, xy, lane0), mz0 = i64_scaled(X0z, -F);
  if (up) {
    c[2] = mx0;
    c[3] = xy;
    c[4] = mz0;
  }
  const float nf = (float)(int)(b - a);
  const double n = f32_to_f64(nf);
  const double rn = recip_count(n, nf);
  const double dx = sx * rn, dy = sy * rn, dz = sz * rn;
  double* w = r + (up ? 4 : 0);
  w[0] = fma(up ? -sy : -sx, up ? dz : dx, c[0]);  // yz or xx
  w[1] = fma(up ? -sz : -sx, up ? dz : dy, c[1]);  // zz or xy
  w[2] = fma(up ? 1.0 : -sx, up ? dx : dz, c[2]);  // m x or xz
  w[3] = fma(up ? 1.0 : -sy, dy, c[3]);            // m y or yy
  if (up) {
    w[4] = c[4] + dz;
    w[5] = n;
  }
}

// kRounds: times a block's pairs of lanes take an observation each (of 128
// kRounds observations in order of length).
template <int kRounds>
__global__ void __launch_bounds__(kOrderBlock, 2)
    aggregate_points_kernel(int64_t n_obs, const int64_t* __restrict__ off, const double* __restrict__ pts,
                            double* __restrict__ out) {
  constexpr int kGroups = kOrderBlock / kAggLanes, kItems = kGroups * kRounds;
  static_assert(kItems <= kOrderBlock, "the ordering takes one observation per thread");
  __shared__ int s_cnt[32], s_order[kOrderBlock];
  __shared__ __int128 s_totals[5 * kOrderBlock];
  const int64_t o0 = (int64_t)blockIdx.x * kItems;
  {
    // the threads past the block's observations come last
    const int64_t o = o0 + threadIdx.x;
    const int64_t len = threadIdx.x < kItems && o < n_obs ? off[o + 1] - off[o] : 0;
    const int key = len < 0 ? 0 : len < 120 ? (int)(len >> 2) : 30;
    block_order_by_key(threadIdx.x < kItems ? key : 31, s_cnt, s_order);
  }
  const int sub = threadIdx.x & (kAggLanes - 1), group = threadIdx.x / kAggLanes;
  const unsigned mask = ((1u << kAggLanes) - 1u) << (threadIdx.x & 31 & ~(kAggLanes - 1));
#pragma unroll 1
  for (int round = 0; round < kRounds; ++round) {
    // every second round from the other end, so that every warp takes short and long ones
    const int64_t o = o0 + s_order[kGroups * round + (round & 1 ? kGroups - 1 - group : group)];
    if (o < n_obs) aggregate_one(off[o], off[o + 1], sub, mask, pts, out + 10 * o, s_totals + threadIdx.x);
  }
}

// One round while that is at most one wave (two blocks an SM), so that half of
// the chip does not idle for the others' second round: us a call with one / two
// rounds, 1,000 observations of 8 points 9.6 / 13.7, of 100 23.8 / 42.5, 20,000
// of 300 108 / 139.
constexpr int64_t kOneRoundObs = 2 * kSMs * (kOrderBlock / kAggLanes);

cudaError_t launch_aggregate_points(int64_t n_obs, const int64_t* point_off, const double* points, double* agg_out,
                                    cudaStream_t stream) {
  if (n_obs <= 0) return cudaSuccess;
  const int rounds = n_obs <= kOneRoundObs ? 1 : kAggLanes;
  const int64_t per = rounds * (kOrderBlock / kAggLanes);
  const auto kernel = rounds == 1 ? aggregate_points_kernel<1> : aggregate_points_kernel<kAggLanes>;
  kernel<<<(unsigned)((n_obs + per - 1) / per), kOrderBlock, 0, stream>>>(n_obs, point_off, points, agg_out);
  return cudaGetLastError();
}

}  // namespace mmba
