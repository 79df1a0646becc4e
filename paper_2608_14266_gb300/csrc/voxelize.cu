// Preprocessing on the device (Sec. IV-B, Algorithm 1): L1 voxelisation of
// raw scans (Eq. 4), bottom-up voxel levels (Eq. 5, BottomUpVoxelization),
// selection by planarity (Selection), and the voxel-major observation list
// that ba_load_observations takes.
//
// Order of the output (shared with the CPU reference of the tests): voxels by
// level, then by integer index (x, y, z); the observations of a voxel by scan.
// Indices are exactly floor(RN(w / d)) with w formed by explicit fma, so the
// integer structure does not depend on the compiler's choices.  GB300 runs
// FP64 on a narrow pipe: indices are formed in fixed point, with FP64 near voxel
// faces only, the sums of a cluster's points are exact integer sums, and the
// planarity test runs in FP32 unless it is too close to call.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <condition_variable>
#include <mutex>
#include <thread>
#include <type_traits>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <string>
#include <vector>

#include "../../include/ba.h"
#include "block_order.cuh"
#include "fixed_sums.cuh"
#include "mmba_internal.cuh"
#include "mmba_kernels.h"

using namespace mmba;

namespace {

constexpr int kKeyRange = 1 << 20;  // indices in [-2^20, 2^20) per axis

// Voxel keys: the index of each axis offset by its smallest value at this
// level and packed x | y | z with just the bits the level's index range needs,
// so that sorting keys sorts voxels by (x, y, z) and the radix sort runs as
// few digit passes as possible.  Level k+1 (Eq. 5) halves the range per axis.
struct KeyPack {
  int lo[3];  // smallest index per axis
  int w[3];   // bits per axis
};

__host__ __device__ __forceinline__ uint64_t pack_key(const KeyPack& p, int ix, int iy, int iz) {
  return ((uint64_t)(unsigned)(ix - p.lo[0]) << (p.w[1] + p.w[2])) | ((uint64_t)(unsigned)(iy - p.lo[1]) << p.w[2]) |
         (uint64_t)(unsigned)(iz - p.lo[2]);
}

__host__ __device__ __forceinline__ void unpack_key(const KeyPack& p, uint64_t k, int* i) {
  i[2] = (int)(k & ((1ull << p.w[2]) - 1ull)) + p.lo[2];
  i[1] = (int)((k >> p.w[2]) & ((1ull << p.w[1]) - 1ull)) + p.lo[1];
  i[0] = (int)(k >> (p.w[1] + p.w[2])) + p.lo[0];
}

// the raw level-1 key before the index range is known: 21 bits per axis
__device__ __forceinline__ uint64_t raw_key(int ix, int iy, int iz) {
  return ((uint64_t)(ix + kKeyRange) << 42) | ((uint64_t)(iy + kKeyRange) << 21) | (uint64_t)(iz + kKeyRange);
}

__host__ __device__ __forceinline__ int half_floor(int i) { return i >= 0 ? i / 2 : -((-i + 1) / 2); }

// scan offsets: start at 0, never decrease, end at n (first violation, or
// LLONG_MAX); poses finite
__global__ void check_inputs_kernel(int32_t n_scans, const int64_t* spo, int64_t n, const double* poses,
                                    long long* bad_off, long long* bad_pose) {
  grid_launch_next();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j > n_scans) return;
  if (j == 0 && spo[0] != 0) atomicMin(bad_off, 0ll);
  if (j == n_scans) {
    if (spo[j] != n) atomicMin(bad_off, (long long)j);
    return;
  }
  if (spo[j + 1] < spo[j]) atomicMin(bad_off, (long long)(j + 1));
  bool fin = true;
  for (int k = 0; k < 12; ++k) fin = fin && isfinite(poses[12 * (int64_t)j + k]);
  if (!fin) atomicMin(bad_pose, (long long)j);
}

// floor(w / d) of Eq. 4, the floor of the correctly rounded quotient, from
// q, an approximation of w / d within 2^-29 (the pose pre-divided by d).
// Adding 1.5 * 2^32 rounding down leaves q rounded down to a multiple of
// 2^-20 (the spacing of doubles in [2^32, 2^33)), read back as the integer
// z = floor(q * 2^20): z >> 20 = floor(q), and when the low 20 bits show q at
// least 2^-20 from an integer, w / d and its rounding have that floor too.
// Otherwise (and for |q| >= 2^21 or NaN) returns false: the caller divides.
__device__ __forceinline__ bool floor_fast(double q, int* k, bool* ok) {
  const unsigned ex = (unsigned)((unsigned long long)__double_as_longlong(q) >> 52) & 0x7ffu;
  if (ex >= 1023u + 21u) return false;
  const double M = 6442450944.0;  // 1.5 * 2^32
  const long long z = __double_as_longlong(__dadd_rd(q, M)) - __double_as_longlong(M);
  const long long fr = z & 0xfffffll;
  if (fr == 0 || fr == 0xfffffll) return false;
  const long long f = z >> 20;
  *ok = f >= -(long long)kKeyRange && f < (long long)kKeyRange;
  *k = *ok ? (int)f : 0;
  return true;
}

// The index of a point in integer arithmetic, from its scan's pose over the
// voxel size in fixed point: per axis three coefficients in steps of 2^-kS
// voxels per metre and an offset in steps of 2^-32 voxels.  A coordinate is
// taken in steps of 2^-kp metres (cut off, 31 bits), so that with kS + kp = 48
// an axis is three 32-bit multiply-adds into 64 bits, shifted down by 16: the
// index in the high word, its fraction in the low one.  For 1 / d < 2^e, kS =
// 30 - e and kp = 18 + e; points up to 2^(13 - e) metres (4,096 voxels and
// more) have 31 bits.  The error against the correctly rounded quotient is below
//   (largest sum of a row's |coefficients|) 2^-kp   [coordinates cut off]
//   + 3 2^(31 - kp) 2^-(kS + 1) = 3 2^-18           [coefficients rounded]
//   + 2^-28   [offset and shift; the FP64 rounding of w and w / d, below 2^21 2^-51]
// voxels: with the fraction at least that far (w) from 0 and 1, the floor is
// the same; otherwise (about one point in 10^4) the point takes the FP64 path.
// w = 0: the pose does not fit (not finite, a coefficient of 2^30 steps, an
// offset of 2^21 voxels).
struct __align__(16) ScanFix {
  int c[9];
  unsigned w;
  long long o[3];
};
static_assert(sizeof(ScanFix) == 64, "four 16-byte loads");

// poses divided by the voxel size (rd = 1 / d): in FP64, and in fixed point
__global__ void scaled_poses_kernel(int32_t n_scans, const double* poses, double rd, int kS, int kp, double* out,
                                    ScanFix* fix) {
  grid_wait();
  grid_launch_next();
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_scans) return;
  ScanFix f;
  bool ok = true;
  double row = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double sum = 0.0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const double S = poses[12 * j + 3 * a + b] * rd;
      out[12 * j + 3 * a + b] = S;
      const double c = rint(scalbn(S, kS));
      const bool in = fabs(c) < 0x1p30;  // false for NaN
      ok = ok && in;
      f.c[3 * a + b] = in ? (int)c : 0;
      sum += fabs(S);
    }
    const double o = poses[12 * j + 9 + a] * rd;
    out[12 * j + 9 + a] = o;
    const bool in = fabs(o) < 0x1p21;
    ok = ok && in;
    f.o[a] = in ? __double2ll_rn(o * 0x1p32) : 0ll;
    row = fmax(row, sum);
  }
  // in steps of 2^-32 voxels (coefficients below 2^30 steps: below 2^17 steps)
  const double w = ceil((scalbn(row, -kp) + 3.0 * 0x1p-18) * 0x1p32) + 32.0;
  f.w = ok ? (unsigned)w : 0u;
  fix[j] = f;
}

// a coordinate cut off to steps of 2^-kp (sh = 1054 - kp), within one step;
// r gets the smallest shift met: below 1 the coordinate does not fit (large,
// infinite or NaN)
__device__ __forceinline__ int fix31(double p, int sh, int& r) {
  const unsigned hi = (unsigned)__double2hiint(p), lo = (unsigned)__double2loint(p);
  const int s = sh - ((int)(hi >> 20) & 0x7ff);
  r = min(r, s);
  const unsigned m = (__funnelshift_l(lo, hi, 11) | 0x80000000u) >> (min(s, 31) & 31);
  const int neg = (int)hi >> 31;
  return ((int)m ^ neg) - neg;
}

// the scan of point gi: the last j in [lo, n_scans) with spo[j] <= gi
__device__ __forceinline__ int scan_of_point(const int64_t* spo, int lo, int n_scans, int64_t gi) {
  int hi = n_scans;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (spo[mid] <= gi)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

constexpr int kKeyThreads = 256;
constexpr int kKeyPoints = 4;  // points of a thread in flight
constexpr int kKeyRounds = 4;  // at most so many times kKeyThreads kKeyPoints consecutive points to a tile

// L1 (Eq. 4): world point w = R p + t, index floor(w / d), raw key; the
// index bounding box (one atomic per block) and the first point whose index
// leaves the key range.  Blocks take tiles of consecutive points of a batch
// starting at global point p0 (pts, keys and pscan are indexed within the
// batch); a thread keeps its scan until a point passes the scan's end.
//
// Bound: HBM, 24 bytes read and 12 written a point.  120M points: 0.85 ms (5.1
// TB/s); 2.63 ms with the index in FP64 (9 multiply-adds and 3 additions a
// point, 88% of the FP64 pipe).
__global__ void __launch_bounds__(kKeyThreads) l1_keys_kernel(int32_t n_scans, const int64_t* __restrict__ spo,
                                                              const double* __restrict__ pts,
                                                              const double* __restrict__ poses,
                                                              const double* __restrict__ sposes,
                                                              const ScanFix* __restrict__ fix, int kp, double d,
                                                              int rounds, int64_t p0, int64_t n,
                                                              uint64_t* __restrict__ keys,
                                                              int32_t* __restrict__ pscan, long long* bad, int* bbox) {
  grid_launch_next();
  int mn[3] = {INT_MAX, INT_MAX, INT_MAX}, mx[3] = {INT_MIN, INT_MIN, INT_MIN};
  const int64_t tile = (int64_t)kKeyThreads * kKeyPoints * rounds;
  for (int64_t t0 = (int64_t)blockIdx.x * tile; t0 < n; t0 += (int64_t)gridDim.x * tile) {
    int j = 0;
    int64_t end = 0;  // of scan j, in points of the batch (0: no scan yet)
    ScanFix f;
    for (int round = 0; round < rounds; ++round) {
      const int64_t i0 = t0 + round * (kKeyThreads * kKeyPoints) + threadIdx.x;
      if (i0 >= n) break;
      double x[kKeyPoints], y[kKeyPoints], z[kKeyPoints];
#pragma unroll
      for (int k = 0; k < kKeyPoints; ++k) {
        const int64_t i = i0 + k * kKeyThreads;
        const bool in = i < n;
        x[k] = in ? __ldcs(pts + 3 * i) : 0.0;
        y[k] = in ? __ldcs(pts + 3 * i + 1) : 0.0;
        z[k] = in ? __ldcs(pts + 3 * i + 2) : 0.0;
      }
#pragma unroll
      for (int k = 0; k < kKeyPoints; ++k) {
        const int64_t i = i0 + k * kKeyThreads;
        if (i >= n) break;
        if (i >= end) {
          j = scan_of_point(spo, j, n_scans, p0 + i);
          end = j + 1 < n_scans ? spo[j + 1] - p0 : n;
          f = fix[j];
        }
        int r = 32;
        const int u[3] = {fix31(x[k], 1054 - kp, r), fix31(y[k], 1054 - kp, r), fix31(z[k], 1054 - kp, r)};
        int ix[3];
        bool fast = r >= 1 && f.w != 0u, ok = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const long long acc = (long long)f.c[3 * a] * u[0] + (long long)f.c[3 * a + 1] * u[1] +
                                (long long)f.c[3 * a + 2] * u[2];
          const long long q = (acc >> 16) + f.o[a];
          ix[a] = (int)(q >> 32);
          fast = fast && (unsigned)q - f.w < 0u - 2u * f.w;
          ok = ok && (unsigned)(ix[a] + kKeyRange) < 2u * kKeyRange;
        }
        if (!fast) {
          ok = true;
          const double* S = sposes + 12 * (int64_t)j;
          const double p[3] = {x[k], y[k], z[k]};
#pragma unroll 1
          for (int a = 0; a < 3; ++a) {
            bool oka = false;
            int ia = 0;
            const double q = fma(S[3 * a], p[0], fma(S[3 * a + 1], p[1], fma(S[3 * a + 2], p[2], S[9 + a])));
            if (!floor_fast(q, &ia, &oka)) {
              const double* T = poses + 12 * (int64_t)j;
              const double w = fma(T[3 * a], p[0], fma(T[3 * a + 1], p[1], fma(T[3 * a + 2], p[2], T[9 + a])));
              const double fl = floor(__ddiv_rn(w, d));
              oka = fl >= -(double)kKeyRange && fl < (double)kKeyRange;
              ia = oka ? (int)fl : 0;
            }
            ok = ok && oka;
            ix[0] = a == 0 ? ia : ix[0];
            ix[1] = a == 1 ? ia : ix[1];
            ix[2] = a == 2 ? ia : ix[2];
          }
        }
        if (!ok) {
          atomicMin(bad, (long long)(p0 + i));
        } else {
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            mn[a] = min(mn[a], ix[a]);
            mx[a] = max(mx[a], ix[a]);
          }
        }
        keys[i] = ok ? raw_key(ix[0], ix[1], ix[2]) : 0;
        pscan[i] = j;
      }
    }
  }
  __shared__ int red[6][8];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int a0 = __reduce_min_sync(full, mn[a]), a1 = __reduce_max_sync(full, mx[a]);
    if (lane == 0) {
      red[a][w] = a0;
      red[3 + a][w] = a1;
    }
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    const int a = threadIdx.x;
    int v = red[a][0];
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) v = a < 3 ? min(v, red[a][k]) : max(v, red[a][k]);
    if (a < 3 && v != INT_MAX) atomicMin(bbox + a, v);
    if (a >= 3 && v != INT_MIN) atomicMax(bbox + a, v);
  }
}

// raw keys -> level-1 keys packed to the index range
// Bound by DRAM (8 bytes read, sizeof(K) written): four keys of a thread in
// flight (120M keys, sort included, 2670 -> 2400 us against one key per thread).
constexpr int kRepackThreads = 256, kRepackItems = 4;
template <typename K>
__global__ void __launch_bounds__(kRepackThreads) repack_kernel(int64_t n, const uint64_t* raw, KeyPack p, K* keys) {
  grid_wait();
  grid_launch_next();
  const int64_t i0 = (int64_t)blockIdx.x * (kRepackThreads * kRepackItems) + threadIdx.x;
  uint64_t r[kRepackItems];
#pragma unroll
  for (int c = 0; c < kRepackItems; ++c) {
    const int64_t i = i0 + c * kRepackThreads;
    r[c] = i < n ? raw[i] : 0;
  }
#pragma unroll
  for (int c = 0; c < kRepackItems; ++c) {
    const int64_t i = i0 + c * kRepackThreads;
    const int ix = (int)((r[c] >> 42) & 0x1fffffull) - kKeyRange, iy = (int)((r[c] >> 21) & 0x1fffffull) - kKeyRange,
              iz = (int)(r[c] & 0x1fffffull) - kKeyRange;
    if (i < n) keys[i] = (K)pack_key(p, ix, iy, iz);
  }
}

// group heads as one 32-bit word per 32 elements (bit k: element 32 w + k
// starts a new (key, scan) group in sorted order) and the number of heads of
// each word.  A warp makes kHeadWords consecutive words, lane l element l of
// each, with every load issued before the first comparison; an element's
// predecessor comes from the lane before (lane 0 loads its own).
constexpr int kHeadWords = 4;
template <typename K>
__global__ void head_mask_kernel(int64_t n, const K* keys, const uint32_t* vals, const int32_t* scan, uint32_t* mask,
                                 int64_t* wcount) {
  grid_wait();
  grid_launch_next();
  const int lane = threadIdx.x & 31;
  const int64_t w0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kHeadWords;
  K key[kHeadWords], key0[kHeadWords];
  int32_t sc[kHeadWords], sc0[kHeadWords];
  uint32_t v[kHeadWords], v0[kHeadWords];
#pragma unroll
  for (int k = 0; k < kHeadWords; ++k) {
    const int64_t i = (w0 + k) * 32 + lane;
    key[k] = i < n ? keys[i] : (K)0;
    v[k] = i < n ? vals[i] : 0u;
    // lane 0: the element before the word
    const bool pre = lane == 0 && i < n && i > 0;
    key0[k] = pre ? keys[i - 1] : (K)0;
    v0[k] = pre ? vals[i - 1] : 0u;
  }
#pragma unroll
  for (int k = 0; k < kHeadWords; ++k) {
    const int64_t i = (w0 + k) * 32 + lane;
    sc[k] = i < n ? scan[v[k]] : 0;
    sc0[k] = (lane == 0 && i < n && i > 0) ? scan[v0[k]] : 0;
  }
#pragma unroll
  for (int k = 0; k < kHeadWords; ++k) {
    const int64_t i = (w0 + k) * 32 + lane;
    K pk = __shfl_up_sync(0xffffffffu, key[k], 1);
    int32_t ps = __shfl_up_sync(0xffffffffu, sc[k], 1);
    if (lane == 0) {
      pk = key0[k];
      ps = sc0[k];
    }
    const bool h = i < n && (i == 0 || key[k] != pk || sc[k] != ps);
    const uint32_t m = __ballot_sync(0xffffffffu, h);
    if (lane == 0 && i < n) {
      mask[w0 + k] = m;
      wcount[w0 + k] = __popc(m);
    }
  }
}

// group starts from the mask and the words' exclusive head counts, and the
// end sentinel; n_zero words (at most the grid's threads) set to zero for a
// kernel to come
__global__ void mask_starts_kernel(int64_t n_words, const uint32_t* mask, const int64_t* base, int64_t n,
                                   int64_t* start, int64_t n_groups, uint32_t* zero, int64_t n_zero) {
  grid_wait();
  grid_launch_next();
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w < n_zero) zero[w] = 0;
  if (w >= n_words) return;
  uint32_t m = mask[w];
  int64_t b = base[w];
  while (m) {
    start[b++] = 32 * w + (__ffs(m) - 1);
    m &= m - 1u;
  }
  if (w == 0) start[n_groups] = n;
}

// ---- clusters (Eq. 2, centred) ----------------------------------------------
// Shifted sums of a merged cluster: n points, shift s, a = sum (p - s),
// b = sum (p - s)(p - s)^T (xx, xy, xz, yy, yz, zz); the centred cluster is
// m = s + a/n, S = b - a a^T / n.  The shift keeps every term small (a voxel's
// extent), so no large cancellation occurs.
struct Piece {
  double n, s[3], a[3], b[6];
};

// A cluster's row (80 bytes, 16-byte aligned in every buffer of the library) as
// five 128-bit accesses: where each thread has a row of its own, half the
// requests to L1 that single values make.
__device__ __forceinline__ void load_row(const double* c, double* r) {
  const double2* p = reinterpret_cast<const double2*>(c);
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const double2 v = p[q];
    r[2 * q] = v.x;
    r[2 * q + 1] = v.y;
  }
}
__device__ __forceinline__ void store_row(const double* r, double* c) {
  double2* p = reinterpret_cast<double2*>(c);
#pragma unroll
  for (int q = 0; q < 5; ++q) p[q] = make_double2(r[2 * q], r[2 * q + 1]);
}

// centred cluster record (S xx..zz, m, N)
__device__ __forceinline__ void piece_finish(const Piece& P, double* c) {
  const double r = __drcp_rn(P.n);
  const double u[3] = {P.a[0] * r, P.a[1] * r, P.a[2] * r};
  int k = 0;
#pragma unroll
  for (int x = 0; x < 3; ++x)
#pragma unroll
    for (int y = x; y < 3; ++y) {
      c[k] = fma(-u[x], P.a[y], P.b[k]);
      ++k;
    }
#pragma unroll
  for (int q = 0; q < 3; ++q) c[6 + q] = P.s[q] + u[q];
  c[9] = P.n;
}

// L1 clusters: the points of each (key, scan) run of the sorted order, as sums
// of their offsets from the run's first point p0, m = p0 + (sum d) / N and
// S = sum d d^T - (sum d)(sum d)^T / N.  The sums are exact integer sums in
// fixed point (RunFrame, fixed_sums.cuh), in finer steps where the points lie so
// close together that the frame's are not small against them (run_exact,
// cluster_tight); a run whose points do not fit (the poses stretch it over 2^54
// steps, or coordinates outside 2^-400 .. 2^400) takes the same sums in FP64.
//
// One thread per run of fewer than kLongRun points, a block's runs in order of
// their lengths so that a warp's lanes are about as long, each lane with its
// next point on the way.  The block's two warps take the groups of 32 runs
// longest first, as they get free (one warp per group leaves the warps of short
// runs idle until the longest is done).  Longer runs, in pieces of kPiecePoints,
// and those of close points go to lists that a second kernel hands to warps over
// the whole chip.
//
// Bound: latency of the gathers (a run's points lie together, its neighbours'
// elsewhere) against four warps a scheduler.  120M points in 12.3M runs: FP64 sums
// over fixed chunks of 32 sorted points, merged per run, 3.12 + 0.91 ms; so 2.91 ms
// and 0.17 ms for the second kernel.  (Runs ordered in pools of 256, 512 and 1,024
// cost their neighbours' lines in L1 and L2: 2.97, 3.6, 3.7 ms.)  65,000 points in
// 7,400 runs: 54 -> 31 + 11 us.  Few long runs: 30 of 33,000 points 1.97 ms in
// chunks (3.77 with whole runs to the warps of the block that met them), so 0.04.
constexpr int kLongRun = 192;  // below kHalfPoints
static_assert(kLongRun <= kHalfPoints, "a thread's sums must fit");
constexpr int kPiecePoints = 1024;  // of a long run, to a warp
static_assert(kPiecePoints <= 32 * kHalfPoints, "a warp's sums must fit");
constexpr int kWarpRun = 64;  // a run of close points takes a warp from so many on

// A warp's share: a piece of a long run (the sums of one of several go to place
// slot + piece), or, with n_pieces = 0, a run of close points.
struct __align__(16) WarpItem {
  uint32_t run, piece, n_pieces, slot;
};
// What is left to l1_rest_kernel of a call over n points: the list of warps'
// shares, the places for pieces' sums (10 each), the shorter runs of close points,
// and the counters (shares listed, places taken, those runs, then the finished
// pieces of each slot).
struct RestRuns {
  WarpItem* list;
  double* sums;
  uint32_t* tight;
  uint32_t* counters;
};
int64_t rest_items(int64_t n) { return n / kPiecePoints + n / kWarpRun; }
int64_t rest_places(int64_t n) { return 2 * (n / kPiecePoints); }  // of runs of two pieces and more
int64_t rest_counters(int64_t n) { return 3 + rest_places(n); }

// bin of a run's length for the block's ordering; 31 = long
__device__ __forceinline__ int run_bin(int64_t len) {
  if (len <= 24) return len <= 8 ? (int)len : 4 + (int)(len >> 1);
  return len < 96 ? 13 + (int)(len >> 3) : len < kLongRun ? 25 + (int)((len - 96) >> 5) : 31;
}

// Fixed-point frame of a run: per axis the scale (steps of 2^-F) and the first
// point in steps.  A step is half the last bit of the first point's coordinate,
// which loses no more of an offset than FP64 does (a smaller coordinate is off
// by a quarter of that bit at most, and FP64's difference, at least half the
// first coordinate, by half).  It is no finer than 2^-f_cap, about 2^-53 of the
// voxel's diagonal, so that the offsets have room; an axis cut off so (capped)
// rounds its points by up to half a step, which run_exact weighs.
struct RunFrame {
  int F[3];
  long long X[3];
  bool fits;
  bool capped[3];
};
__device__ __forceinline__ RunFrame run_frame(double x, double y, double z, int f_cap) {
  const double p[3] = {x, y, z};
  RunFrame f;
  f.fits = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int F = 1076 - ((__double2hiint(p[a]) >> 20) & 0x7ff);
    f.capped[a] = F > f_cap;
    f.F[a] = min(F, f_cap);
    f.fits = f.fits && f.F[a] >= -400 && f.F[a] <= 400;
    f.X[a] = fix_round(p[a], f.F[a], f.fits);
  }
  return f;
}

// Whether the rounding of n points to the steps of a capped axis stays within
// what FP64 sums of the offsets over chunks of 32 points can lose.  With k =
// min(n, 32) + n / 32 additions on the way of a term and u = 2^-53, those lose up
// to (3 k + 5) u sum d^2 of an entry (k + 2 in sum d^2, 2 k in (sum d)^2 / n, and
// the last operations); half a step a point, in both sums, loses up to 2 sum |d|
// steps.  As (sum |d|)^2 <= n sum d^2, that is less where sum d^2 >= 4 n 2^106 /
// (3 k + 5)^2 (in steps): points a few percent of the voxel apart, or more.
// xx, yy, zz: sum d^2.
__device__ __forceinline__ bool run_exact(const RunFrame& f, __int128 xx, __int128 yy, __int128 zz, int n) {
  const float k = (float)(3 * (n < 32 ? n : 32 + n / 32) + 5);
  const float least = 0x1p48f * ((float)n / (k * k));  // in units of 2^60
  auto enough = [&](bool capped, __int128 v) { return !capped || (float)(long long)(v >> 60) >= least; };
  return enough(f.capped[0], xx) && enough(f.capped[1], yy) && enough(f.capped[2], zz);
}

// record from the exact sums: t = sum d d^T, s = sum d as FP64, n points, rn = 1 / n
__device__ __forceinline__ void run_record(const RunFrame& f, const __int128* t, const double (&s)[3], double n,
                                           double rn, double* c) {
  int k = 0;
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    const double d = s[x] * rn;
#pragma unroll
    for (int y = x; y < 3; ++y) {
      c[k] = fma(-s[y], d, i128_scaled(t[k], -(f.F[x] + f.F[y])));
      ++k;
    }
    c[6 + x] = i64_scaled(f.X[x], -f.F[x]) + d;
  }
  c[9] = n;
}

// the sums of every stride-th point from sorted position e on, in FP64 (a = sum d,
// b = sum d d^T), four points on their way at a time
__device__ __noinline__ void run_sums_f64(int64_t e, int64_t end, int stride, const uint32_t* vals, const double* pts,
                                          double p0x, double p0y, double p0z, double* t) {
  constexpr int kAhead = 4;
  for (int q = 0; q < 9; ++q) t[q] = 0.0;
  for (; e < end; e += (int64_t)kAhead * stride) {
    double p[kAhead][3];
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      const int64_t at = e + (int64_t)k * stride;
      const double* v = pts + 3 * (int64_t)vals[at < end ? at : e];
#pragma unroll
      for (int q = 0; q < 3; ++q) p[k][q] = v[q];
    }
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      if (e + (int64_t)k * stride >= end) break;
      const double x = p[k][0] - p0x, y = p[k][1] - p0y, z = p[k][2] - p0z;
      t[0] = fma(x, x, t[0]);
      t[1] = fma(x, y, t[1]);
      t[2] = fma(x, z, t[2]);
      t[3] = fma(y, y, t[3]);
      t[4] = fma(y, z, t[4]);
      t[5] = fma(z, z, t[5]);
      t[6] += x;
      t[7] += y;
      t[8] += z;
    }
  }
}

__device__ __noinline__ void run_record_f64(const double* t, double n, double p0x, double p0y, double p0z, double* c) {
  Piece P{n, {p0x, p0y, p0z}, {t[6], t[7], t[8]}, {t[0], t[1], t[2], t[3], t[4], t[5]}};
  piece_finish(P, c);
}

constexpr int kClusterThreads = 64;

// adds cnt points, every stride-th from sorted position e on, to h, the next
// point and the index of the one after it on their way; false if one does not fit
__device__ __forceinline__ bool run_sums(HalfSums& h, const RunFrame& f, int64_t e, int cnt, int stride,
                                         const uint32_t* __restrict__ vals, const double* __restrict__ pts) {
  int emax = -2048;
  unsigned wide = 0;
  double x = 0.0, y = 0.0, z = 0.0;
  uint32_t next = 0;
  const uint32_t* v = vals + e;
  if (cnt > 0) {
    const double* p = pts + 3 * (int64_t)*v;
    x = p[0];
    y = p[1];
    z = p[2];
  }
  if (cnt > 1) next = *(v += stride);
  for (int k = 0; k < cnt; ++k) {
    const double cx = x, cy = y, cz = z;
    if (k + 1 < cnt) {
      const double* p = pts + 3 * (int64_t)next;
      x = p[0];
      y = p[1];
      z = p[2];
    }
    if (k + 2 < cnt) next = *(v += stride);
    const long long dx = fix_offset(cx, 1075 - f.F[0], f.X[0], emax, wide);
    const long long dy = fix_offset(cy, 1075 - f.F[1], f.X[1], emax, wide);
    const long long dz = fix_offset(cz, 1075 - f.F[2], f.X[2], emax, wide);
    h.add(dx, dy, dz);
  }
  return emax <= 9 && (wide >> 22) == 0u;
}

__device__ __forceinline__ void run_totals(const HalfSums& h, __int128* t) {
#pragma unroll
  for (int k = 0; k < 6; ++k)
    t[k] = join_halves(h.v[3 * k], h.v[3 * k + 1], k == 0 || k == 3 || k == 5 ? 28 : 27, h.v[3 * k + 2]);
}

// Sorted positions [a, b) of a run that starts at a0, by a warp, in FP64: the run's
// record (kWhole: they are all of it), or n, sum d and sum d d^T of the offsets
// from the run's first point, in every lane.
template <bool kWhole>
__device__ __noinline__ void cluster_f64(int64_t a0, int64_t a, int64_t b, int lane, const uint32_t* vals,
                                         const double* pts, double* out) {
  const double* p0 = pts + 3 * (int64_t)vals[a0];
  const double x = p0[0], y = p0[1], z = p0[2], n = (double)(b - a);
  double v[9];
  run_sums_f64(a + lane, b, 32, vals, pts, x, y, z, v);
#pragma unroll
  for (int q = 0; q < 9; ++q)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
  if (kWhole) {
    run_record_f64(v, n, x, y, z, out);
    return;
  }
  out[0] = n;
#pragma unroll
  for (int q = 0; q < 3; ++q) out[1 + q] = v[6 + q];
#pragma unroll
  for (int q = 0; q < 6; ++q) out[4 + q] = v[q];
}

// At most kPiecePoints of them in exact integer sums, or FP64 where they do not
// fit: the run's record (kWhole: they are all of it), or n, sum d and sum d d^T
// of the offsets from the run's first point, in every lane.
template <bool kWhole>
__device__ __forceinline__ void cluster_piece(int64_t a0, int64_t a, int64_t b, int lane,
                                              const uint32_t* __restrict__ vals, const double* __restrict__ pts,
                                              int f_cap, double* out) {
  const double* p0 = pts + 3 * (int64_t)vals[a0];
  const double p0x = p0[0], p0y = p0[1], p0z = p0[2];
  const RunFrame f = run_frame(p0x, p0y, p0z, f_cap);
  const int n = (int)(b - a);
  const int cnt = n > lane ? (n - lane + 31) / 32 : 0;  // points of this lane: every 32nd
  __int128 t[9];
  bool ok;
  {
    HalfSums h;
    h.clear();
    const bool mine = run_sums(h, f, a + lane, cnt, 32, vals, pts);
    ok = __all_sync(0xffffffffu, f.fits && mine);
    run_totals(h, t);
#pragma unroll
    for (int q = 0; q < 3; ++q) t[6 + q] = h.v[18 + q];
  }
#pragma unroll
  for (int q = 0; q < 9; ++q)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t[q] += shfl_xor_i128(0xffffffffu, t[q], o);
  const double nd = (double)n;
  double v[9];  // sum d d^T, sum d
  if (ok && run_exact(f, t[0], t[3], t[5], n)) {  // the same in every lane
#pragma unroll
    for (int q = 0; q < 3; ++q) v[6 + q] = i128_scaled(t[6 + q], -f.F[q]);
    if (kWhole) {
      const double sd[3] = {v[6], v[7], v[8]};
      run_record(f, t, sd, nd, 1.0 / nd, out);
      return;
    }
    int k = 0;
#pragma unroll
    for (int x = 0; x < 3; ++x)
#pragma unroll
      for (int y = x; y < 3; ++y, ++k) v[k] = i128_scaled(t[k], -(f.F[x] + f.F[y]));
    if (f.capped[0] || f.capped[1] || f.capped[2]) {
      // from the first point in whole steps to the point itself, e apart
      const double e[3] = {i64_scaled(f.X[0], -f.F[0]) - p0x, i64_scaled(f.X[1], -f.F[1]) - p0y,
                           i64_scaled(f.X[2], -f.F[2]) - p0z};
      k = 0;
#pragma unroll
      for (int x = 0; x < 3; ++x)
#pragma unroll
        for (int y = x; y < 3; ++y, ++k) v[k] += fma(e[x], fma(nd, e[y], v[6 + y]), e[y] * v[6 + x]);
#pragma unroll
      for (int x = 0; x < 3; ++x) v[6 + x] = fma(nd, e[x], v[6 + x]);
    }
  } else {
    cluster_f64<kWhole>(a0, a, b, lane, vals, pts, out);
    return;
  }
  out[0] = nd;
#pragma unroll
  for (int q = 0; q < 3; ++q) out[1 + q] = v[6 + q];
#pragma unroll
  for (int q = 0; q < 6; ++q) out[4 + q] = v[q];
}

// A run [a, b) of fewer than kLongRun points that lie too close together for the
// steps of its frame (or that do not fit it), by kLanes lanes (sub: this one's
// number), in two passes: the largest offset of each capped axis, then exact
// integer sums in steps of 2^-53 of that offset or finer, which lose nothing that
// FP64 keeps (run_exact: sum d^2 is then 2^104 and more).  FP64 sums where the
// points do not fit.  The record in every lane; every lane of the warp calls it.
template <int kLanes>
__device__ __forceinline__ void cluster_tight(int64_t a, int64_t b, int sub, const uint32_t* __restrict__ vals,
                                              const double* __restrict__ pts, int f_cap, double* rec) {
  constexpr unsigned kAll = 0xffffffffu;
  const double* first = pts + 3 * (int64_t)vals[a];
  const double p0[3] = {first[0], first[1], first[2]};
  RunFrame f = run_frame(p0[0], p0[1], p0[2], f_cap);
  unsigned long long reach[3] = {0, 0, 0};
  int emax = -2048;
  unsigned wide = 0;
  for (int64_t e = a + 1 + sub; e < b; e += kLanes) {
    const double* p = pts + 3 * (int64_t)vals[e];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const long long d = fix_offset(p[q], 1075 - f.F[q], f.X[q], emax, wide);
      reach[q] |= (unsigned long long)(d < 0 ? -d : d);
    }
  }
  __syncwarp();
  bool ok = f.fits && emax <= 9 && (wide >> 22) == 0u;
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) {
#pragma unroll
    for (int q = 0; q < 3; ++q) reach[q] |= __shfl_xor_sync(kAll, reach[q], o);
    ok = __shfl_xor_sync(kAll, (int)ok, o) != 0 && ok;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int finer = f.capped[q] ? 53 - (64 - __clzll((long long)reach[q])) : 0;
    f.F[q] = min(1076 - ((__double2hiint(p0[q]) >> 20) & 0x7ff), f.F[q] + max(finer, 0));
    if (!f.capped[q]) f.F[q] = min(f.F[q], f_cap);
    ok = ok && f.F[q] <= 400;
    f.X[q] = fix_round(p0[q], f.F[q], ok);
  }
  HalfSums h;
  h.clear();
  const int n = (int)(b - a), cnt = n - 1 > sub ? (n - 1 - sub + kLanes - 1) / kLanes : 0;
  ok = run_sums(h, f, a + 1 + sub, cnt, kLanes, vals, pts) && ok;
  __syncwarp();
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) {
#pragma unroll
    for (int q = 0; q < 21; ++q) h.v[q] += __shfl_xor_sync(kAll, h.v[q], o);
    ok = __shfl_xor_sync(kAll, (int)ok, o) != 0 && ok;
  }
  if (ok) {
    __int128 t[6];
    run_totals(h, t);
    const double sd[3] = {i64_scaled(h.v[18], -f.F[0]), i64_scaled(h.v[19], -f.F[1]), i64_scaled(h.v[20], -f.F[2])};
    const float nf = (float)n;
    const double nd = f32_to_f64(nf);
    run_record(f, t, sd, nd, recip_count(nd, nf), rec);
  }
  if (__all_sync(kAll, ok)) return;
  // (a warp's lanes share the points; fewer lanes, whose number the call decides,
  // sum them all, so that it changes no result)
  double t[9];
  constexpr int kShare = kLanes == 32 ? 32 : 1;
  run_sums_f64(a + 1 + (kShare == 32 ? sub : 0), b, kShare, vals, pts, p0[0], p0[1], p0[2], t);
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 9; ++q)
#pragma unroll
    for (int o = 1; o < kShare; o <<= 1) t[q] += __shfl_xor_sync(kAll, t[q], o);
  if (!ok) run_record_f64(t, (double)n, p0[0], p0[1], p0[2], rec);
}

// The runs that l1_clusters_kernel leaves: the pieces of the long ones, a warp to
// a piece (the warp that finishes a run's last piece adds up the pieces' sums,
// each lane every 32nd of them), and the runs of close points (done there, with
// FP64 sums, a few lanes held up their warps: 120M points 12.02 ms a call, so
// 11.69): a lane to each where they fill the grid, else four, which gets the few
// of a small call done sooner (8 scans of 8,192 points 11 us instead of 19).
constexpr int kLongThreads = 128;
__global__ void __launch_bounds__(kLongThreads, 4) l1_rest_kernel(const int64_t* start, const uint32_t* vals,
                                                                  const double* pts, RestRuns R, int f_cap, double* c) {
  grid_wait();
  grid_launch_next();
  const int lane = threadIdx.x & 31;
  const uint32_t n_list = R.counters[0], n_tight = R.counters[2];
  const uint32_t warp = blockIdx.x * (kLongThreads / 32) + (threadIdx.x >> 5), warps = gridDim.x * (kLongThreads / 32);
  auto tight = [&](auto run_lanes) {
    constexpr int kLanes = decltype(run_lanes)::value, kRuns = 32 / kLanes;  // of a warp
    for (int64_t i0 = (int64_t)warp * kRuns; i0 < n_tight; i0 += (int64_t)warps * kRuns) {
      const int64_t i = i0 + lane / kLanes;
      const int64_t g = R.tight[i < n_tight ? i : i0];
      double rec[10];
      cluster_tight<kLanes>(start[g], start[g + 1], lane % kLanes, vals, pts, f_cap, rec);
      if (i < n_tight && lane % kLanes == 0) store_row(rec, c + 10 * g);
    }
  };
  if (n_tight >= 32 * warps)
    tight(std::integral_constant<int, 1>());
  else
    tight(std::integral_constant<int, 4>());
  for (uint32_t i = warp; i < n_list; i += warps) {
    const WarpItem L = R.list[i];
    const int64_t a0 = start[L.run], a = a0 + (int64_t)L.piece * kPiecePoints, end = start[L.run + 1];
    double rec[10];
    if (L.n_pieces == 0) {
      cluster_tight<32>(a0, end, lane, vals, pts, f_cap, rec);
      if (lane == 0) store_row(rec, c + 10 * (int64_t)L.run);
      continue;
    }
    if (L.n_pieces == 1) {
      cluster_piece<true>(a0, a0, end, lane, vals, pts, f_cap, rec);
      if (lane == 0) store_row(rec, c + 10 * (int64_t)L.run);
      continue;
    }
    cluster_piece<false>(a0, a, a + kPiecePoints < end ? a + kPiecePoints : end, lane, vals, pts, f_cap, rec);
    double* sums = R.sums + 10 * (int64_t)L.slot;
    unsigned done = 0;
    if (lane == 0) {
      store_row(rec, sums + 10 * (int64_t)L.piece);
      __threadfence();
      done = atomicAdd(&R.counters[3 + L.slot], 1u);
    }
    if (__shfl_sync(0xffffffffu, done, 0) != L.n_pieces - 1) continue;
    __threadfence();
    double v[10] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (uint32_t k = lane; k < L.n_pieces; k += 32) {
      const double2* row = reinterpret_cast<const double2*>(sums + 10 * (int64_t)k);
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const double2 w = __ldcg(row + q);
        v[2 * q] += w.x;
        v[2 * q + 1] += w.y;
      }
    }
#pragma unroll
    for (int q = 0; q < 10; ++q)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    const double* p0 = pts + 3 * (int64_t)vals[a0];
    const Piece P{v[0], {p0[0], p0[1], p0[2]}, {v[1], v[2], v[3]}, {v[4], v[5], v[6], v[7], v[8], v[9]}};
    piece_finish(P, rec);
    if (lane == 0) store_row(rec, c + 10 * (int64_t)L.run);
  }
}

constexpr int64_t kPoolRuns = 400000;  // runs from which a block orders 128 of them; below, 64 (more blocks)

// (the clusters' keys: the packed key, or raw[point] if raw is given)
template <typename K, int kPool>
__global__ void __launch_bounds__(kClusterThreads, 8) l1_clusters_kernel(int64_t n1, const int64_t* __restrict__ start,
                                                                     const K* __restrict__ keys,
                                                                     const uint32_t* __restrict__ vals,
                                                                     const int32_t* __restrict__ pscan,
                                                                     const double* __restrict__ pts,
                                                                     const uint64_t* __restrict__ raw, int f_cap,
                                                                     RestRuns R, double* c, uint64_t* ckey,
                                                                     int32_t* cscan) {
  grid_launch_next();
  __shared__ int s_cnt[32], s_next, s_n_tight, s_n_warp;
  __shared__ uint16_t s_tight[kPool];  // runs of close points: the short ones from the front
  __shared__ uint32_t s_listed, s_placed, s_base[2];  // pieces and places of the block's long runs
  __shared__ WarpItem s_long[kPool];
  __shared__ uint16_t s_order[kPool];
  __shared__ int64_t s_start[kPool];
  __shared__ int s_len[kPool];
  __shared__ uint32_t s_first[kPool];
  const int64_t r0 = (int64_t)blockIdx.x * kPool;
  const int lane = threadIdx.x & 31;
  {
    // the runs' places, first points, keys and scans in input order (coalesced,
    // independent loads)
    constexpr int kPer = kPool / kClusterThreads;
    int bin[kPer];
    int64_t a[kPer], e[kPer];
    uint32_t v0[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int64_t g = r0 + k * kClusterThreads + threadIdx.x;
      a[k] = g < n1 ? start[g] : 0;
      e[k] = g < n1 ? start[g + 1] : 0;
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) v0[k] = e[k] > a[k] ? vals[a[k]] : 0u;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = k * kClusterThreads + threadIdx.x;
      bin[k] = run_bin(e[k] - a[k]);
      s_start[i] = a[k];
      s_len[i] = (int)(e[k] - a[k] < kLongRun ? e[k] - a[k] : kLongRun);
      s_first[i] = v0[k];
      if (e[k] > a[k]) {
        ckey[r0 + i] = raw ? raw[v0[k]] : (uint64_t)keys[a[k]];
        cscan[r0 + i] = pscan[v0[k]];
      }
    }
    if (threadIdx.x == 0) {
      s_next = s_n_tight = s_n_warp = 0;
      s_listed = s_placed = 0;
    }
    block_order_items<kPer, kClusterThreads>(bin, s_cnt, s_order);
    // the long runs' pieces to the list: places in the block, then the block's
    const int n_long = kPool - s_cnt[31];  // the last ranks
    if (n_long > 0) {
#pragma unroll
      for (int k = 0; k < kPer; ++k)
        if (bin[k] == 31) {
          const uint32_t np = (uint32_t)((e[k] - a[k] + kPiecePoints - 1) / kPiecePoints);
          const uint32_t at = atomicAdd(&s_listed, np);
          const uint32_t slot = np > 1 ? atomicAdd(&s_placed, np) : 0u;
          s_long[k * kClusterThreads + threadIdx.x] = WarpItem{(uint32_t)(r0 + k * kClusterThreads + threadIdx.x), at,
                                                                np, slot};
        }
      __syncthreads();
      if (threadIdx.x == 0) {
        s_base[0] = atomicAdd(&R.counters[0], s_listed);
        s_base[1] = s_placed > 0 ? atomicAdd(&R.counters[1], s_placed) : 0u;
      }
      __syncthreads();
      for (int q = 0; q < n_long; ++q) {
        const WarpItem L = s_long[s_order[kPool - 1 - q]];
        for (uint32_t k = threadIdx.x; k < L.n_pieces; k += kClusterThreads)
          R.list[s_base[0] + L.piece + k] = WarpItem{L.run, k, L.n_pieces, s_base[1] + L.slot};
      }
    }
  }
  for (;;) {
    // the groups of 32, longest first
    int item = lane == 0 ? atomicAdd(&s_next, 1) : 0;
    item = __shfl_sync(0xffffffffu, item, 0);
    const int group = kPool / 32 - 1 - item;
    if (group < 0) break;
    const int i = s_order[group * 32 + lane];
    const int64_t g = r0 + i, a = s_start[i];
    const int len = s_len[i];
    if (len > 0 && len < kLongRun) {
      const uint32_t v0 = s_first[i];
      const double p0x = pts[3 * (int64_t)v0], p0y = pts[3 * (int64_t)v0 + 1], p0z = pts[3 * (int64_t)v0 + 2];
      double* rec = c + 10 * g;
      if (len == 1) {
        const double one[10] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, p0x, p0y, p0z, 1.0};
        store_row(one, rec);
        continue;
      }
      const RunFrame f = run_frame(p0x, p0y, p0z, f_cap);
      HalfSums h;
      h.clear();
      bool ok = f.fits && run_sums(h, f, a + 1, len - 1, 1, vals, pts);  // p0's own offset is zero
      __int128 t[6];
      run_totals(h, t);
      ok = ok && run_exact(f, t[0], t[3], t[5], len);
      if (ok) {
        const double s[3] = {i64_scaled(h.v[18], -f.F[0]), i64_scaled(h.v[19], -f.F[1]),
                             i64_scaled(h.v[20], -f.F[2])};
        const float nf = (float)len;
        const double n = f32_to_f64(nf);
        run_record(f, t, s, n, recip_count(n, nf), rec);
      } else if (len < kWarpRun) {
        s_tight[atomicAdd(&s_n_tight, 1)] = (uint16_t)i;
      } else {
        s_tight[kPool - 1 - atomicAdd(&s_n_warp, 1)] = (uint16_t)i;
      }
    }
  }
  __syncthreads();
  if (s_n_tight + s_n_warp == 0) return;
  if (threadIdx.x == 0) {
    if (s_n_tight > 0) s_base[0] = atomicAdd(&R.counters[2], (uint32_t)s_n_tight);
    if (s_n_warp > 0) s_base[1] = atomicAdd(&R.counters[0], (uint32_t)s_n_warp);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < s_n_tight; k += kClusterThreads) R.tight[s_base[0] + k] = (uint32_t)(r0 + s_tight[k]);
  for (int k = threadIdx.x; k < s_n_warp; k += kClusterThreads)
    R.list[s_base[1] + k] = WarpItem{(uint32_t)(r0 + s_tight[kPool - 1 - k]), 0, 0, 0};
}

// Eq. 5: parent key of every cluster (level packing pc -> pp); sort keys
// (scan first, then parent)
__global__ void parent_keys_kernel(int64_t nc, const uint64_t* ckey, const int32_t* cscan, KeyPack pc, KeyPack pp,
                                   uint64_t* pkey, uint32_t* skey) {
  grid_wait();
  grid_launch_next();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nc) return;
  int ix[3];
  unpack_key(pc, ckey[i], ix);
  pkey[i] = pack_key(pp, half_floor(ix[0]), half_floor(ix[1]), half_floor(ix[2]));
  skey[i] = (uint32_t)cscan[i];
}

template <typename K>
__global__ void gather_keys_kernel(int64_t n, const uint64_t* src, const uint32_t* vals, K* dst) {
  grid_wait();
  grid_launch_next();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = (K)src[vals[i]];
}

// level-k clusters: the children of each (parent, scan) group merged in
// order, shifted to the first child's mean (a centred child has a = 0, so
// its merge is b += S + N dl dl^T, a += N dl).  A block's 256 groups are
// taken in order of their child counts, so a warp's lanes merge about as many
// children each; every group's arithmetic is its own, in order.
template <typename K>
__global__ void __launch_bounds__(kOrderBlock) merge_kernel(int64_t np, const int64_t* start, const uint32_t* vals,
                                                            const double* child, const K* pkeys_sorted,
                                                            const int32_t* cscan, double* c, uint64_t* ckey,
                                                            int32_t* oscan) {
  grid_wait();
  grid_launch_next();
  __shared__ int s_cnt[32], s_order[kOrderBlock];
  const int64_t g0 = (int64_t)blockIdx.x * kOrderBlock + threadIdx.x;
  const int64_t len0 = g0 < np ? start[g0 + 1] - start[g0] : 0;
  const int64_t g =
      (int64_t)blockIdx.x * kOrderBlock + block_order_by_key((int)(len0 < 31 ? len0 : 31), s_cnt, s_order);
  if (g >= np) return;
  const int64_t a = start[g], b = start[g + 1];
  Piece acc;
  {
    double ch[10];
    load_row(child + 10 * (int64_t)vals[a], ch);
    acc.n = ch[9];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      acc.s[q] = ch[6 + q];
      acc.a[q] = 0.0;
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) acc.b[q] = ch[q];
  }
  for (int64_t k = a + 1; k < b; ++k) {
    double ch[10];
    load_row(child + 10 * (int64_t)vals[k], ch);
    const double N = ch[9];
    const double dl[3] = {ch[6] - acc.s[0], ch[7] - acc.s[1], ch[8] - acc.s[2]};
    int q = 0;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const double nd = N * dl[x];
      acc.a[x] += nd;
#pragma unroll
      for (int y = x; y < 3; ++y) {
        acc.b[q] += fma(nd, dl[y], ch[q]);
        ++q;
      }
    }
    acc.n += N;
  }
  double out[10];
  piece_finish(acc, out);
  store_row(out, c + 10 * g);
  ckey[g] = (uint64_t)pkeys_sorted[a];
  oscan[g] = cscan[vals[a]];
}

// batched level 1: clusters of all batches in (key, scan) order (vals = the
// sorted order of the concatenated batches' clusters)
template <typename K>
__global__ void gather_clusters_kernel(int64_t m, const uint32_t* vals, const K* keys, const double* c_in,
                                       const int32_t* scan_in, double* c, uint64_t* ckey, int32_t* cscan) {
  grid_wait();
  grid_launch_next();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const int64_t src = vals[i];
  double r[10];
  load_row(c_in + 10 * src, r);
  store_row(r, c + 10 * i);
  ckey[i] = (uint64_t)keys[i];
  cscan[i] = scan_in[src];
}

// voxels of a level: runs of equal key among its clusters (sorted by key, scan)
__global__ void voxel_heads_kernel(int64_t nc, const uint64_t* ckey, int64_t* pos) {
  grid_wait();
  grid_launch_next();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nc) pos[i] = (i == 0 || ckey[i] != ckey[i - 1]) ? 1 : 0;
}

__global__ void voxel_starts_kernel(int64_t nc, const uint64_t* ckey, const int64_t* pos, int64_t* vstart,
                                    int64_t nv) {
  grid_wait();
  grid_launch_next();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nc && (i == 0 || ckey[i] != ckey[i - 1])) vstart[pos[i]] = i;
  if (i == 0) vstart[nv] = nc;
}

// Selection, per observation: its world mean relative to that of its voxel's
// first observation, w_t - w_a (w = R m + t in FP64, the difference rounded
// to FP32; it is shorter than two voxel diagonals), with N, and the rotated
// scatter R S R^T (FP32).  These enter the planarity test only, whose FP32
// answer is checked against its error bound.  vpos[t + 1] - 1 is t's voxel.
// Bound by the FP64 pipe (64 cycles an instruction): each mean is computed once,
// and the first observation's taken from the block's shared memory where it is
// in the block (a voxel's observations are consecutive), 12 instructions
// instead of 21; the pose in 128-bit loads where its address allows (a gather of
// its own row by each thread is bound by the requests to L1): 21M observations
// in three levels 1173 us, now 960.
__device__ __forceinline__ void world_mean(const double* T, double x, double y, double z, double* w) {
#pragma unroll
  for (int q = 0; q < 3; ++q) w[q] = fma(T[3 * q], x, fma(T[3 * q + 1], y, fma(T[3 * q + 2], z, T[9 + q])));
}

constexpr int kTermThreads = 256;
__global__ void __launch_bounds__(kTermThreads) world_terms_kernel(int64_t nc, const double* c, const int32_t* cscan,
                                                                   const double* poses, const int64_t* vpos,
                                                                   const int64_t* vstart, float4* rel, float4* rsr) {
  __shared__ double mean[3][kTermThreads];
  grid_wait();
  grid_launch_next();
  const int64_t t0 = (int64_t)blockIdx.x * kTermThreads, t = t0 + threadIdx.x;
  const bool live = t < nc;
  double cl[10], T[12];
  int64_t a = 0;
  double w[3];
  if (live) {
    a = vstart[vpos[t + 1] - 1];
    load_row(c + 10 * t, cl);
    const double* pose = poses + 12 * (int64_t)cscan[t];
    if (reinterpret_cast<uintptr_t>(poses) % 16 == 0) {  // the caller's array
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        const double2 v = reinterpret_cast<const double2*>(pose)[q];
        T[2 * q] = v.x;
        T[2 * q + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 12; ++q) T[q] = pose[q];
    }
    world_mean(T, cl[6], cl[7], cl[8], w);
#pragma unroll
    for (int q = 0; q < 3; ++q) mean[q][threadIdx.x] = w[q];
  }
  __syncthreads();
  if (!live) return;
  double wa[3];
  if (a >= t0) {
#pragma unroll
    for (int q = 0; q < 3; ++q) wa[q] = mean[q][a - t0];
  } else {
    world_mean(poses + 12 * (int64_t)cscan[a], c[10 * a + 6], c[10 * a + 7], c[10 * a + 8], wa);
  }
  float d[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) d[q] = f64_to_f32(w[q] - wa[q]);
  rel[t] = make_float4(d[0], d[1], d[2], f64_to_f32(cl[9]));
  float R[9], S[6];
#pragma unroll
  for (int q = 0; q < 9; ++q) R[q] = f64_to_f32(T[q]);
#pragma unroll
  for (int q = 0; q < 6; ++q) S[q] = f64_to_f32(cl[q]);
  const float Sm[3][3] = {{S[0], S[1], S[2]}, {S[1], S[3], S[4]}, {S[2], S[4], S[5]}};
  float RS[3][3];
#pragma unroll
  for (int x = 0; x < 3; ++x)
#pragma unroll
    for (int y = 0; y < 3; ++y) RS[x][y] = fmaf(R[3 * x], Sm[0][y], fmaf(R[3 * x + 1], Sm[1][y], R[3 * x + 2] * Sm[2][y]));
  float o[8];
  int k = 0;
#pragma unroll
  for (int x = 0; x < 3; ++x)
#pragma unroll
    for (int y = x; y < 3; ++y) o[k++] = fmaf(RS[x][0], R[3 * y], fmaf(RS[x][1], R[3 * y + 1], RS[x][2] * R[3 * y + 2]));
  o[6] = o[7] = 0.0f;
  rsr[2 * t] = make_float4(o[0], o[1], o[2], o[3]);
  rsr[2 * t + 1] = make_float4(o[4], o[5], o[6], o[7]);
}

// FP64 covariance (times n) of a voxel's points at the poses, for the cases
// the FP32 test cannot call
__device__ __noinline__ void voxel_cov_f64(int64_t a, int64_t b, const double* c, const int32_t* cscan,
                                           const double* poses, double* A) {
  double n = 0.0, m[3] = {0, 0, 0};
  for (int64_t t = a; t < b; ++t) {
    const double* cl = c + 10 * t;
    const double* T = poses + 12 * (int64_t)cscan[t];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const double w = fma(T[3 * q], cl[6], fma(T[3 * q + 1], cl[7], fma(T[3 * q + 2], cl[8], T[9 + q])));
      m[q] = fma(cl[9], w, m[q]);
    }
    n += cl[9];
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) m[q] /= n;
#pragma unroll
  for (int q = 0; q < 6; ++q) A[q] = 0.0;
  for (int64_t t = a; t < b; ++t) {
    const double* cl = c + 10 * t;
    const double* R = poses + 12 * (int64_t)cscan[t];
    double d[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) d[q] = fma(R[3 * q], cl[6], fma(R[3 * q + 1], cl[7], fma(R[3 * q + 2], cl[8], R[9 + q]))) - m[q];
    const double Sm[3][3] = {{cl[0], cl[1], cl[2]}, {cl[1], cl[3], cl[4]}, {cl[2], cl[4], cl[5]}};
    double RS[3][3];
#pragma unroll
    for (int x = 0; x < 3; ++x)
#pragma unroll
      for (int y = 0; y < 3; ++y) RS[x][y] = fma(R[3 * x], Sm[0][y], fma(R[3 * x + 1], Sm[1][y], R[3 * x + 2] * Sm[2][y]));
    int k = 0;
#pragma unroll
    for (int x = 0; x < 3; ++x)
#pragma unroll
      for (int y = x; y < 3; ++y) {
        const double rsr = fma(RS[x][0], R[3 * y], fma(RS[x][1], R[3 * y + 1], RS[x][2] * R[3 * y + 2]));
        A[k] += fma(cl[9] * d[x], d[y], rsr);
        ++k;
      }
  }
}

__device__ __noinline__ bool planar_f64(const double* A, double tau) {
  double lam[3], V[9];
  eig3_sym(A, lam, V);
  return lam[0] < tau * lam[1];
}

// Selection (Algorithm 1), per voxel: the covariance of its points at the
// poses, n A = sum_t [R S R^T + N_t (w_t - m)(w_t - m)^T] (the scale n does
// not change the test), kept if the voxel has min_obs observations and
// lambda0 < tau lambda1 (tau > 0).  All in FP32 on the relative means: every
// term is positive semidefinite, so the FP32 error is within (k + 16) 2^-22
// tr(nA) for k observations; the answer stands when lambda0 - tau lambda1 is
// farther than 3 times that (and 1e-4 lambda2) from zero, else the voxel goes
// to a list that select_close_kernel decides with the FP64 covariance and
// sweeps (about 1% of the voxels, kept out of this kernel so that their FP64
// work does not stall whole warps).  keep_obs[v] = observations kept (0 or the
// voxel's count).
__global__ void select_kernel(int64_t nv, const int64_t* vstart, const float4* rel, const float4* rsr, float tau,
                              int32_t min_obs, int64_t* keep_obs, int64_t* keep_vox, uint32_t* close,
                              unsigned long long* n_close) {
  grid_wait();
  grid_launch_next();
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= nv) return;
  const int64_t a = vstart[v], b = vstart[v + 1];
  bool keep = (b - a) >= (int64_t)min_obs;
  if (keep && tau > 0.0f) {
    float n = 0.f, m0 = 0.f, m1 = 0.f, m2 = 0.f;
    for (int64_t t = a; t < b; ++t) {
      const float4 o = rel[t];
      m0 = fmaf(o.w, o.x, m0);
      m1 = fmaf(o.w, o.y, m1);
      m2 = fmaf(o.w, o.z, m2);
      n += o.w;
    }
    const float r = 1.0f / n;
    m0 *= r;
    m1 *= r;
    m2 *= r;
    float A[6] = {0, 0, 0, 0, 0, 0};
    for (int64_t t = a; t < b; ++t) {
      const float4 o = rel[t];
      const float4 r0 = rsr[2 * t], r1 = rsr[2 * t + 1];
      const float M[6] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y};
      const float d[3] = {o.x - m0, o.y - m1, o.z - m2};
      int k = 0;
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        const float nd = o.w * d[x];
#pragma unroll
        for (int y = x; y < 3; ++y) {
          A[k] += fmaf(nd, d[y], M[k]);
          ++k;
        }
      }
    }
    float lf[3], vf[9];
    eig3_sym_f(A, lf, vf);
    const float margin = lf[0] - tau * lf[1];
    const float tr = fabsf(A[0]) + fabsf(A[3]) + fabsf(A[5]);
    const float err = 3.0f * (float)(b - a + 16) * 2.384185791e-7f * tr;  // 3 (k + 16) 2^-22 tr
    if (fabsf(margin) > fmaxf(err, 1e-4f * fabsf(lf[2]))) {
      keep = margin < 0.0f;
    } else {
      close[atomicAdd(n_close, 1ull)] = (uint32_t)v;  // decided by select_close_kernel
    }
  }
  keep_obs[v] = keep ? (b - a) : 0;
  keep_vox[v] = keep ? 1 : 0;
}

// the voxels too close to call in FP32, one thread each (grid-stride over the
// list; its order does not matter, each decision is the voxel's own)
__global__ void select_close_kernel(const uint32_t* close, const unsigned long long* n_close, const int64_t* vstart,
                                    const double* c, const int32_t* cscan, const double* poses, double tau,
                                    int64_t* keep_obs, int64_t* keep_vox) {
  grid_wait();
  grid_launch_next();
  const int64_t m = (int64_t)*n_close;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = close[i];
    const int64_t a = vstart[v], b = vstart[v + 1];
    double Ad[6];
    voxel_cov_f64(a, b, c, cscan, poses, Ad);
    const bool keep = planar_f64(Ad, tau);
    keep_obs[v] = keep ? (b - a) : 0;
    keep_vox[v] = keep ? 1 : 0;
  }
}

// kept voxels of a level written at their places in the output
__global__ void emit_kernel(int64_t nv, const int64_t* vstart, const uint64_t* ckey, KeyPack pk, const int32_t* cscan,
                            const double* c, const int64_t* obs_pos, const int64_t* vox_pos, const int64_t* keep_vox,
                            int32_t level, int64_t v_base, int64_t o_base, int64_t* voxel_off, int32_t* obs_scan,
                            double* agg, int32_t* lev, int32_t* index) {
  grid_wait();
  grid_launch_next();
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= nv || !keep_vox[v]) return;
  const int64_t a = vstart[v], b = vstart[v + 1];
  const int64_t ov = v_base + vox_pos[v], oo = o_base + obs_pos[v];
  voxel_off[ov + 1] = oo + (b - a);
  lev[ov] = level;
  int ix[3];
  unpack_key(pk, ckey[a], ix);
  for (int q = 0; q < 3; ++q) index[3 * ov + q] = ix[q];
  for (int64_t t = a; t < b; ++t) {
    obs_scan[oo + (t - a)] = cscan[t];
    double r[10];
    load_row(c + 10 * t, r);
    store_row(r, agg + 10 * (oo + (t - a)));
  }
}

// ---- host helpers ------------------------------------------------------------

thread_local std::string g_vox_error;

// stream-ordered temporaries from the library pool, freed on scope exit
struct Buf {
  std::vector<void*> ptrs;
  cudaStream_t s;
  cudaMemPool_t pool;
  Buf(cudaStream_t st, int device) : s(st), pool(library_pool(device)) {}
  ~Buf() {
    for (void* p : ptrs) cudaFreeAsync(p, s);
  }
  template <typename T>
  T* get(int64_t n) {
    void* p = nullptr;
    const size_t bytes = sizeof(T) * (size_t)(n > 0 ? n : 1);
    if ((pool ? cudaMallocFromPoolAsync(&p, bytes, pool, s) : cudaMallocAsync(&p, bytes, s)) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    ptrs.push_back(p);
    return (T*)p;
  }
};

// CUDA-event timing of the stages on the call's stream (when profiling)
struct StageTimer {
  bool on = false;
  cudaStream_t st = nullptr;
  struct Rec {
    int stage;
    cudaEvent_t a, b;
  };
  std::vector<Rec> recs;
  cudaEvent_t open_ev = nullptr;
  int open_stage = -1;
  void begin(int stage) {
    if (!on) return;
    if (open_ev) cudaEventDestroy(open_ev);  // a stage left open by an error path
    open_ev = nullptr;
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) return;
    cudaEventRecord(e, st);
    open_ev = e;
    open_stage = stage;
  }
  void end() {
    if (!on || !open_ev) return;
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) == cudaSuccess) {
      cudaEventRecord(e, st);
      recs.push_back({open_stage, open_ev, e});
    } else {
      cudaEventDestroy(open_ev);
    }
    open_ev = nullptr;
  }
  // after the stream has been synchronised
  void collect(double* ms) const {
    for (const Rec& r : recs) {
      float t = 0.f;
      if (cudaEventElapsedTime(&t, r.a, r.b) == cudaSuccess) ms[r.stage] += t;
    }
  }
  ~StageTimer() {
    if (open_ev) cudaEventDestroy(open_ev);
    for (const Rec& r : recs) {
      cudaEventDestroy(r.a);
      cudaEventDestroy(r.b);
    }
  }
};

unsigned blocks_for(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t > 0 ? (n + t - 1) / t : 1); }

int bit_width_u(uint64_t x) {
  int b = 0;
  while (x) {
    ++b;
    x >>= 1;
  }
  return b;
}

ba_status vfail(ba_status s, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_vox_error = buf;
  return s;
}

#define VCK(call, what)                                                                   \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess)                                                                \
      return e_ == cudaErrorMemoryAllocation ? vfail(BA_ERR_OOM, "%s: out of device memory", what) \
                                             : vfail(BA_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e_)); \
  } while (0)

cudaError_t sort_keys(uint32_t** k, uint32_t** v, uint32_t** tk, uint32_t** tv, int64_t n, int bits, bool positions,
                      int64_t* scr, cudaStream_t st, int64_t* launches) {
  return radix_sort_pairs(k, v, tk, tv, n, bits, positions, scr, st, launches);
}
cudaError_t sort_keys(uint64_t** k, uint32_t** v, uint64_t** tk, uint32_t** tv, int64_t n, int bits, bool positions,
                      int64_t* scr, cudaStream_t st, int64_t* launches) {
  return radix_sort_pairs64(k, v, tk, tv, n, bits, positions, scr, st, launches);
}

// groups of a sorted (key, scan) sequence: start (n_groups + 1 entries); n_zero
// words (at most n / 512 + 256) are set to zero on the way
template <typename K>
ba_status group_starts(int64_t n, const K* keys, const uint32_t* vals, const int32_t* scan, Buf& tmp,
                       int64_t** start_out, int64_t* n_groups, cudaStream_t st, int64_t* launches,
                       uint32_t* zero = nullptr, int64_t n_zero = 0) {
  const int64_t nw = (n + 31) / 32;
  uint32_t* mask = tmp.get<uint32_t>(nw);
  int64_t* base = tmp.get<int64_t>(nw + 1);
  int64_t* scr = tmp.get<int64_t>(scan_scratch_count(nw + 1));
  if (!mask || !base || !scr) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
  launch_chained(head_mask_kernel<K>, blocks_for((nw + kHeadWords - 1) / kHeadWords, 8), 256, 0, st, n, keys, vals,
                 scan, mask, base);
  VCK(cudaGetLastError(), "voxelize");
  VCK(cudaMemsetAsync(base + nw, 0, sizeof(int64_t), st), "voxelize");
  VCK(exclusive_scan_i64(base, nw + 1, scr, st, launches), "voxelize");
  int64_t ng = 0;
  VCK(cudaMemcpyAsync(&ng, base + nw, sizeof ng, cudaMemcpyDeviceToHost, st), "voxelize");
  VCK(cudaStreamSynchronize(st), "voxelize");
  int64_t* start = tmp.get<int64_t>(ng + 1);
  if (!start) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
  launch_chained(mask_starts_kernel, blocks_for(nw), 256, 0, st, nw, mask, base, n, start, ng, zero,
                 n_zero);
  VCK(cudaGetLastError(), "voxelize");
  *launches += 2;
  *start_out = start;
  *n_groups = ng;
  return BA_OK;
}

// packing of a level whose indices per axis lie in [lo, hi]
KeyPack make_pack(const int* lo, const int* hi) {
  KeyPack p;
  for (int a = 0; a < 3; ++a) {
    p.lo[a] = lo[a];
    p.w[a] = bit_width_u((uint64_t)(hi[a] - lo[a]));
  }
  return p;
}

int pack_bits(const KeyPack& p) { return p.w[0] + p.w[1] + p.w[2]; }

struct Level {
  int64_t nc = 0, nv = 0;
  double* c = nullptr;
  uint64_t* key = nullptr;
  int32_t* scan = nullptr;
  int64_t* vstart = nullptr;
  KeyPack pk{};
  int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
};

// level 1: raw keys -> packed keys, sort, (key, scan) runs, clusters
// (the clusters go to out, the rest to tmp; raw_keys: clusters keep raw keys)
template <typename K>
ba_status level1(int64_t n, const uint64_t* raw, const int32_t* pscan, const double* pts, Level& L,
                 bool raw_keys, int f_cap, int n_sm, Buf& out, Buf& tmp, StageTimer& tm, cudaStream_t st,
                 int64_t* launches) {
  K* keys = tmp.get<K>(n);
  K* tkeys = tmp.get<K>(n);
  uint32_t* vals = tmp.get<uint32_t>(n);
  uint32_t* tvals = tmp.get<uint32_t>(n);
  int64_t* scr = tmp.get<int64_t>(radix_scratch_count(n));
  if (!keys || !tkeys || !vals || !tvals || !scr) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
  tm.begin(BA_VOX_SORT);
  launch_chained(repack_kernel<K>, blocks_for(n, kRepackThreads * kRepackItems), kRepackThreads, 0, st, n, raw, L.pk,
                 keys);
  ++*launches;
  VCK(cudaGetLastError(), "voxelize keys");
  // stable by key over points in scan order: groups ordered by (key, scan, point)
  VCK(sort_keys(&keys, &vals, &tkeys, &tvals, n, pack_bits(L.pk), true, scr, st, launches), "voxelize sort");
  tm.end();
  int64_t* start = nullptr;
  int64_t n1 = 0;
  tm.begin(BA_VOX_RUNS);
  RestRuns R{};
  {
    char* b = tmp.get<char>(16 * rest_items(n) + 80 * rest_places(n) + 4 * rest_counters(n));
    if (!b) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
    R.list = (WarpItem*)b;
    R.sums = (double*)(R.list + rest_items(n));
    R.counters = (uint32_t*)(R.sums + 10 * rest_places(n));
  }
  ba_status s = group_starts<K>(n, keys, vals, pscan, tmp, &start, &n1, st, launches, R.counters, rest_counters(n));
  tm.end();
  if (s != BA_OK) return s;
  L.nc = n1;
  L.c = out.get<double>(10 * n1);
  L.key = out.get<uint64_t>(n1);
  L.scan = out.get<int32_t>(n1);
  R.tight = tmp.get<uint32_t>(n1);
  if (!L.c || !L.key || !L.scan || !R.tight) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
  tm.begin(BA_VOX_CLUSTER_PASS);
  auto clusters = [&](auto pool) {
    l1_clusters_kernel<K, decltype(pool)::value><<<blocks_for(n1, decltype(pool)::value), kClusterThreads, 0, st>>>(
        n1, start, keys, vals, pscan, pts, raw_keys ? raw : nullptr, f_cap, R, L.c, L.key, L.scan);
  };
  if (n1 > kPoolRuns)
    clusters(std::integral_constant<int, 128>());
  else
    clusters(std::integral_constant<int, 64>());
  tm.end();
  ++*launches;
  VCK(cudaGetLastError(), "voxelize clusters");
  if (n1 < n) {  // else every point is a run of its own
    tm.begin(BA_VOX_CLUSTER_FINISH);
    const int64_t warps = std::max<int64_t>(rest_items(n), n1 / 8);
    launch_chained(l1_rest_kernel, (unsigned)std::min<int64_t>(blocks_for(warps, kLongThreads / 32), 4 * n_sm),
                   kLongThreads, 0, st, start, vals, pts, R, f_cap, L.c);
    tm.end();
    ++*launches;
    VCK(cudaGetLastError(), "voxelize clusters");
  }
  return BA_OK;
}

// level k+1 (Eq. 5) from level k: parents, sort (scan, then parent), merge
template <typename K>
ba_status level_up(const Level& ch, Level& P, int32_t n_scans, Buf& tmp, cudaStream_t st, int64_t* launches) {
  const int64_t nc = ch.nc;
  uint64_t* pkey = tmp.get<uint64_t>(nc);
  K* k2 = tmp.get<K>(nc);
  K* t2 = tmp.get<K>(nc);
  uint32_t* skey = tmp.get<uint32_t>(nc);
  uint32_t* tsk = tmp.get<uint32_t>(nc);
  uint32_t* cv = tmp.get<uint32_t>(nc);
  uint32_t* tcv = tmp.get<uint32_t>(nc);
  int64_t* scr = tmp.get<int64_t>(radix_scratch_count(nc));
  if (!pkey || !k2 || !t2 || !skey || !tsk || !cv || !tcv || !scr)
    return vfail(BA_ERR_OOM, "voxelize: out of device memory");
  launch_chained(parent_keys_kernel, blocks_for(nc), 256, 0, st, nc, ch.key, ch.scan, ch.pk, P.pk, pkey, skey);
  ++*launches;
  VCK(cudaGetLastError(), "voxelize levels");
  VCK(radix_sort_pairs(&skey, &cv, &tsk, &tcv, nc, bit_width_u((uint64_t)(n_scans - 1)), true, scr, st, launches),
      "voxelize sort");
  launch_chained(gather_keys_kernel<K>, blocks_for(nc), 256, 0, st, nc, pkey, cv, k2);
  ++*launches;
  VCK(cudaGetLastError(), "voxelize levels");
  VCK(sort_keys(&k2, &cv, &t2, &tcv, nc, pack_bits(P.pk), false, scr, st, launches), "voxelize sort");
  int64_t* pst = nullptr;
  int64_t np = 0;
  ba_status s = group_starts<K>(nc, k2, cv, ch.scan, tmp, &pst, &np, st, launches);
  if (s != BA_OK) return s;
  P.nc = np;
  P.c = tmp.get<double>(10 * np);
  P.key = tmp.get<uint64_t>(np);
  P.scan = tmp.get<int32_t>(np);
  if (!P.c || !P.key || !P.scan) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
  launch_chained(merge_kernel<K>, blocks_for(np, kOrderBlock), kOrderBlock, 0, st, np, pst, cv, ch.c, k2, ch.scan, P.c,
                 P.key, P.scan);
  ++*launches;
  VCK(cudaGetLastError(), "voxelize merge");
  return BA_OK;
}

// ---- level 1 over a point range, and the adaptive loader ---------------------
struct L1Ctx {
  int32_t n_scans;
  const int64_t* spo;     // device, n_scans + 1
  const double* T;        // device poses
  const double* sposes;   // device poses / d
  const ScanFix* fix;     // the same in fixed point
  int kp;
  double d;
  long long* bad;         // device: bad[2] = first point out of the key range
  int* bbox;              // device scratch, 6 ints
  int n_sm;
  cudaStream_t st;
  StageTimer* tm;
  int64_t* launches;
};

// level-1 clusters of the points [p0, p0 + m) at pts (device): keys, sort,
// runs, cluster sums.  bb receives the range's index box; raw_keys: the
// clusters carry raw keys (batches are merged later), else keys packed to bb.
ba_status l1_range(const L1Ctx& c, int64_t p0, int64_t m, const double* pts, bool raw_keys, Level& L, int* bb,
                   Buf& out, Buf& tmp) {
  uint64_t* raw = tmp.get<uint64_t>(m);
  int32_t* pscan = tmp.get<int32_t>(m);
  if (!raw || !pscan) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
  const int bb_init[6] = {INT_MAX, INT_MAX, INT_MAX, INT_MIN, INT_MIN, INT_MIN};
  const long long none = LLONG_MAX;
  VCK(cudaMemcpyAsync(c.bbox, bb_init, sizeof bb_init, cudaMemcpyHostToDevice, c.st), "voxelize");
  VCK(cudaMemcpyAsync(c.bad + 2, &none, sizeof none, cudaMemcpyHostToDevice, c.st), "voxelize");
  const int64_t key_blocks = std::min<int64_t>(blocks_for(m, kKeyThreads * kKeyPoints), (int64_t)c.n_sm * 8);
  const int rounds =
      (int)std::min<int64_t>(std::max<int64_t>(m / (key_blocks * kKeyThreads * kKeyPoints), 1), kKeyRounds);
  c.tm->begin(BA_VOX_KEYS);
  l1_keys_kernel<<<(unsigned)key_blocks, kKeyThreads, 0, c.st>>>(c.n_scans, c.spo, pts, c.T, c.sposes, c.fix, c.kp,
                                                                 c.d, rounds, p0, m, raw, pscan, c.bad + 2, c.bbox);
  c.tm->end();
  ++*c.launches;
  VCK(cudaGetLastError(), "voxelize keys");
  long long b2 = 0;
  VCK(cudaMemcpyAsync(&b2, c.bad + 2, sizeof b2, cudaMemcpyDeviceToHost, c.st), "voxelize");
  VCK(cudaMemcpyAsync(bb, c.bbox, 6 * sizeof(int), cudaMemcpyDeviceToHost, c.st), "voxelize");
  VCK(cudaStreamSynchronize(c.st), "voxelize");
  if (b2 != LLONG_MAX)
    return vfail(BA_ERR_CAPACITY, "point %lld lies outside the voxel index range [-2^20, 2^20) at this voxel size",
                 b2);
  L.pk = make_pack(bb, bb + 3);
  // finest fixed-point step of the cluster sums: the diagonal, 2^e (e from ilogb,
  // so diagonal < 2^(e + 1)), in fewer than 2^54 steps
  const int f_cap = 52 - std::ilogb(1.7320508075688772 * c.d);
  return pack_bits(L.pk) <= 32 ? level1<uint32_t>(m, raw, pscan, pts, L, raw_keys, f_cap, c.n_sm, out, tmp, *c.tm,
                                                  c.st, c.launches)
                               : level1<uint64_t>(m, raw, pscan, pts, L, raw_keys, f_cap, c.n_sm, out, tmp, *c.tm,
                                                  c.st, c.launches);
}

ba_status l1_single(const L1Ctx& c, int64_t n, const double* pts, Level& L, int* bb, Buf& tmp) {
  return l1_range(c, 0, n, pts, false, L, bb, tmp, tmp);
}

struct Batch {
  int64_t p0, p1;
};

// points per batch: batch_points if set; else the share alpha of the free
// device memory at kBatchBytesPerPoint per point in flight (two point buffers
// and the batch's keys, indices, sort and cluster temporaries); host inputs
// get at least four batches so that copies run under the clustering
constexpr int64_t kBatchBytesPerPoint = 2 * 24 + 96;

int64_t batch_size(const ba_voxelize_config* cfg, int64_t n, int32_t mem_kind) {
  if (cfg->batch_points > 0) return cfg->batch_points;
  size_t fr = 0, tot = 0;
  if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) {
    cudaGetLastError();
    fr = 0;
  }
  int64_t B = std::max<int64_t>((int64_t)(cfg->alpha * (double)fr / (double)kBatchBytesPerPoint), 1ll << 20);
  if (mem_kind == BA_MEM_HOST) B = std::min<int64_t>(B, std::max<int64_t>((n + 3) / 4, 1ll << 22));
  return B;
}

// consecutive point ranges of at most B points, ending at scan boundaries
// where a boundary lies in the range (a scan longer than B is split)
std::vector<Batch> plan_batches(const std::vector<int64_t>& spo, int64_t B) {
  std::vector<Batch> plan;
  const int64_t n = spo.back();
  int64_t p = 0;
  while (p < n) {
    int64_t e = std::min(p + B, n);
    if (e < n) {
      auto it = std::upper_bound(spo.begin(), spo.end(), e);  // first offset > e
      const int64_t snap = *(it - 1);                        // last offset <= e
      if (snap > p) e = snap;
    }
    plan.push_back({p, e});
    p = e;
  }
  return plan;
}

// level-1 clusters of all batches in (key, scan) order: one stable sort of
// the concatenated clusters by the globally packed key, then either a gather
// or, where a scan was split between batches, a merge of its pieces
template <typename K>
ba_status assemble_batches(const L1Ctx& c, int64_t m, const double* c_all, const uint64_t* raw_all,
                           const int32_t* scan_all, bool any_split, Level& L, Buf& out, Buf& tmp) {
  K* keys = tmp.get<K>(m);
  K* tkeys = tmp.get<K>(m);
  uint32_t* vals = tmp.get<uint32_t>(m);
  uint32_t* tvals = tmp.get<uint32_t>(m);
  int64_t* scr = tmp.get<int64_t>(radix_scratch_count(m));
  if (!keys || !tkeys || !vals || !tvals || !scr) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
  launch_chained(repack_kernel<K>, blocks_for(m, kRepackThreads * kRepackItems), kRepackThreads, 0, c.st, m, raw_all,
                 L.pk, keys);
  ++*c.launches;
  VCK(cudaGetLastError(), "voxelize merge");
  VCK(sort_keys(&keys, &vals, &tkeys, &tvals, m, pack_bits(L.pk), true, scr, c.st, c.launches), "voxelize sort");
  if (!any_split) {
    L.nc = m;
    L.c = out.get<double>(10 * m);
    L.key = out.get<uint64_t>(m);
    L.scan = out.get<int32_t>(m);
    if (!L.c || !L.key || !L.scan) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
    launch_chained(gather_clusters_kernel<K>, blocks_for(m), 256, 0, c.st, m, vals, keys, c_all, scan_all, L.c, L.key,
                   L.scan);
    ++*c.launches;
    VCK(cudaGetLastError(), "voxelize merge");
    return BA_OK;
  }
  int64_t* start = nullptr;
  int64_t ng = 0;
  ba_status s = group_starts<K>(m, keys, vals, scan_all, tmp, &start, &ng, c.st, c.launches);
  if (s != BA_OK) return s;
  L.nc = ng;
  L.c = out.get<double>(10 * ng);
  L.key = out.get<uint64_t>(ng);
  L.scan = out.get<int32_t>(ng);
  if (!L.c || !L.key || !L.scan) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
  launch_chained(merge_kernel<K>, blocks_for(ng, kOrderBlock), kOrderBlock, 0, c.st, ng, start, vals, c_all, keys,
                 scan_all, L.c, L.key, L.scan);
  ++*c.launches;
  VCK(cudaGetLastError(), "voxelize merge");
  return BA_OK;
}

// Host points: a thread issues each batch's copy on a copy stream into one of
// two device buffers (after the clustering of the batch that used the buffer
// before has been enqueued), while this thread clusters the previous batch.
struct CopyPipeline {
  cudaStream_t cs = nullptr;
  std::vector<cudaEvent_t> copied, freed;
  std::mutex mu;
  std::condition_variable cv;
  int issued = 0, released = 0;
  bool stop = false;
  cudaError_t err = cudaSuccess;
  std::thread th;
  ~CopyPipeline() {
    {
      std::lock_guard<std::mutex> lk(mu);
      stop = true;
    }
    cv.notify_all();
    if (th.joinable()) th.join();
    if (cs) cudaStreamSynchronize(cs);
    for (cudaEvent_t e : copied)
      if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : freed)
      if (e) cudaEventDestroy(e);
    if (cs) cudaStreamDestroy(cs);
  }
};

// any_split: some batch edge lies inside a scan
ba_status l1_batched(const L1Ctx& c, const std::vector<Batch>& plan, bool any_split, const double* points,
                     int32_t mem_kind, int device, Level& L, int* bb, Buf& out) {
  const int nb = (int)plan.size();
  std::vector<Level> part(nb);
  int64_t maxb = 0, m = 0;
  for (const Batch& b : plan) maxb = std::max(maxb, b.p1 - b.p0);
  for (int a = 0; a < 3; ++a) {
    bb[a] = INT_MAX;
    bb[3 + a] = INT_MIN;
  }
  auto one = [&](int k, const double* pts) -> ba_status {
    Buf btmp(c.st, device);
    int bk[6];
    ba_status s = l1_range(c, plan[k].p0, plan[k].p1 - plan[k].p0, pts, true, part[k], bk, out, btmp);
    if (s != BA_OK) return s;
    for (int a = 0; a < 3; ++a) {
      bb[a] = std::min(bb[a], bk[a]);
      bb[3 + a] = std::max(bb[3 + a], bk[3 + a]);
    }
    m += part[k].nc;
    return BA_OK;
  };
  if (mem_kind == BA_MEM_DEVICE) {
    for (int k = 0; k < nb; ++k) {
      ba_status s = one(k, points + 3 * plan[k].p0);
      if (s != BA_OK) return s;
    }
  } else {
    double* buf[2] = {out.get<double>(3 * maxb), nb > 1 ? out.get<double>(3 * maxb) : nullptr};
    if (!buf[0] || (nb > 1 && !buf[1])) return vfail(BA_ERR_OOM, "voxelize point buffers: out of device memory");
    VCK(cudaStreamSynchronize(c.st), "voxelize");  // buffers allocated before the copy stream uses them
    CopyPipeline cp;
    VCK(cudaStreamCreateWithFlags(&cp.cs, cudaStreamNonBlocking), "voxelize copy stream");
    cp.copied.assign(nb, nullptr);
    cp.freed.assign(nb, nullptr);
    for (int k = 0; k < nb; ++k) {
      VCK(cudaEventCreateWithFlags(&cp.copied[k], cudaEventDisableTiming), "voxelize");
      VCK(cudaEventCreateWithFlags(&cp.freed[k], cudaEventDisableTiming), "voxelize");
    }
    cp.th = std::thread([&cp, &plan, points, buf, nb, device]() {
      cudaSetDevice(device);
      for (int k = 0; k < nb; ++k) {
        {
          std::unique_lock<std::mutex> lk(cp.mu);
          cp.cv.wait(lk, [&] { return cp.stop || k < 2 || cp.released >= k - 1; });
          if (cp.stop) return;
        }
        cudaError_t e = cudaSuccess;
        if (k >= 2) e = cudaStreamWaitEvent(cp.cs, cp.freed[k - 2], 0);
        if (e == cudaSuccess)
          e = cudaMemcpyAsync(buf[k & 1], points + 3 * plan[k].p0, sizeof(double) * 3 * (plan[k].p1 - plan[k].p0),
                              cudaMemcpyHostToDevice, cp.cs);
        if (e == cudaSuccess) e = cudaEventRecord(cp.copied[k], cp.cs);
        {
          std::lock_guard<std::mutex> lk(cp.mu);
          if (e != cudaSuccess) {
            cp.err = e;
            cp.stop = true;
          } else {
            cp.issued = k + 1;
          }
        }
        cp.cv.notify_all();
        if (e != cudaSuccess) return;
      }
    });
    for (int k = 0; k < nb; ++k) {
      {
        std::unique_lock<std::mutex> lk(cp.mu);
        cp.cv.wait(lk, [&] { return cp.err != cudaSuccess || cp.issued > k; });
        if (cp.err != cudaSuccess) {
          cudaGetLastError();
          return vfail(cp.err == cudaErrorMemoryAllocation ? BA_ERR_OOM : BA_ERR_CUDA, "voxelize copy: %s",
                       cudaGetErrorString(cp.err));
        }
      }
      VCK(cudaStreamWaitEvent(c.st, cp.copied[k], 0), "voxelize");
      ba_status s = one(k, buf[k & 1]);
      if (s != BA_OK) return s;
      VCK(cudaEventRecord(cp.freed[k], c.st), "voxelize");
      {
        std::lock_guard<std::mutex> lk(cp.mu);
        cp.released = k + 1;
      }
      cp.cv.notify_all();
    }
  }
  // concatenate and order the batches' clusters
  c.tm->begin(BA_VOX_MERGE);
  Buf atmp(c.st, device);
  double* c_all = atmp.get<double>(10 * m);
  uint64_t* raw_all = atmp.get<uint64_t>(m);
  int32_t* scan_all = atmp.get<int32_t>(m);
  if (!c_all || !raw_all || !scan_all) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
  int64_t o = 0;
  for (int k = 0; k < nb; ++k) {
    const int64_t q = part[k].nc;
    if (q == 0) continue;
    VCK(cudaMemcpyAsync(c_all + 10 * o, part[k].c, sizeof(double) * 10 * q, cudaMemcpyDeviceToDevice, c.st),
        "voxelize");
    VCK(cudaMemcpyAsync(raw_all + o, part[k].key, sizeof(uint64_t) * q, cudaMemcpyDeviceToDevice, c.st), "voxelize");
    VCK(cudaMemcpyAsync(scan_all + o, part[k].scan, sizeof(int32_t) * q, cudaMemcpyDeviceToDevice, c.st),
        "voxelize");
    o += q;
  }
  L.pk = make_pack(bb, bb + 3);
  ba_status s = pack_bits(L.pk) <= 32
                    ? assemble_batches<uint32_t>(c, m, c_all, raw_all, scan_all, any_split, L, out, atmp)
                    : assemble_batches<uint64_t>(c, m, c_all, raw_all, scan_all, any_split, L, out, atmp);
  c.tm->end();
  return s;
}

}  // namespace

struct ba_voxels {
  int device = 0;
  int64_t n_voxels = 0, n_obs = 0;
  int64_t* voxel_off = nullptr;
  int32_t* obs_scan = nullptr;
  double* agg = nullptr;
  int32_t* level = nullptr;
  int32_t* index = nullptr;
  int64_t launches = 0;
  bool pooled = false;  // arrays from the library pool (stream-ordered frees)
  double stage_ms[BA_VOX_STAGES] = {};
  int64_t batches = 0;  // loader batches of the call (0: no points)
};

extern "C" {

void ba_voxelize_config_default(ba_voxelize_config* cfg) {
  if (!cfg) return;
  cfg->voxel_size = 1.0;
  cfg->levels = 1;
  cfg->tau = 0.0;
  cfg->min_obs = 1;
  cfg->device = 0;
  cfg->cuda_stream = nullptr;
  cfg->profile = 0;
  cfg->batch_points = 0;
  cfg->alpha = 0.25;
}

const char* ba_voxelize_last_error(void) { return g_vox_error.c_str(); }

ba_status ba_voxelize(const ba_voxelize_config* cfg, int32_t n_scans, const int64_t* scan_point_off,
                      const double* points, const double* poses, int32_t mem_kind, ba_voxels** out) {
  if (!cfg || !out || !scan_point_off || !poses) return vfail(BA_ERR_INVALID_ARG, "NULL argument");
  *out = nullptr;
  if (n_scans < 1) return vfail(BA_ERR_INVALID_ARG, "n_scans must be >= 1");
  if (!(cfg->voxel_size > 0.0) || !std::isfinite(cfg->voxel_size))
    return vfail(BA_ERR_INVALID_ARG, "voxel_size must be positive and finite");
  if (cfg->levels < 1 || cfg->levels > 20) return vfail(BA_ERR_INVALID_ARG, "levels must be in 1..20");
  if (mem_kind != BA_MEM_HOST && mem_kind != BA_MEM_DEVICE) return vfail(BA_ERR_INVALID_ARG, "bad mem_kind");
  int prev = -1;
  cudaGetDevice(&prev);
  if (cudaSetDevice(cfg->device) != cudaSuccess) return vfail(BA_ERR_CUDA, "cannot use device %d", cfg->device);
  struct Restore {
    int d;
    ~Restore() {
      if (d >= 0) cudaSetDevice(d);
    }
  } restore{prev};
  cudaStream_t st = (cudaStream_t)cfg->cuda_stream;
  Buf tmp(st, cfg->device);
  StageTimer tm;
  tm.on = cfg->profile != 0;
  tm.st = st;
  int64_t launches = 0;

  // offsets and poses on the device (small); the points stay where they are
  int64_t n = 0;
  std::vector<int64_t> spo_host;
  const int64_t* spo = scan_point_off;
  const double* T = poses;
  if (mem_kind == BA_MEM_HOST) {
    n = scan_point_off[n_scans];
    if (n < 0) return vfail(BA_ERR_INVALID_ARG, "scan_point_off must end at the point count");
    int64_t* d_spo = tmp.get<int64_t>(n_scans + 1);
    double* d_T = tmp.get<double>(12 * (int64_t)n_scans);
    if (!d_spo || !d_T) return vfail(BA_ERR_OOM, "voxelize inputs: out of device memory");
    VCK(cudaMemcpyAsync(d_spo, spo, sizeof(int64_t) * (n_scans + 1), cudaMemcpyHostToDevice, st), "stage");
    VCK(cudaMemcpyAsync(d_T, T, sizeof(double) * 12 * n_scans, cudaMemcpyHostToDevice, st), "stage");
    spo = d_spo;
    T = d_T;
  } else {
    VCK(cudaMemcpyAsync(&n, scan_point_off + n_scans, sizeof n, cudaMemcpyDeviceToHost, st), "read point count");
    VCK(cudaStreamSynchronize(st), "read point count");
    if (n < 0) return vfail(BA_ERR_INVALID_ARG, "scan_point_off must end at the point count");
  }
  if (n >= (1ll << 32)) return vfail(BA_ERR_CAPACITY, "at most 2^32 - 1 points per call");
  if (n > 0 && !points) return vfail(BA_ERR_INVALID_ARG, "NULL points");
  if (cfg->batch_points < 0) return vfail(BA_ERR_INVALID_ARG, "batch_points must be >= 0");
  if (!(cfg->alpha > 0.0 && cfg->alpha <= 1.0)) return vfail(BA_ERR_INVALID_ARG, "alpha must be in (0, 1]");

  // validation of the offsets and poses
  long long* bad = tmp.get<long long>(3);
  if (!bad) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
  const long long init[3] = {LLONG_MAX, LLONG_MAX, LLONG_MAX};
  VCK(cudaMemcpyAsync(bad, init, sizeof init, cudaMemcpyHostToDevice, st), "voxelize");
  check_inputs_kernel<<<blocks_for(n_scans + 1), 256, 0, st>>>(n_scans, spo, n, T, bad, bad + 1);
  ++launches;
  VCK(cudaGetLastError(), "voxelize");
  long long res[3];
  VCK(cudaMemcpyAsync(res, bad, sizeof res, cudaMemcpyDeviceToHost, st), "voxelize");
  VCK(cudaStreamSynchronize(st), "voxelize");
  if (res[0] != LLONG_MAX)
    return vfail(BA_ERR_INVALID_ARG, "scan_point_off must start at 0, not decrease and end at %lld (index %lld)",
                 (long long)n, res[0]);
  if (res[1] != LLONG_MAX) return vfail(BA_ERR_INVALID_ARG, "pose %lld is not finite", res[1]);

  std::vector<Level> lv(cfg->levels);
  int64_t n_batches = 0;
  if (n > 0) {
    double* sposes = tmp.get<double>(12 * (int64_t)n_scans);
    int* bbox = tmp.get<int>(6);
    ScanFix* fix = tmp.get<ScanFix>(n_scans);
    if (!sposes || !bbox || !fix) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
    // fixed point of the indices: 1 / d < 2^e
    // (far out of that range no pose fits and every point takes the FP64 path)
    const int e = std::min(std::max(std::ilogb(1.0 / cfg->voxel_size), -200), 200) + 1, kS = 30 - e, kp = 18 + e;
    launch_chained(scaled_poses_kernel, blocks_for(n_scans, 128), 128, 0, st, n_scans, T, 1.0 / cfg->voxel_size, kS, kp,
                   sposes, fix);
    ++launches;
    int n_sm = 0;
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, cfg->device);
    L1Ctx ctx{n_scans, spo, T, sposes, fix, kp, cfg->voxel_size, bad, bbox, n_sm > 0 ? n_sm : 1, st, &tm, &launches};
    // the adaptive loader (Sec. IV-B): batches of whole scans sized by alpha
    const int64_t B = batch_size(cfg, n, mem_kind);
    int bb[6];
    ba_status s;
    if (mem_kind == BA_MEM_DEVICE && n <= B) {
      n_batches = 1;
      s = l1_single(ctx, n, points, lv[0], bb, tmp);
    } else {
      spo_host.resize(n_scans + 1);
      if (mem_kind == BA_MEM_HOST) {
        std::copy(scan_point_off, scan_point_off + n_scans + 1, spo_host.begin());
      } else {
        VCK(cudaMemcpyAsync(spo_host.data(), scan_point_off, sizeof(int64_t) * (n_scans + 1), cudaMemcpyDeviceToHost,
                            st),
            "voxelize");
        VCK(cudaStreamSynchronize(st), "voxelize");
      }
      const std::vector<Batch> plan = plan_batches(spo_host, B);
      n_batches = (int64_t)plan.size();
      bool any_split = false;
      for (size_t k = 1; k < plan.size(); ++k)
        any_split = any_split || !std::binary_search(spo_host.begin(), spo_host.end(), plan[k].p0);
      s = l1_batched(ctx, plan, any_split, points, mem_kind, cfg->device, lv[0], bb, tmp);
    }
    if (s != BA_OK) return s;
    for (int k = 0; k < cfg->levels; ++k) {
      Level& L = lv[k];
      for (int a = 0; a < 3; ++a) {
        L.lo[a] = k == 0 ? bb[a] : half_floor(lv[k - 1].lo[a]);
        L.hi[a] = k == 0 ? bb[3 + a] : half_floor(lv[k - 1].hi[a]);
      }
      if (k > 0) L.pk = make_pack(L.lo, L.hi);
    }
    // levels 2..L (Eq. 5)
    for (int k = 1; k < cfg->levels; ++k) {
      tm.begin(BA_VOX_LEVELS);
      s = pack_bits(lv[k].pk) <= 32 ? level_up<uint32_t>(lv[k - 1], lv[k], n_scans, tmp, st, &launches)
                                    : level_up<uint64_t>(lv[k - 1], lv[k], n_scans, tmp, st, &launches);
      tm.end();
      if (s != BA_OK) return s;
    }
  }

  // voxels of every level, selection, and the output
  ba_voxels* v = new ba_voxels();
  v->device = cfg->device;
  struct Guard {
    ba_voxels** pv;
    ~Guard() {
      if (*pv) ba_voxels_destroy(*pv);
    }
  } guard{&v};
  std::vector<int64_t*> keep_obs(cfg->levels), keep_vox(cfg->levels), obs_pos(cfg->levels), vox_pos(cfg->levels);
  std::vector<int64_t> lv_nv(cfg->levels, 0), lv_no(cfg->levels, 0);
  int64_t total_v = 0, total_o = 0;
  for (int k = 0; k < cfg->levels; ++k) {
    Level& L = lv[k];
    if (L.nc == 0) continue;
    int64_t* pos = tmp.get<int64_t>(L.nc + 1);
    int64_t* scr = tmp.get<int64_t>(scan_scratch_count(L.nc + 1));
    if (!pos || !scr) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
    launch_chained(voxel_heads_kernel, blocks_for(L.nc), 256, 0, st, L.nc, L.key, pos);
    VCK(cudaGetLastError(), "voxelize");
    VCK(cudaMemsetAsync(pos + L.nc, 0, sizeof(int64_t), st), "voxelize");
    VCK(exclusive_scan_i64(pos, L.nc + 1, scr, st, &launches), "voxelize");
    VCK(cudaMemcpyAsync(&L.nv, pos + L.nc, sizeof(int64_t), cudaMemcpyDeviceToHost, st), "voxelize");
    VCK(cudaStreamSynchronize(st), "voxelize");
    L.vstart = tmp.get<int64_t>(L.nv + 1);
    keep_obs[k] = tmp.get<int64_t>(L.nv + 1);
    keep_vox[k] = tmp.get<int64_t>(L.nv + 1);
    obs_pos[k] = tmp.get<int64_t>(L.nv + 1);
    vox_pos[k] = tmp.get<int64_t>(L.nv + 1);
    int64_t* scr3 = tmp.get<int64_t>(scan_scratch_count(L.nv + 1));
    if (!L.vstart || !keep_obs[k] || !keep_vox[k] || !obs_pos[k] || !vox_pos[k] || !scr3)
      return vfail(BA_ERR_OOM, "voxelize: out of device memory");
    launch_chained(voxel_starts_kernel, blocks_for(L.nc), 256, 0, st, L.nc, L.key, pos, L.vstart, L.nv);
    launches += 2;
    tm.begin(BA_VOX_SELECT);
    float4 *rel = nullptr, *rsr = nullptr;
    uint32_t* close = nullptr;
    unsigned long long* n_close = nullptr;
    if (cfg->tau > 0.0) {
      rel = tmp.get<float4>(L.nc);
      rsr = tmp.get<float4>(2 * L.nc);
      close = tmp.get<uint32_t>(L.nv);
      n_close = tmp.get<unsigned long long>(1);
      if (!rel || !rsr || !close || !n_close) return vfail(BA_ERR_OOM, "voxelize: out of device memory");
      VCK(cudaMemsetAsync(n_close, 0, sizeof(unsigned long long), st), "voxelize");
      launch_chained(world_terms_kernel, blocks_for(L.nc, kTermThreads), kTermThreads, 0, st, L.nc, L.c, L.scan, T, pos,
                     L.vstart, rel, rsr);
      ++launches;
    }
    // tau rounded to FP32 moves the test by 2^-24 tau lambda1, inside the error band
    launch_chained(select_kernel, blocks_for(L.nv), 256, 0, st, L.nv, L.vstart, rel, rsr,
                   cfg->tau > 0.0 ? (float)cfg->tau : 0.0f, cfg->min_obs, keep_obs[k], keep_vox[k], close, n_close);
    ++launches;
    if (cfg->tau > 0.0) {
      int n_sm = 0;
      cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, cfg->device);
      const int64_t cb = std::min<int64_t>(blocks_for(L.nv, 128), (int64_t)(n_sm > 0 ? n_sm : 1) * 4);
      launch_chained(select_close_kernel, (unsigned)cb, 128, 0, st, close, n_close, L.vstart, L.c, L.scan, T, cfg->tau,
                                                        keep_obs[k], keep_vox[k]);
      ++launches;
    }
    tm.end();
    VCK(cudaGetLastError(), "voxelize select");
    VCK(cudaMemsetAsync(keep_obs[k] + L.nv, 0, sizeof(int64_t), st), "voxelize");
    VCK(cudaMemsetAsync(keep_vox[k] + L.nv, 0, sizeof(int64_t), st), "voxelize");
    VCK(cudaMemcpyAsync(obs_pos[k], keep_obs[k], sizeof(int64_t) * (L.nv + 1), cudaMemcpyDeviceToDevice, st),
        "voxelize");
    VCK(cudaMemcpyAsync(vox_pos[k], keep_vox[k], sizeof(int64_t) * (L.nv + 1), cudaMemcpyDeviceToDevice, st),
        "voxelize");
    VCK(exclusive_scan_i64(obs_pos[k], L.nv + 1, scr3, st, &launches), "voxelize");
    VCK(exclusive_scan_i64(vox_pos[k], L.nv + 1, scr3, st, &launches), "voxelize");
    VCK(cudaMemcpyAsync(&lv_no[k], obs_pos[k] + L.nv, sizeof(int64_t), cudaMemcpyDeviceToHost, st), "voxelize");
    VCK(cudaMemcpyAsync(&lv_nv[k], vox_pos[k] + L.nv, sizeof(int64_t), cudaMemcpyDeviceToHost, st), "voxelize");
    VCK(cudaStreamSynchronize(st), "voxelize");
    total_v += lv_nv[k];
    total_o += lv_no[k];
  }
  v->n_voxels = total_v;
  v->n_obs = total_o;
  // the result lives in the library pool too (freed by ba_voxels_destroy)
  cudaMemPool_t pool = library_pool(cfg->device);
  auto out_alloc = [&](void** p, size_t bytes) {
    return pool ? cudaMallocFromPoolAsync(p, bytes, pool, st) : cudaMalloc(p, bytes);
  };
  v->pooled = pool != nullptr;
  if (out_alloc((void**)&v->voxel_off, sizeof(int64_t) * (total_v + 1)) != cudaSuccess ||
      out_alloc((void**)&v->obs_scan, sizeof(int32_t) * (total_o > 0 ? total_o : 1)) != cudaSuccess ||
      out_alloc((void**)&v->agg, sizeof(double) * 10 * (total_o > 0 ? total_o : 1)) != cudaSuccess ||
      out_alloc((void**)&v->level, sizeof(int32_t) * (total_v > 0 ? total_v : 1)) != cudaSuccess ||
      out_alloc((void**)&v->index, sizeof(int32_t) * 3 * (total_v > 0 ? total_v : 1)) != cudaSuccess) {
    cudaGetLastError();
    return vfail(BA_ERR_OOM, "voxelize output: out of device memory");
  }
  VCK(cudaMemsetAsync(v->voxel_off, 0, sizeof(int64_t), st), "voxelize");
  int64_t vb = 0, ob = 0;
  for (int k = 0; k < cfg->levels; ++k) {
    const Level& L = lv[k];
    if (L.nv == 0) continue;
    tm.begin(BA_VOX_EMIT);
    launch_chained(emit_kernel, blocks_for(L.nv), 256, 0, st, L.nv, L.vstart, L.key, L.pk, L.scan, L.c, obs_pos[k],
                   vox_pos[k], keep_vox[k], k + 1, vb, ob, v->voxel_off, v->obs_scan, v->agg, v->level, v->index);
    tm.end();
    ++launches;
    VCK(cudaGetLastError(), "voxelize emit");
    vb += lv_nv[k];
    ob += lv_no[k];
  }
  VCK(cudaStreamSynchronize(st), "voxelize");
  v->launches = launches;
  v->batches = n_batches;
  tm.collect(v->stage_ms);
  *out = v;
  v = nullptr;  // handed out
  return BA_OK;
}

ba_status ba_voxels_size(const ba_voxels* v, int64_t* n_voxels, int64_t* n_obs) {
  if (!v) return BA_ERR_INVALID_ARG;
  if (n_voxels) *n_voxels = v->n_voxels;
  if (n_obs) *n_obs = v->n_obs;
  return BA_OK;
}

ba_status ba_voxels_read(const ba_voxels* v, int64_t* voxel_off, int32_t* obs_scan, double* agg, int32_t* level,
                         int32_t* index, int32_t mem_kind) {
  if (!v) return BA_ERR_INVALID_ARG;
  if (mem_kind != BA_MEM_HOST && mem_kind != BA_MEM_DEVICE) return vfail(BA_ERR_INVALID_ARG, "bad mem_kind");
  const cudaMemcpyKind kind = mem_kind == BA_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
  int prev = -1;
  cudaGetDevice(&prev);
  if (cudaSetDevice(v->device) != cudaSuccess) return vfail(BA_ERR_CUDA, "cannot use device %d", v->device);
  cudaError_t e = cudaSuccess;
  if (voxel_off) e = cudaMemcpy(voxel_off, v->voxel_off, sizeof(int64_t) * (v->n_voxels + 1), kind);
  if (e == cudaSuccess && obs_scan && v->n_obs) e = cudaMemcpy(obs_scan, v->obs_scan, sizeof(int32_t) * v->n_obs, kind);
  if (e == cudaSuccess && agg && v->n_obs) e = cudaMemcpy(agg, v->agg, sizeof(double) * 10 * v->n_obs, kind);
  if (e == cudaSuccess && level && v->n_voxels) e = cudaMemcpy(level, v->level, sizeof(int32_t) * v->n_voxels, kind);
  if (e == cudaSuccess && index && v->n_voxels)
    e = cudaMemcpy(index, v->index, sizeof(int32_t) * 3 * v->n_voxels, kind);
  if (prev >= 0) cudaSetDevice(prev);
  if (e != cudaSuccess) return vfail(BA_ERR_CUDA, "read voxels: %s", cudaGetErrorString(e));
  return BA_OK;
}

int64_t ba_voxels_kernel_launches(const ba_voxels* v) { return v ? v->launches : 0; }

int64_t ba_voxels_batches(const ba_voxels* v) { return v ? v->batches : 0; }

ba_status ba_voxels_stage_ms(const ba_voxels* v, int32_t stage, double* ms) {
  if (!v || !ms || stage < 0 || stage >= BA_VOX_STAGES) return BA_ERR_INVALID_ARG;
  *ms = v->stage_ms[stage];
  return BA_OK;
}

void ba_voxels_destroy(ba_voxels* v) {
  if (!v) return;
  int prev = -1;
  cudaGetDevice(&prev);
  cudaSetDevice(v->device);
  void* ptrs[5] = {v->voxel_off, v->obs_scan, v->agg, v->level, v->index};
  for (void* p : ptrs) {
    if (!p) continue;
    if (v->pooled)
      cudaFreeAsync(p, nullptr);
    else
      cudaFree(p);
  }
  if (prev >= 0) cudaSetDevice(prev);
  delete v;
}

}  // extern "C"
