// Allocation-free cost evaluation (ba_eval_cost_noalloc, see include/ba.h).
//
// Some callers cannot allocate device memory at the point where they need a
// cost: a mapping loop running on a vehicle under a fixed memory budget
// (cudaMalloc/cudaFree may synchronise the device and stall the loop), or a
// host application whose own allocator has already reserved the GPU memory.
// This entry point therefore takes only caller-owned inputs and outputs; its
// scratch (the per-block partial sums of the cost and an error word) is a
// file-scope __device__ array that every GPU loading the library holds until
// the process exits.  Host code may not use the array's name as a device
// address, so the address is fetched once per device with
// cudaGetSymbolAddress and passed to the kernels.  The cached address belongs
// to the device's context of that moment: after cudaDeviceReset (or anything
// else that tears down and recreates the primary context) the library's
// module is loaded anew and the cache is stale, so the entry point must not
// be used across a device reset.
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "../../include/ba.h"
#include "block_order.cuh"
#include "mmba_internal.cuh"

namespace {

template <int kLanes>
constexpr int kThreadsOf = kLanes == 1 ? 128 : 256;  // per block
constexpr int64_t kMaxPartials = BA_NOALLOC_MAX_VOXELS / 128;  // the cost's partial sums: of 128 voxels or more
static_assert(BA_NOALLOC_MAX_VOXELS % 128 == 0, "capacity must be a whole number of partials");

// scratch shared by every call on a device: partials, then the error word
static __device__ __align__(256) double g_noalloc_scratch[kMaxPartials + 32];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
bool g_ready[kMaxDevices];
double* g_ptr[kMaxDevices];

// kLanes lanes per voxel over the caller's voxel-major CSR, each every kLanes-th
// observation: posed cluster means q = R m + t, anchored sums about the
// voxel's first q, covariance, smallest eigenvalue (the voxel's cost, Eq. 1).
// Invalid offsets or scan indices set the error word and leave the voxel out.
//
// Bound: the FP64 pipe (~70 operations an observation, a warp instruction 64
// cycles of its scheduler whatever its active lanes).  A block takes its
// voxels in order of their lengths, so that those of a warp are about as
// long, and solves their eigenproblems in full warps.  Four lanes to a voxel:
// 40,003 voxels of 2-40 observations in 206 us with the FP64 pipe 85% active
// (352 us with one thread per voxel in input order: warps as long as their
// longest voxel, each scheduler with one warp).  One lane where voxels are many
// and short (noalloc_lanes).
template <int kLanes>
__global__ void __launch_bounds__(kThreadsOf<kLanes>) noalloc_cost_kernel(int64_t n_voxels, int64_t n_obs,
                                                                const int64_t* __restrict__ off,
                                                                const int32_t* __restrict__ obs_scan,
                                                                const double* __restrict__ agg,
                                                                const double* __restrict__ poses, int32_t n_scans,
                                                                double* __restrict__ lam0_out, double* scratch) {
  constexpr int kThreads = kThreadsOf<kLanes>, kVoxels = kThreads / kLanes;
  __shared__ double sums[10][kVoxels];
  __shared__ int valid[kVoxels];
  __shared__ double red[kVoxels / 32];
  __shared__ int s_cnt[32], s_order[mmba::kOrderBlock];
  static_assert(kThreads <= mmba::kOrderBlock, "the ordering takes one item per thread");
  unsigned long long* err = reinterpret_cast<unsigned long long*>(scratch + kMaxPartials);
  const int64_t v0 = (int64_t)blockIdx.x * kVoxels;
  {
    // the block's voxels by length; the threads past them come last
    const int64_t i = v0 + threadIdx.x;
    int64_t len = threadIdx.x < kVoxels && i < n_voxels ? off[i + 1] - off[i] : 0;
    len = len < 0 ? 0 : len;
    const int key = kLanes == 1 ? (int)(len < 31 ? len : 31) : len < 60 ? (int)(len >> 1) : 30;
    mmba::block_order_by_key(threadIdx.x >= kVoxels ? 31 : key, s_cnt, s_order);
  }
  const int w = threadIdx.x >> 5;
  {
    // ranks dealt to the warps so that each scheduler's two take short and long ones
    const int wr = kLanes == 1 || w < 4 ? w : 11 - w;
    const int vl = s_order[wr * (32 / kLanes) + (threadIdx.x & 31) / kLanes];
    const int sub = threadIdx.x & (kLanes - 1);
    const int64_t i = v0 + vl;
    const bool in = i < n_voxels;
    const int64_t a = in ? off[i] : 0, b = in ? off[i + 1] : 0;
    bool ok = in && a >= 0 && b > a && b <= n_obs;
    double n = 0.0, ax = 0.0, ay = 0.0, az = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
    double m00 = 0.0, m01 = 0.0, m02 = 0.0, m11 = 0.0, m12 = 0.0, m22 = 0.0;
    if (ok) {
      const int32_t j = obs_scan[a];
      ok = j >= 0 && j < n_scans;
      if (ok && kLanes > 1) {  // the anchor, formed by every lane
        const double* P = poses + 12 * (int64_t)j;
        const double* c = agg + 10 * a;
        ax = fma(P[0], c[6], fma(P[1], c[7], fma(P[2], c[8], P[9])));
        ay = fma(P[3], c[6], fma(P[4], c[7], fma(P[5], c[8], P[10])));
        az = fma(P[6], c[6], fma(P[7], c[7], fma(P[8], c[8], P[11])));
      }
    }
    for (int64_t o = a + sub; ok && o < b; o += kLanes) {
      const int32_t j = obs_scan[o];
      if (j < 0 || j >= n_scans) {
        ok = false;
        break;
      }
      const double* P = poses + 12 * (int64_t)j;
      const double* c = agg + 10 * o;
      const double qx = fma(P[0], c[6], fma(P[1], c[7], fma(P[2], c[8], P[9])));
      const double qy = fma(P[3], c[6], fma(P[4], c[7], fma(P[5], c[8], P[10])));
      const double qz = fma(P[6], c[6], fma(P[7], c[7], fma(P[8], c[8], P[11])));
      if (kLanes == 1 && o == a) {
        ax = qx;
        ay = qy;
        az = qz;
      }
      const double dx = qx - ax, dy = qy - ay, dz = qz - az, N = c[9];
      // R S R^T from the packed scatter (xx, xy, xz, yy, yz, zz)
      double RS[3][3];
      const double S[3][3] = {{c[0], c[1], c[2]}, {c[1], c[3], c[4]}, {c[2], c[4], c[5]}};
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int k = 0; k < 3; ++k) RS[r][k] = fma(P[3 * r], S[0][k], fma(P[3 * r + 1], S[1][k], P[3 * r + 2] * S[2][k]));
      auto add = [&](double m, int r, int k, double nd, double d) {
        return fma(RS[r][0], P[3 * k], fma(RS[r][1], P[3 * k + 1], fma(RS[r][2], P[3 * k + 2], fma(nd, d, m))));
      };
      const double Nx = N * dx, Ny = N * dy, Nz = N * dz;
      m00 = add(m00, 0, 0, Nx, dx);
      m01 = add(m01, 0, 1, Nx, dy);
      m02 = add(m02, 0, 2, Nx, dz);
      m11 = add(m11, 1, 1, Ny, dy);
      m12 = add(m12, 1, 2, Ny, dz);
      m22 = add(m22, 2, 2, Nz, dz);
      sx += Nx;
      sy += Ny;
      sz += Nz;
      n += N;
    }
    const unsigned bad = __ballot_sync(0xffffffffu, !ok);
    double acc[10] = {n, sx, sy, sz, m00, m01, m02, m11, m12, m22};
#pragma unroll
    for (int o = 1; o < kLanes; o <<= 1)
#pragma unroll
      for (int q = 0; q < 10; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
    if (sub == 0) {
#pragma unroll
      for (int q = 0; q < 10; ++q) sums[q][vl] = acc[q];
      const unsigned group = ((1u << kLanes) - 1u) << (threadIdx.x & 31 & ~(kLanes - 1));
      valid[vl] = (bad & group) == 0u;
    }
  }
  __syncthreads();
  // the eigenproblems, a voxel to a thread of kVoxels / 32 warps: with four lanes
  // two, on other schedulers from block to block
  constexpr int kEigWarps = kVoxels / 32;
  const int first = kLanes == 1 ? 0 : (int)(blockIdx.x & 3) * kEigWarps;
  if (w < first || w >= first + kEigWarps) return;
  const int vl = threadIdx.x - 32 * first;
  const int64_t i = v0 + vl;
  double lam0 = 0.0;
  if (i < n_voxels) {
    const bool ok = valid[vl] != 0;
    const double n = sums[0][vl];
    if (ok && n > 0.0) {
      const double inv = 1.0 / n;
      const double cx = sums[1][vl] * inv, cy = sums[2][vl] * inv, cz = sums[3][vl] * inv;
      const double A[6] = {fma(-cx, cx, sums[4][vl] * inv), fma(-cx, cy, sums[5][vl] * inv),
                           fma(-cx, cz, sums[6][vl] * inv), fma(-cy, cy, sums[7][vl] * inv),
                           fma(-cy, cz, sums[8][vl] * inv), fma(-cz, cz, sums[9][vl] * inv)};
      double lam[3], V[9];
      mmba::eig3_sym(A, lam, V);
      lam0 = lam[0];
    } else {
      atomicMin(err, (unsigned long long)i);
    }
    if (lam0_out) lam0_out[i] = ok ? lam0 : __longlong_as_double(0x7ff8000000000000ll);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lam0 += __shfl_down_sync(0xffffffffu, lam0, o);
  if ((threadIdx.x & 31) == 0) red[w - first] = lam0;
  asm volatile("bar.sync 1, %0;" ::"n"(kVoxels) : "memory");  // these warps
  if (threadIdx.x == 32 * first) {
    double tot = red[0];
#pragma unroll
    for (int q = 1; q < kEigWarps; ++q) tot += red[q];
    // two blocks of 64 voxels share a partial: (0 + x) + y rounds as (0 + y) + x, so
    // their order does not matter
    atomicAdd(scratch + (kLanes == 1 ? blockIdx.x : blockIdx.x >> 1), tot);
  }
}

// Lanes per voxel: one where voxels are many and short, so that most of four
// would be idle.  Us a call with four / one: 30,000 voxels of 1-2 observations 71
// / 41, of 4-6 96 / 58; 100,000 of 2-3 140 / 104, of 10-14 279 / 248; 300,000 of
// 4-6 534 / 356; but 5,000 of 5-12 39 / 57, 40,000 of 2-40 200 / 240.
int noalloc_lanes(int64_t n_voxels, int64_t n_obs) { return n_voxels >= 25000 && n_obs <= 14 * n_voxels ? 1 : 4; }

__global__ void noalloc_reset_kernel(double* scratch, int64_t n_partials) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n_partials) scratch[k] = 0.0;
  if (k == 0) *reinterpret_cast<unsigned long long*>(scratch + kMaxPartials) = ~0ull;
}

// Sums the partials in a fixed order; a recorded error makes the cost NaN.
__global__ void __launch_bounds__(256) noalloc_sum_kernel(int64_t n_partials, const double* scratch, double* cost_out) {
  __shared__ double red[256 / 32];
  double v = 0.0;
  for (int64_t k = threadIdx.x; k < n_partials; k += 256) v += scratch[k];
  const double tot = mmba::block_sum<256>(v, red);
  if (threadIdx.x == 0) {
    const unsigned long long e = *reinterpret_cast<const unsigned long long*>(scratch + kMaxPartials);
    *cost_out = e == ~0ull ? tot : __longlong_as_double(0x7ff8000000000000ll);
  }
}

}  // namespace

extern "C" ba_status ba_eval_cost_noalloc(int32_t n_scans, int64_t n_voxels, int64_t n_obs,
                                          const int64_t* voxel_offsets, const int32_t* obs_scan,
                                          const double* agg_centred, const double* poses, double* cost_out,
                                          double* lambda0_out, void* stream) {
  if (n_scans < 1 || n_voxels < 1 || n_obs < n_voxels) return BA_ERR_INVALID_ARG;
  if (n_voxels > BA_NOALLOC_MAX_VOXELS) return BA_ERR_CAPACITY;
  if (!voxel_offsets || !obs_scan || !agg_centred || !poses || !cost_out) return BA_ERR_INVALID_ARG;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return BA_ERR_CUDA;
  double* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_ready[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
        cudaGetLastError();
        return BA_ERR_CUDA;
      }
      g_ptr[dev] = static_cast<double*>(p);
      g_ready[dev] = true;
    }
    scratch = g_ptr[dev];
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int lanes = noalloc_lanes(n_voxels, n_obs);
  const int threads = lanes == 1 ? kThreadsOf<1> : kThreadsOf<4>;
  const int64_t per = threads / lanes, blocks = (n_voxels + per - 1) / per;
  // an error left pending by earlier, unrelated work on this thread is not
  // this call's to report: clear it, then check each launch on its own
  (void)cudaGetLastError();
  const int64_t partials = lanes == 1 ? blocks : (blocks + 1) / 2;
  noalloc_reset_kernel<<<(unsigned)((partials + 255) / 256), 256, 0, s>>>(scratch, partials);
  if (cudaGetLastError() != cudaSuccess) return BA_ERR_CUDA;
  const auto kernel = lanes == 1 ? noalloc_cost_kernel<1> : noalloc_cost_kernel<4>;
  kernel<<<(unsigned)blocks, threads, 0, s>>>(n_voxels, n_obs, voxel_offsets, obs_scan, agg_centred, poses, n_scans,
                                              lambda0_out, scratch);
  if (cudaGetLastError() != cudaSuccess) return BA_ERR_CUDA;
  noalloc_sum_kernel<<<1, 256, 0, s>>>(partials, scratch, cost_out);
  return cudaGetLastError() == cudaSuccess ? BA_OK : BA_ERR_CUDA;
}
