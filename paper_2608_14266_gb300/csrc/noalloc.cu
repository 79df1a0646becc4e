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

constexpr int kThreads = 256;
constexpr int kLanes = 4;                      // threads per voxel
constexpr int kVoxels = kThreads / kLanes;     // voxels per block
constexpr int64_t kMaxPairs = BA_NOALLOC_MAX_VOXELS / (2 * kVoxels);  // two blocks add into one partial
static_assert(BA_NOALLOC_MAX_VOXELS % (2 * kVoxels) == 0, "capacity must be a whole number of partials");

// scratch shared by every call on a device: partials, then the error word
static __device__ __align__(256) double g_noalloc_scratch[kMaxPairs + 32];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
bool g_ready[kMaxDevices];
double* g_ptr[kMaxDevices];

// Four lanes per voxel over the caller's voxel-major CSR, each every fourth
// observation: posed cluster means q = R m + t, anchored sums about the
// voxel's first q, covariance, smallest eigenvalue (the voxel's cost, Eq. 1).
// Invalid offsets or scan indices set the error word and leave the voxel out.
//
// Bound: the FP64 pipe (~70 operations an observation, a warp instruction 64
// cycles of its scheduler whatever its active lanes).  A block takes its 64
// voxels in order of their lengths, so that the eight of a warp are about as
// long, and solves their eigenproblems in two full warps.  40,003 voxels of
// 2-40 observations: 352 us with one thread per voxel (warps as long as their
// longest voxel, each scheduler with one warp), now 206 us with the FP64 pipe
// 85% active.
__global__ void __launch_bounds__(kThreads) noalloc_cost_kernel(int64_t n_voxels, int64_t n_obs,
                                                                const int64_t* __restrict__ off,
                                                                const int32_t* __restrict__ obs_scan,
                                                                const double* __restrict__ agg,
                                                                const double* __restrict__ poses, int32_t n_scans,
                                                                double* __restrict__ lam0_out, double* scratch) {
  __shared__ double sums[10][kVoxels];
  __shared__ int valid[kVoxels];
  __shared__ double red[kVoxels / 32];
  __shared__ int s_cnt[32], s_order[mmba::kOrderBlock];
  static_assert(mmba::kOrderBlock == kThreads, "the ordering takes one item per thread");
  unsigned long long* err = reinterpret_cast<unsigned long long*>(scratch + kMaxPairs);
  const int64_t v0 = (int64_t)blockIdx.x * kVoxels;
  {
    // the block's voxels by length; the threads past them come last
    const int64_t i = v0 + threadIdx.x;
    int64_t len = threadIdx.x < kVoxels && i < n_voxels ? off[i + 1] - off[i] : 0;
    len = len < 0 ? 0 : len;
    mmba::block_order_by_key(threadIdx.x >= kVoxels ? 31 : len < 60 ? (int)(len >> 1) : 30, s_cnt, s_order);
  }
  const int w = threadIdx.x >> 5;
  {
    // ranks dealt to the warps so that each scheduler's two take short and long ones
    const int wr = w < 4 ? w : 11 - w;
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
      if (ok) {  // the anchor, formed by every lane
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
      const double dx = fma(P[0], c[6], fma(P[1], c[7], fma(P[2], c[8], P[9]))) - ax;
      const double dy = fma(P[3], c[6], fma(P[4], c[7], fma(P[5], c[8], P[10]))) - ay;
      const double dz = fma(P[6], c[6], fma(P[7], c[7], fma(P[8], c[8], P[11]))) - az;
      const double N = c[9];
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
      const double inv = 1.0 / acc[0];
      const double cx = acc[1] * inv, cy = acc[2] * inv, cz = acc[3] * inv;
      sums[0][vl] = acc[0];
      sums[1][vl] = fma(-cx, cx, acc[4] * inv);
      sums[2][vl] = fma(-cx, cy, acc[5] * inv);
      sums[3][vl] = fma(-cx, cz, acc[6] * inv);
      sums[4][vl] = fma(-cy, cy, acc[7] * inv);
      sums[5][vl] = fma(-cy, cz, acc[8] * inv);
      sums[6][vl] = fma(-cz, cz, acc[9] * inv);
      const unsigned group = ((1u << kLanes) - 1u) << (threadIdx.x & 31 & ~(kLanes - 1));
      valid[vl] = (bad & group) == 0u;
    }
  }
  __syncthreads();
  // the eigenproblems: two warps, on other schedulers from block to block
  const int first = (int)(blockIdx.x & 3) * 2;
  if (w - first != 0 && w - first != 1) return;
  const int vl = threadIdx.x - 32 * first;
  const int64_t i = v0 + vl;
  double lam0 = 0.0;
  if (i < n_voxels) {
    const bool ok = valid[vl] != 0;
    if (ok && sums[0][vl] > 0.0) {
      const double A[6] = {sums[1][vl], sums[2][vl], sums[3][vl], sums[4][vl], sums[5][vl], sums[6][vl]};
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
  asm volatile("bar.sync 1, 64;" ::: "memory");  // the two warps
  // (0 + x) + y rounds as (0 + y) + x, so the order of the two blocks does not matter
  if (threadIdx.x == 32 * first) atomicAdd(scratch + (blockIdx.x >> 1), red[0] + red[1]);
}

__global__ void noalloc_reset_kernel(double* scratch, int64_t n_partials) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n_partials) scratch[k] = 0.0;
  if (k == 0) *reinterpret_cast<unsigned long long*>(scratch + kMaxPairs) = ~0ull;
}

// Sums the partials in a fixed order; a recorded error makes the cost NaN.
__global__ void __launch_bounds__(256) noalloc_sum_kernel(int64_t n_partials, const double* scratch, double* cost_out) {
  __shared__ double red[256 / 32];
  double v = 0.0;
  for (int64_t k = threadIdx.x; k < n_partials; k += 256) v += scratch[k];
  const double tot = mmba::block_sum<256>(v, red);
  if (threadIdx.x == 0) {
    const unsigned long long e = *reinterpret_cast<const unsigned long long*>(scratch + kMaxPairs);
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
  const int64_t blocks = (n_voxels + kVoxels - 1) / kVoxels;
  // an error left pending by earlier, unrelated work on this thread is not
  // this call's to report: clear it, then check each launch on its own
  (void)cudaGetLastError();
  const int64_t partials = (blocks + 1) / 2;
  noalloc_reset_kernel<<<(unsigned)((partials + 255) / 256), 256, 0, s>>>(scratch, partials);
  if (cudaGetLastError() != cudaSuccess) return BA_ERR_CUDA;
  noalloc_cost_kernel<<<(unsigned)blocks, kThreads, 0, s>>>(n_voxels, n_obs, voxel_offsets, obs_scan, agg_centred,
                                                            poses, n_scans, lambda0_out, scratch);
  if (cudaGetLastError() != cudaSuccess) return BA_ERR_CUDA;
  noalloc_sum_kernel<<<1, 256, 0, s>>>(partials, scratch, cost_out);
  return cudaGetLastError() == cudaSuccess ? BA_OK : BA_ERR_CUDA;
}
