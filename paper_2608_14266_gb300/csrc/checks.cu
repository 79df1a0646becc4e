// Device-side self-checks of helpers whose results must match a hardware
// reference bit for bit (run by the tests on the GPU).
#include <cuda_runtime.h>

#include "../../include/ba.h"
#include "fixed_sums.cuh"
#include "mmba_internal.cuh"
#include "mmba_kernels.h"

namespace {

__device__ inline unsigned long long mix64(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

// Bit patterns: random doubles over the whole binary32 range and beyond,
// values next to rounding ties, and special values; each is converted both
// ways by the integer helpers and by the hardware.
__global__ void conversion_check_kernel(long long n, unsigned long long seed, unsigned long long* bad) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const unsigned long long r = mix64(seed + 0x9e3779b97f4a7c15ull * (unsigned long long)(i + 1));
  double x;
  switch (i % 4) {
    case 0:  // any exponent around the binary32 range (incl. subnormal and overflow results)
      x = __longlong_as_double((long long)((r & 0x800fffffffffffffull) |
                                           ((unsigned long long)(1023 - 160 + (int)((r >> 52) % 330)) << 52)));
      break;
    case 1: {  // near and exactly at ties: low 29 fraction bits around 0x10000000
      const unsigned long long low = 0x10000000ull + (long long)((r >> 40) % 5) - 2;
      x = __longlong_as_double((long long)(((r & 0x800fffffe0000000ull) | low) |
                                           ((unsigned long long)(1023 + (int)((r >> 52) % 60) - 30) << 52)));
      break;
    }
    case 2:  // values of the sizes the set-up converts (metres, squared metres)
      x = (double)(long long)(r >> 11) * 0x1.0p-53 * 4000.0 - 2000.0;
      break;
    default: {  // special values and the extremes
      const double sp[8] = {0.0, -0.0, 1.0 / 0.0, -1.0 / 0.0, 3.4028234663852886e38, 3.4028235677973366e38,
                            1.1754943508222875e-38, 1.401298464324817e-45};
      x = sp[(r >> 7) % 8];
      break;
    }
  }
  const float a = mmba::f64_to_f32(x), b = (float)x;
  if (__float_as_uint(a) != __float_as_uint(b) && !(isnan(a) && isnan(b))) atomicAdd(bad, 1ull);
  const double c = mmba::f32_to_f64(b), d = (double)b;
  if (__double_as_longlong(c) != __double_as_longlong(d) && !(isnan(c) && isnan(d))) atomicAdd(bad + 1, 1ull);
}

// |1 - d y| in units of 2^-53, y the reciprocal of d by the solve's recip_pivot
// (worst[0]) and of a whole number by the clusters' recip_count (worst[1]), as
// the bits of a non-negative double (whose order is the numbers').  A correctly
// rounded reciprocal is within 1.  Where the pivot's exponent makes it divide, the
// division's own bits are asked for.
__global__ void reciprocal_check_kernel(long long n, unsigned long long seed, unsigned long long* worst) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const unsigned long long r = mix64(seed + 0x9e3779b97f4a7c15ull * (unsigned long long)(i + 1));
  unsigned long long m = r & 0xfffffffffffffull;  // fraction
  int ex = 1023;
  switch (i % 4) {
    case 0:  // any normal pivot
      ex = 1 + (int)((r >> 52) % 2046);
      break;
    case 1:  // both ends of a binade, and powers of two
      m = (r >> 60) & 1 ? 0xfffffffffffffull - (m >> 46) : m >> 46;
      ex = 1023 + (int)((r >> 52) % 200) - 100;
      break;
    case 2:  // the exponents at which it changes to a division
      ex = 1023 + ((r >> 60) & 1 ? 1 : -1) * (998 + (int)((r >> 52) % 6));
      break;
    default:  // the sizes of a Hessian's diagonal
      ex = 1023 + (int)((r >> 52) % 60) - 20;
      break;
  }
  const double d = __longlong_as_double((long long)(m | ((unsigned long long)ex << 52)));
  const double y = mmba::recip_pivot(d);
  const double e = ex - 1023 < -1000 || ex - 1023 > 1000
                       ? (__double_as_longlong(y) == __double_as_longlong(1.0 / d) ? 0.0 : 1e300)
                       : fabs(fma(-d, y, 1.0)) * 0x1p53;
  atomicMax(worst, (unsigned long long)__double_as_longlong(e));
  const int c = 1 + (int)(r % (1u << 24));
  const double nd = (double)c;
  atomicMax(worst + 1, (unsigned long long)__double_as_longlong(
                           fabs(fma(-nd, mmba::recip_count(nd, (float)c), 1.0)) * 0x1p53));
}

template <typename K>
__global__ void sort_check_fill_kernel(long long n, int bits, unsigned long long seed, K* keys, K* kept) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  unsigned long long r = mix64(seed + 0x9e3779b97f4a7c15ull * (unsigned long long)(i + 1));
  if (r >> 63) r &= 7;  // half of them on a few keys
  keys[i] = kept[i] = (K)(r & (bits < 64 ? (1ull << bits) - 1ull : ~0ull));
}

// pairs out of order, not in the order they came in among equal keys, or not pairs of the input
template <typename K>
__global__ void sort_check_kernel(long long n, const K* keys, const uint32_t* vals, const K* kept,
                                  unsigned long long* bad) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t v = vals[i];
  const bool wrong = v >= n || kept[v] != keys[i] ||
                     (i > 0 && (keys[i - 1] > keys[i] || (keys[i - 1] == keys[i] && vals[i - 1] >= v)));
  if (wrong) atomicAdd(bad, 1ull);
}

template <typename K, typename Sort>
cudaError_t check_sort(int64_t n, int bits, bool wait, uint64_t seed, Sort sort, unsigned long long* bad) {
  K *keys = nullptr, *tk = nullptr, *kept = nullptr;
  uint32_t *vals = nullptr, *tv = nullptr;
  int64_t* scratch = nullptr;
  unsigned long long* d = nullptr;
  int64_t launches = 0;
  const unsigned blocks = (unsigned)((n + 255) / 256);
  cudaError_t e = cudaMalloc(&keys, sizeof(K) * n);
  if (e == cudaSuccess) e = cudaMalloc(&tk, sizeof(K) * n);
  if (e == cudaSuccess) e = cudaMalloc(&kept, sizeof(K) * n);
  if (e == cudaSuccess) e = cudaMalloc(&vals, 4 * n);
  if (e == cudaSuccess) e = cudaMalloc(&tv, 4 * n);
  if (e == cudaSuccess) e = cudaMalloc(&scratch, 8 * mmba::radix_scratch_count(n));
  if (e == cudaSuccess) e = cudaMalloc(&d, sizeof *d);
  if (e == cudaSuccess) e = cudaMemset(d, 0, sizeof *d);
  if (e == cudaSuccess) {
    sort_check_fill_kernel<K><<<blocks, 256>>>((long long)n, bits, (unsigned long long)seed, keys, kept);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = sort(&keys, &vals, &tk, &tv, n, bits, true, scratch, (cudaStream_t) nullptr, &launches, wait);
  if (e == cudaSuccess) {
    sort_check_kernel<K><<<blocks, 256>>>((long long)n, keys, vals, kept, d);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(bad, d, sizeof *d, cudaMemcpyDeviceToHost);
  cudaFree(keys);
  cudaFree(tk);
  cudaFree(kept);
  cudaFree(vals);
  cudaFree(tv);
  cudaFree(scratch);
  cudaFree(d);
  return e;
}

}  // namespace

extern "C" ba_status ba_check_reciprocals(int32_t device, int64_t n, uint64_t seed, double* worst) {
  if (n < 1 || !worst) return BA_ERR_INVALID_ARG;
  int prev = -1;
  cudaGetDevice(&prev);
  if (cudaSetDevice(device) != cudaSuccess) return BA_ERR_CUDA;
  unsigned long long* d = nullptr;
  cudaError_t e = cudaMalloc(&d, 2 * sizeof *d);
  if (e == cudaSuccess) e = cudaMemset(d, 0, 2 * sizeof *d);
  if (e == cudaSuccess) {
    reciprocal_check_kernel<<<(unsigned)((n + 255) / 256), 256>>>((long long)n, (unsigned long long)seed, d);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(worst, d, 2 * sizeof *d, cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (prev >= 0) cudaSetDevice(prev);
  return e == cudaSuccess ? BA_OK : BA_ERR_CUDA;
}

extern "C" ba_status ba_check_sort(int32_t device, int64_t n, int32_t bits, int32_t wait, uint64_t seed,
                                   uint64_t* mismatches) {
  if (n < 1 || n >= (1ll << 31) || bits < 0 || bits > 64 || !mismatches) return BA_ERR_INVALID_ARG;
  int prev = -1;
  cudaGetDevice(&prev);
  if (cudaSetDevice(device) != cudaSuccess) return BA_ERR_CUDA;
  unsigned long long bad = 0;
  const cudaError_t e = bits <= 32 ? check_sort<uint32_t>(n, bits, wait != 0, seed, mmba::radix_sort_pairs, &bad)
                                   : check_sort<uint64_t>(n, bits, wait != 0, seed, mmba::radix_sort_pairs64, &bad);
  if (prev >= 0) cudaSetDevice(prev);
  if (e != cudaSuccess) return BA_ERR_CUDA;
  *mismatches = bad;
  return BA_OK;
}

extern "C" ba_status ba_check_conversions(int32_t device, int64_t n, uint64_t seed, uint64_t* mismatches) {
  if (n < 1 || !mismatches) return BA_ERR_INVALID_ARG;
  int prev = -1;
  cudaGetDevice(&prev);
  if (cudaSetDevice(device) != cudaSuccess) return BA_ERR_CUDA;
  unsigned long long* d = nullptr;
  unsigned long long h[2] = {0, 0};
  cudaError_t e = cudaMalloc(&d, sizeof h);
  if (e == cudaSuccess) e = cudaMemset(d, 0, sizeof h);
  if (e == cudaSuccess) {
    conversion_check_kernel<<<(unsigned)((n + 255) / 256), 256>>>((long long)n, (unsigned long long)seed, d);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost);
  if (d) cudaFree(d);
  if (prev >= 0) cudaSetDevice(prev);
  if (e != cudaSuccess) return BA_ERR_CUDA;
  mismatches[0] = h[0];
  mismatches[1] = h[1];
  return BA_OK;
}
