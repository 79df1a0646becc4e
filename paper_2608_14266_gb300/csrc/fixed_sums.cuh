// Exact integer sums of point coordinates in fixed point, shared by the point
// clusters of observations (layout.cu) and of voxelised scans (voxelize.cu).
//
// Coordinates are whole steps of 2^-F (F from the first point's largest
// exponent); offsets d from the first point below 2^54 steps are split at 27
// bits into two 32-bit halves, and each product of halves goes into a 64-bit
// sum of its own, one multiply-add each: 21 a point for the six entries of
// sum d d^T and the three of sum d, on the integer pipe (GB300's FP64 pipe runs
// at 1/64 of FP32).  Both halves are below 2^27 in size, a pair of cross
// products is below 2^55, so kHalfPoints points stay below 2^63.
#pragma once
#include <cuda_runtime.h>

#include "mmba_internal.cuh"

namespace mmba {

constexpr int kHalfPoints = 254;

// round(p 2^F) to the nearest integer (halves away from zero); ok is cleared
// when the result would reach 2^62
__device__ __forceinline__ long long fix_round(double p, int F, bool& ok) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(p);
  const int E = (int)((b >> 52) & 0x7ffu);
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = E - 1075 + F;
  unsigned long long v = 0;
  if (E != 0) {  // zero and subnormal values are below the resolution
    if (sh >= 0) {
      ok = ok && sh <= 9;
      v = m << (sh & 15);
    } else if (sh > -63) {
      const int r = -sh;
      v = (m + (1ull << (r - 1))) >> r;
    }
  }
  return (b >> 63) ? -(long long)v : (long long)v;
}

// v 2^e as an FP64 value in integer arithmetic (the conversions of the hardware
// run on the FP64 pipe), for |v| < 2^127 and results in the normal range: the
// leading 64 bits of |v| rounded to 53, halves away from zero (what is dropped
// below the 64 bits is 2^-11 of a last place); no branches
__device__ __forceinline__ double i128_scaled(__int128 v, int e) {
  const long long top64 = (long long)((unsigned __int128)v >> 64);
  const unsigned long long neg = (unsigned long long)(top64 >> 63);
  unsigned __int128 u = (unsigned __int128)v;  // |v|
  u = (u ^ (((unsigned __int128)neg << 64) | neg)) + (neg & 1ull);
  const unsigned long long h = (unsigned long long)(u >> 64), l = (unsigned long long)u;
  const bool small = h == 0;
  const unsigned long long a = small ? l : h, b = small ? 0ull : l;
  const int lz = __clzll((long long)a);  // 64 for zero
  // the leading 64 bits (lz = 64 only for v = 0)
  const unsigned long long m = (a << (lz & 63)) | ((b >> 1) >> (63 - (lz & 63)));
  const int top = (small ? 63 : 127) - lz;
  // 53 bits rounded, a carry out of the fraction moving to the next binade; the
  // leading bit adds one to the exponent field
  const unsigned long long r = ((unsigned long long)(unsigned)(1022 + top + e) << 52) + (m >> 11) + ((m >> 10) & 1ull);
  return __longlong_as_double(a == 0 ? 0ll : (long long)(r | (neg & 0x8000000000000000ull)));
}

// the same for |v| < 2^63
__device__ __forceinline__ double i64_scaled(long long v, int e) {
  const long long neg = v >> 63;
  const unsigned long long u = (unsigned long long)((v ^ neg) - neg);
  const int lz = __clzll((long long)u);
  const unsigned long long m = u << (lz & 63);
  const unsigned long long r =
      ((unsigned long long)(unsigned)(1022 + 63 - lz + e) << 52) + (m >> 11) + ((m >> 10) & 1ull);
  return __longlong_as_double(u == 0 ? 0ll : (long long)(r | ((unsigned long long)neg & 0x8000000000000000ull)));
}

__device__ __forceinline__ __int128 shfl_xor_i128(unsigned mask, __int128 v, int lane) {
  const unsigned long long lo = (unsigned long long)v, hi = (unsigned long long)((unsigned __int128)v >> 64);
  const unsigned long long lo2 = __shfl_xor_sync(mask, lo, lane), hi2 = __shfl_xor_sync(mask, hi, lane);
  return (__int128)(((unsigned __int128)hi2 << 64) | lo2);
}

// 1 / n for a whole n <= 2^24: Newton's iteration for the reciprocal from the
// binary32 quotient, twice (24 -> 48 -> 53 bits)
__device__ __forceinline__ double recip_count(double n, float nf) {
  const double r0 = f32_to_f64(__frcp_rn(nf));
  const double r1 = fma(r0, fma(-n, r0, 1.0), r0);
  return fma(r1, fma(-n, r1, 1.0), r1);
}

// A coordinate in steps of 2^-F as fix_round gives it, minus X0, for the short
// sums: no test inside; the largest exponent met, in steps (emax, at most 9 for
// the result to hold), and the bits of the offsets (wide, below 2^22 for |d| <
// 2^54) are kept and tested once per cluster.  sh = 1075 - F, so that the value
// is mantissa 2^(E - sh).
__device__ __forceinline__ long long fix_offset(double p, int sh, long long X0, int& emax, unsigned& wide) {
  const unsigned hi = (unsigned)__double2hiint(p), lo = (unsigned)__double2loint(p);
  const int E = (int)(hi >> 20) & 0x7ff;
  emax = max(emax, E - sh);
  // the mantissa as a 63-bit value (up 10 bits), down to twice the result, then
  // halved with the last bit rounded away from zero: exact where the result
  // holds every bit of the mantissa (E - sh from 0 to 9), nearest below; zero
  // and subnormal values shift out entirely
  const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  const unsigned long long v = (((m << 10) >> (min(9 + sh - E, 63) & 63)) + 1ull) >> 1;
  const long long neg = (long long)((int)hi >> 31);
  const long long d = (((long long)v ^ neg) - neg) - X0;
  const int dh = (int)(d >> 32);
  wide |= (unsigned)(dh ^ (dh >> 31));
  return d;
}

// The sums of up to kHalfPoints offsets: h, c, l (products of the high halves,
// cross products, products of the low halves) of xx, xy, xz, yy, yz, zz, then
// sum d; the diagonal entries hold half their cross products.
struct HalfSums {
  long long v[21];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < 21; ++k) v[k] = 0;
  }
  __device__ __forceinline__ void add(long long dx, long long dy, long long dz) {
    const int xh = (int)(dx >> 27), yh = (int)(dy >> 27), zh = (int)(dz >> 27);
    const int xl = (int)dx & 0x7ffffff, yl = (int)dy & 0x7ffffff, zl = (int)dz & 0x7ffffff;
    v[0] += (long long)xh * xh;  // xx
    v[1] += (long long)xh * xl;
    v[2] += (long long)xl * xl;
    v[3] += (long long)xh * yh;  // xy
    v[4] += (long long)xh * yl;
    v[4] += (long long)xl * yh;
    v[5] += (long long)xl * yl;
    v[6] += (long long)xh * zh;  // xz
    v[7] += (long long)xh * zl;
    v[7] += (long long)xl * zh;
    v[8] += (long long)xl * zl;
    v[9] += (long long)yh * yh;  // yy
    v[10] += (long long)yh * yl;
    v[11] += (long long)yl * yl;
    v[12] += (long long)yh * zh;  // yz
    v[13] += (long long)yh * zl;
    v[13] += (long long)yl * zh;
    v[14] += (long long)yl * zl;
    v[15] += (long long)zh * zh;  // zz
    v[16] += (long long)zh * zl;
    v[17] += (long long)zl * zl;
    v[18] += dx;
    v[19] += dy;
    v[20] += dz;
  }
};

// an entry of sum d d^T from its sums; cs = 28 for a diagonal entry, else 27
__device__ __forceinline__ __int128 join_halves(long long h, long long c, int cs, long long l) {
  return ((__int128)h << 54) + ((__int128)c << cs) + (__int128)l;
}

}  // namespace mmba
