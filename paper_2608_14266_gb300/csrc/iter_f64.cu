// FP64 iteration kernels: voxel pass (CalRes), scan pass (CalJH), per-scan
// damped solve + retraction (Solver) and the device-side LM decision
// (Algorithm 2 and Sec. IV-C of the paper).
#include <type_traits>

#include "checked.cuh"
#include "mmba_internal.cuh"
#include "mmba_kernels.h"

namespace mmba {

// ---------------------------------------------------------------------------
// Voxel pass: a block of 128 threads takes kV voxels (a slice or a part of
// one) of the SELL-32 slices, 128 / kV threads to a voxel, each thread every
// (128 / kV)-th of the voxel's observations.
//
// For voxel i with observations o = (i, j): q_o = R_j m_o + t_j is the posed
// cluster mean; with an anchor a (the first q_o of the voxel) the threads sum
//   n = sum N_o,  s = sum N_o (q_o - a),  M = sum [R_j S_o R_j^T + N_o (q_o - a)(q_o - a)^T]
// so that the centroid is c = a + s / n and the world-point covariance of
// Eq. 1 is A = M / n - (c - a)(c - a)^T.  The anchor keeps the subtraction
// small (plane-sized instead of scene-sized).  R_j S_o R_j^T comes from the
// slot's pivoted LDL^T of S_o (ldlt3_pivoted): 61 FP64 operations per
// observation instead of 76 with S itself.  Then lambda_min(A) and its
// eigenvector give the plane (u, d = u^T c); the voxel's cost is lambda_min.
//
// Bound: the FP64 pipe, which a warp instruction holds for 64 cycles of its
// scheduler whatever the number of its active lanes.  A voxel's observations
// are therefore a chain of ~80 such instructions each, and a problem of a few
// hundred voxels with one thread per voxel is that chain on a few warps.
// Splitting a voxel over the block's warps shortens it; the 3x3 eigenproblem
// (~250 instructions) runs once per voxel, in one warp of the block (warp
// blk % 4, so that the four schedulers share them).  Against one thread per
// voxel: 118 -> 32 us at 200 voxels, 258 -> 206 us at 50,000, 2.01 -> 1.97 ms
// at 500,000 (15M observations).
// ---------------------------------------------------------------------------
// Two forms with the same sums in the same order, so the same bits.  The split
// form (voxel_pass_f64_split) is the above.  The whole form
// (voxel_pass_f64_whole) gives a voxel to one thread, which forms the partial sums
// of as many threads as the problem's size asks for (voxel_pass_f64_rows) one
// after another and adds them up in the order of the split form's shuffles.  It
// does less work a voxel (an anchor instead of four, no idle rows, the
// eigenproblems of 128 voxels in four full warps) and has fewer warps, so it
// serves problems of many short voxels and the batches that fill the GPU.

// Posed mean of the voxel's observation at slot e (x by P's first row and so on)
__device__ __forceinline__ void voxel_anchor(const DevLayout& L, const double* poses, int64_t e, DevState* st,
                                             double (&a)[3]) {
  const int64_t ne = L.n_elems;
  const uint32_t sv = (uint32_t)__ldg(L.ve_scan + e);
  int p0, p1, p2;
  perm_decode(sv >> kPermShift, p0, p1, p2);
  const double* P = poses + 12 * (int64_t)MMBA_IDX((int32_t)(sv & kScanMask), L.n_scans, st);
  const double m0 = __ldg(L.ve + 6 * ne + e), m1 = __ldg(L.ve + 7 * ne + e), m2 = __ldg(L.ve + 8 * ne + e);
#pragma unroll
  for (int r = 0; r < 3; ++r)
    a[r] = fma(P[3 * r + p0], m0, fma(P[3 * r + p1], m1, fma(P[3 * r + p2], m2, P[9 + r])));
}

// The observation at slot e added to the sums n, s, M about the anchor a
__device__ __forceinline__ void voxel_add(const DevLayout& L, const double* poses, int64_t e, DevState* st,
                                          const double (&a)[3], double (&acc)[10]) {
  const int64_t ne = L.n_elems;
  const uint32_t sv = (uint32_t)__ldg(L.ve_scan + e);
  int p0, p1, p2;
  perm_decode(sv >> kPermShift, p0, p1, p2);
  const double* P = poses + 12 * (int64_t)MMBA_IDX((int32_t)(sv & kScanMask), L.n_scans, st);
  const double l10 = __ldg(L.ve + e), l20 = __ldg(L.ve + ne + e), l21 = __ldg(L.ve + 2 * ne + e);
  const double D0 = __ldg(L.ve + 3 * ne + e), D1 = __ldg(L.ve + 4 * ne + e), D2 = __ldg(L.ve + 5 * ne + e);
  const double m0 = __ldg(L.ve + 6 * ne + e), m1 = __ldg(L.ve + 7 * ne + e), m2 = __ldg(L.ve + 8 * ne + e);
  const double N = __ldg(L.ve + 9 * ne + e);
  // columns pi0, pi1, pi2 of R
  const double a0 = P[p0], a1 = P[3 + p0], a2 = P[6 + p0];
  const double b0 = P[p1], b1 = P[3 + p1], b2 = P[6 + p1];
  const double c0 = P[p2], c1 = P[3 + p2], c2 = P[6 + p2];
  const double qx = fma(a0, m0, fma(b0, m1, fma(c0, m2, P[9])));
  const double qy = fma(a1, m0, fma(b1, m1, fma(c1, m2, P[10])));
  const double qz = fma(a2, m0, fma(b2, m1, fma(c2, m2, P[11])));
  const double dx = qx - a[0], dy = qy - a[1], dz = qz - a[2];
  // R S R^T = sum_a D_a W_a W_a^T with W = R P^T L
  const double w00 = fma(l10, b0, fma(l20, c0, a0)), w01 = fma(l10, b1, fma(l20, c1, a1)),
               w02 = fma(l10, b2, fma(l20, c2, a2));
  const double w10 = fma(l21, c0, b0), w11 = fma(l21, c1, b1), w12 = fma(l21, c2, b2);
  const double u00 = D0 * w00, u01 = D0 * w01, u02 = D0 * w02;
  const double u10 = D1 * w10, u11 = D1 * w11, u12 = D1 * w12;
  const double u20 = D2 * c0, u21 = D2 * c1, u22 = D2 * c2;
  const double Nx = __dmul_rn(N, dx), Ny = __dmul_rn(N, dy), Nz = __dmul_rn(N, dz);
  acc[4] = fma(u00, w00, fma(u10, w10, fma(u20, c0, fma(Nx, dx, acc[4]))));
  acc[5] = fma(u00, w01, fma(u10, w11, fma(u20, c1, fma(Nx, dy, acc[5]))));
  acc[6] = fma(u00, w02, fma(u10, w12, fma(u20, c2, fma(Nx, dz, acc[6]))));
  acc[7] = fma(u01, w01, fma(u11, w11, fma(u21, c1, fma(Ny, dy, acc[7]))));
  acc[8] = fma(u01, w02, fma(u11, w12, fma(u21, c2, fma(Ny, dz, acc[8]))));
  acc[9] = fma(u02, w02, fma(u12, w12, fma(u22, c2, fma(Nz, dz, acc[9]))));
  acc[1] = __dadd_rn(acc[1], Nx);
  acc[2] = __dadd_rn(acc[2], Ny);
  acc[3] = __dadd_rn(acc[3], Nz);
  acc[0] = __dadd_rn(acc[0], N);
}

// The plane of the voxel at sorted position p from its sums and anchor, written
// out; returns lambda_min.
template <bool kFull>
__device__ __forceinline__ double voxel_plane(const DevLayout& L, double* planes, double* full_out, int64_t p,
                                              const double (&a)[3], const double (&acc)[10]) {
  const double inv = 1.0 / acc[0];
  const double cx = __dmul_rn(acc[1], inv), cy = __dmul_rn(acc[2], inv), cz = __dmul_rn(acc[3], inv);  // - anchor
  double A[6] = {fma(-cx, cx, __dmul_rn(acc[4], inv)), fma(-cx, cy, __dmul_rn(acc[5], inv)),
                 fma(-cx, cz, __dmul_rn(acc[6], inv)), fma(-cy, cy, __dmul_rn(acc[7], inv)),
                 fma(-cy, cz, __dmul_rn(acc[8], inv)), fma(-cz, cz, __dmul_rn(acc[9], inv))};
  double lam[3], V[9];
  eig3_sym(A, lam, V);
  const double ux = V[0], uy = V[1], uz = V[2];
  const double Cx = __dadd_rn(a[0], cx), Cy = __dadd_rn(a[1], cy), Cz = __dadd_rn(a[2], cz);
  double* pl = planes + p * kPlaneStride;
  pl[0] = ux;
  pl[1] = uy;
  pl[2] = uz;
  pl[3] = fma(ux, Cx, fma(uy, Cy, __dmul_rn(uz, Cz)));
  if (kFull) {
    double* f = full_out + 9 * (int64_t)L.vperm[p];
    f[0] = lam[0];
    f[1] = lam[1];
    f[2] = lam[2];
    f[3] = ux;
    f[4] = uy;
    f[5] = uz;
    f[6] = Cx;
    f[7] = Cy;
    f[8] = Cz;
  }
  return lam[0];
}

// The split form.  kTiles > 1: the block takes that many of the tiles of kV
// voxels one after another, with the same sums, and solves their eigenproblems
// together (kV kTiles = 32 lanes of the warp at work): what a batch too small
// for the whole form does with the narrow tiles of its jobs.
template <int kV, bool kFull, int kTiles>
__device__ __forceinline__ void voxel_pass_f64_split(const DevLayout& L, const double* poses2, double* planes2,
                                                     double* full_out, double* cost_part, const double* pred_part,
                                                     DevState* st, int use_trial, int decide_mode, int64_t blk,
                                                     double* red, double (*sums)[10][32], double (*anchor)[32],
                                                     int* is_last) {
  static_assert(kVoxelThreads == 128 && (kV == 8 || kV == 16 || kV == 32), "four warps per block");
  static_assert(kTiles == 1 || kTiles * kV == 32, "a slice");
  int64_t p = blk * (kV * kTiles) + (threadIdx.x & (kV - 1));
  int len = p < L.n_voxels ? L.vlen[p] : 0;
  int64_t base = p < L.n_voxels ? L.slice_off[p >> 5] + (p & 31) : 0;
  grid_wait();
  grid_launch_next();
  st = after_wait(st);
  if (st->honor_stop && st->stop) {
    // a stopped solve takes no step, so no gradient is pending either
    if (decide_mode == 0 && blk == 0 && threadIdx.x == 0) st->scan_pending = 0;
    return;
  }
  constexpr int kRows = kVoxelThreads / kV;  // threads per voxel
  const int buf = use_trial ? 1 - st->cur : st->cur;
  const double* poses = after_wait(poses2) + (int64_t)buf * L.n_scans * 12;
  double* planes = planes2 + (int64_t)buf * L.n_voxels * kPlaneStride;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the sums n, s, M of this thread's observations
  double acc[10] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  double a[3] = {0.0, 0.0, 0.0};
#pragma unroll 1
  for (int tile = 0; tile < kTiles; ++tile) {
    if (kTiles > 1 && tile > 0) {
      p += kV;
      len = p < L.n_voxels ? L.vlen[p] : 0;
      base = p < L.n_voxels ? L.slice_off[p >> 5] + (p & 31) : 0;
#pragma unroll
      for (int q = 0; q < 10; ++q) acc[q] = 0.0;
    }
    if (p < L.n_voxels) {
      const int k0 = threadIdx.x / kV;
      // the anchor: the first observation's posed mean, formed by every thread
      if (k0 < len || (kTiles == 1 && w == (int)(blk & 3))) voxel_anchor(L, poses, base, st, a);
      for (int k = k0; k < len; k += kRows) voxel_add(L, poses, base + (int64_t)k * kSlice, st, a, acc);
    }
    // a voxel's threads of one warp (kV < 32), then of the four warps, in a fixed order
#pragma unroll
    for (int o = 16; o >= kV; o >>= 1)
#pragma unroll
      for (int q = 0; q < 10; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
    if (lane < kV)
#pragma unroll
      for (int q = 0; q < 10; ++q) sums[w][q][tile * kV + lane] = acc[q];
    if (kTiles > 1 && threadIdx.x < kV)  // (the first row's threads: they have the anchor)
#pragma unroll
      for (int r = 0; r < 3; ++r) anchor[r][tile * kV + lane] = a[r];
  }
  __syncthreads();
  if (w == (int)(blk & 3)) {
    double lam0 = 0.0;
    if (kTiles > 1) {
      p = blk * (kV * kTiles) + lane;
#pragma unroll
      for (int r = 0; r < 3; ++r) a[r] = anchor[r][lane];
    }
    if (lane < kV * kTiles && p < L.n_voxels) {
#pragma unroll
      for (int q = 0; q < 10; ++q)
        acc[q] = (sums[0][q][lane] + sums[1][q][lane]) + (sums[2][q][lane] + sums[3][q][lane]);
      lam0 = voxel_plane<kFull>(L, planes, full_out, p, a, acc);
    }
#pragma unroll
    for (int o = kV / 2; o > 0; o >>= 1) lam0 += __shfl_down_sync(0xffffffffu, lam0, o);
    // (of each tile, in its first lane)
#pragma unroll
    for (int tile = 0; tile < kTiles; ++tile) {
      const double c = kTiles == 1 ? lam0 : __shfl_sync(0xffffffffu, lam0, tile * kV);
      const int64_t part = blk * kTiles + tile;
      if (lane == 0 && (kTiles == 1 || part < voxel_pass_f64_parts(L.n_voxels, L.n_obs))) cost_part[part] = c;
    }
  }
  const int64_t parts = voxel_pass_f64_parts(L.n_voxels, L.n_obs);
  voxel_pass_decide<kVoxelThreads>(cost_part, parts, pred_part, pred_parts(L.n_scans), st, decide_mode, red, is_last,
                                   (int)(blk & 3) * 32, kTiles == 1 ? parts : (L.n_voxels + 31) / 32);
}

// The whole form: the sums of kRows rows (observations row, row + kRows, ..) are
// formed one after another and added up pairwise, in the order in which the
// split form's shuffles pair the rows of a warp (0 with 2 and 1 with 3 of four)
// and then its warps.  The sums that wait for their partner are kept in shared
// memory, one place for each level of the tree; a row past the warp's longest
// voxel is empty, and nothing is added for it.
template <int kRows, int kLevels, bool kFull>
__device__ __forceinline__ void voxel_pass_f64_whole(const DevLayout& L, const double* poses2, double* planes2,
                                                     double* full_out, double* cost_part, const double* pred_part,
                                                     DevState* st, int use_trial, int decide_mode, int64_t blk,
                                                     double* red, double (*wait)[10][kVoxelThreads], int* is_last) {
  static_assert(kRows <= 1 << kLevels, "a place for each level");
  constexpr int kV = kRows == 1 ? 32 : kVoxelThreads / kRows;  // voxels to a partial sum of the cost
  const int64_t p = blk * kVoxelThreads + threadIdx.x;
  const int len = p < L.n_voxels ? L.vlen[p] : 0;
  const int64_t base = p < L.n_voxels ? L.slice_off[p >> 5] + (p & 31) : 0;
  const int longest = __reduce_max_sync(0xffffffffu, len);
  grid_wait();
  grid_launch_next();
  st = after_wait(st);
  if (st->honor_stop && st->stop) {
    if (decide_mode == 0 && blk == 0 && threadIdx.x == 0) st->scan_pending = 0;
    return;
  }
  const int buf = use_trial ? 1 - st->cur : st->cur;
  const double* poses = after_wait(poses2) + (int64_t)buf * L.n_scans * 12;
  double* planes = planes2 + (int64_t)buf * L.n_voxels * kPlaneStride;
  const int lane = threadIdx.x & 31;
  double acc[10] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  double a[3] = {0.0, 0.0, 0.0};
  if (len > 0) voxel_anchor(L, poses, base, st, a);
  unsigned waiting = 0;  // levels whose place holds a sum
#pragma unroll 1
  for (int i = 0; i < kRows; ++i) {
    const int row = kRows == 16 ? (i & 12) | ((i & 1) << 1) | ((i >> 1) & 1) : i;  // of four: 0, 2, 1, 3
    bool any = row < longest;
    if (any) {
#pragma unroll
      for (int q = 0; q < 10; ++q) acc[q] = 0.0;
      for (int k = row; k < len; k += kRows) voxel_add(L, poses, base + (int64_t)k * kSlice, st, a, acc);
    }
    int level = 0;
    for (; (i >> level) & 1; ++level) {
      if (!((waiting >> level) & 1u)) continue;
#pragma unroll
      for (int q = 0; q < 10; ++q) {
        const double other = wait[level][q][threadIdx.x];
        acc[q] = any ? other + acc[q] : other;
      }
      any = true;
      waiting &= ~(1u << level);
    }
    if (any && i < kRows - 1) {
      waiting |= 1u << level;
#pragma unroll
      for (int q = 0; q < 10; ++q) wait[level][q][threadIdx.x] = acc[q];
    }
  }
  double lam0 = p < L.n_voxels ? voxel_plane<kFull>(L, planes, full_out, p, a, acc) : 0.0;
#pragma unroll
  for (int o = kV / 2; o > 0; o >>= 1) lam0 += __shfl_down_sync(0xffffffffu, lam0, o);
  if (lane % kV == 0 && p < L.n_voxels) {
    cost_part[p / kV] = lam0;
    __threadfence();
  }
  __syncthreads();
  voxel_pass_decide<kVoxelThreads>(cost_part, voxel_pass_f64_parts(L.n_voxels, L.n_obs), pred_part,
                                   pred_parts(L.n_scans), st, decide_mode, red, is_last, 0,
                                   voxel_pass_blocks(L.n_voxels));
}

// the split form for a problem of this size (voxel_pass_f64_rows), a tile of its
// width or (kSlices) a slice of 32 voxels to a block
template <bool kFull, bool kSlices>
__device__ __forceinline__ void voxel_pass_f64_sized(const DevLayout& L, const double* poses2, double* planes2,
                                                     double* full_out, double* cost_part, const double* pred_part,
                                                     DevState* st, int use_trial, int decide_mode, int64_t blk) {
  __shared__ double red[kVoxelThreads / 32];
  __shared__ double sums[kVoxelThreads / 32][10][32];
  __shared__ double anchor[kSlices ? 3 : 1][32];
  __shared__ int is_last;
  switch (voxel_pass_f64_rows(L.n_voxels, L.n_obs)) {
    case 16:
      voxel_pass_f64_split<8, kFull, kSlices ? 4 : 1>(L, poses2, planes2, full_out, cost_part, pred_part, st,
                                                      use_trial, decide_mode, blk, red, sums, anchor, &is_last);
      break;
    case 8:
      voxel_pass_f64_split<16, kFull, kSlices ? 2 : 1>(L, poses2, planes2, full_out, cost_part, pred_part, st,
                                                       use_trial, decide_mode, blk, red, sums, anchor, &is_last);
      break;
    default:
      voxel_pass_f64_split<32, kFull, 1>(L, poses2, planes2, full_out, cost_part, pred_part, st, use_trial,
                                         decide_mode, blk, red, sums, anchor, &is_last);
  }
}

template <bool kFull, bool kWhole>
__global__ void __launch_bounds__(kVoxelThreads) voxel_pass_f64_kernel(DevLayout L, const double* poses2,
                                                                      double* planes2, double* full_out,
                                                                      double* cost_part, const double* pred_part,
                                                                      DevState* st, int use_trial, int decide_mode) {
  if (kWhole) {  // one row
    __shared__ double red[kVoxelThreads / 32];
    __shared__ int is_last;
    voxel_pass_f64_whole<1, 0, kFull>(L, poses2, planes2, full_out, cost_part, pred_part, st, use_trial, decide_mode,
                                      blockIdx.x, red, nullptr, &is_last);
  } else {
    voxel_pass_f64_sized<kFull, false>(L, poses2, planes2, full_out, cost_part, pred_part, st, use_trial, decide_mode,
                                       blockIdx.x);
  }
}

template <bool kWhole>
__global__ void __launch_bounds__(kVoxelThreads) voxel_pass_f64_batch_kernel(const __grid_constant__ JobGroup G,
                                                                             int use_trial) {
  const int job = find_job(G.vblk, G.n_jobs, blockIdx.x);
  const JobView& J = G.jobs[job];
  const int64_t blk = (int64_t)blockIdx.x - G.vblk[job];
  if (!kWhole) {
    voxel_pass_f64_sized<false, true>(J.L, J.poses2, J.planes2, nullptr, J.cost_part, J.pred_part, J.st, use_trial,
                                      use_trial ? 0 : 1, blk);
    return;
  }
  __shared__ double red[kVoxelThreads / 32];
  __shared__ double wait[4][10][kVoxelThreads];
  __shared__ int is_last;
  auto whole = [&](auto rows) {
    voxel_pass_f64_whole<decltype(rows)::value, 4, false>(J.L, J.poses2, J.planes2, nullptr, J.cost_part, J.pred_part,
                                                          J.st, use_trial, use_trial ? 0 : 1, blk, red, wait, &is_last);
  };
  switch (voxel_pass_f64_rows(J.L.n_voxels, J.L.n_obs)) {
    case 16:
      whole(std::integral_constant<int, 16>());
      break;
    case 8:
      whole(std::integral_constant<int, 8>());
      break;
    case 4:
      whole(std::integral_constant<int, 4>());
      break;
    default:
      whole(std::integral_constant<int, 1>());
  }
}

// ---------------------------------------------------------------------------
// Scan pass: one block per scan over the scan-major copy.
//
// Per observation (voxel i, scan j) the surrogate's gradient and Hessian are
// accumulated in scan coordinates and rotated to the world frame once per
// scan.  With w = R^T u (normal in scan coordinates), r = w^T m + u^T t - d
// (residual of the cluster mean) and m' = S w + N r m:
//   g_rot = m' x w,               g_trans = N r w,
//   H_rr  = [w]x (S + N m m^T) [w]x^T + (w m'^T + m' w^T)/2 - (w^T m') I,
//   H_rt  = N (m x w) w^T,        H_tt = N w w^T,
// all carrying the factor 2 / N_i, which the scan-major copy has folded into
// S and N.  The world-frame blocks are R (.) R^T.  Gauss-Newton mode drops
// the (w m'^T + m' w^T)/2 - (w^T m') I term.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void scan_pass_f64_body(const DevLayout& L, const double* poses2, const double* planes2,
                                                   double* gH, const DevState* st, int force, int order, int64_t blk,
                                                   double (*red)[32]) {
  int j = 0;
  int64_t lo = 0, hi = 0;
  auto range = [&] {
    j = MMBA_IDX(scan_of_block(L, blk), L.n_scans, st);
    lo = L.scan_off[j];
    hi = L.scan_off[j + 1];
  };
  // (before the test below only in a launch that waits: 40,000 rejected scans 42.6 us, after it 28.6)
  if (order & kWaits) range();
  grid_order(order);
  st = after_wait(st);
  // a rejected step (or an iteration after the solve stopped) leaves g, H unchanged
  if (!force && !st->scan_pending) return;
  if (!(order & kWaits)) range();
  const int buf = st->cur;
  const double* P = after_wait(poses2) + ((int64_t)buf * L.n_scans + j) * 12;
  const double* planes = after_wait(planes2) + (int64_t)buf * L.n_voxels * kPlaneStride;
  const bool gn = st->hess_mode != 0;
  const double r00 = P[0], r01 = P[1], r02 = P[2], r10 = P[3], r11 = P[4], r12 = P[5], r20 = P[6], r21 = P[7],
               r22 = P[8];
  const double tx = P[9], ty = P[10], tz = P[11];
  // the 27 sums, then those of w_a m'_a (exact Hessian's diagonal), padded to
  // a warp for the reduce-scatter
  double acc[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) acc[k] = 0.0;
  const int64_t no = L.n_obs;
  for (int64_t o = lo + threadIdx.x; o < hi; o += kScanThreads) {
    const double4_32a pl =
        *reinterpret_cast<const double4_32a*>(planes + (int64_t)MMBA_IDX(__ldg(L.se_vox + o), L.n_voxels, st) * kPlaneStride);
    const double S00 = __ldg(L.se + o), S01 = __ldg(L.se + no + o), S02 = __ldg(L.se + 2 * no + o);
    const double S11 = __ldg(L.se + 3 * no + o), S12 = __ldg(L.se + 4 * no + o), S22 = __ldg(L.se + 5 * no + o);
    const double mx = __ldg(L.se + 6 * no + o), my = __ldg(L.se + 7 * no + o), mz = __ldg(L.se + 8 * no + o);
    const double N = __ldg(L.se + 9 * no + o);
    // w = R^T u
    const double wx = fma(r00, pl.x, fma(r10, pl.y, r20 * pl.z));
    const double wy = fma(r01, pl.x, fma(r11, pl.y, r21 * pl.z));
    const double wz = fma(r02, pl.x, fma(r12, pl.y, r22 * pl.z));
    const double e = fma(pl.x, tx, fma(pl.y, ty, fma(pl.z, tz, -pl.w)));
    const double r = fma(wx, mx, fma(wy, my, fma(wz, mz, e)));
    const double Nr = N * r;
    // S w and m' = S w + N r m
    const double swx = fma(S00, wx, fma(S01, wy, S02 * wz));
    const double swy = fma(S01, wx, fma(S11, wy, S12 * wz));
    const double swz = fma(S02, wx, fma(S12, wy, S22 * wz));
    const double mpx = fma(Nr, mx, swx), mpy = fma(Nr, my, swy), mpz = fma(Nr, mz, swz);
    // gradient (FMA chains into the sums)
    acc[0] = fma(mpy, wz, fma(-mpz, wy, acc[0]));
    acc[1] = fma(mpz, wx, fma(-mpx, wz, acc[1]));
    acc[2] = fma(mpx, wy, fma(-mpy, wx, acc[2]));
    acc[3] = fma(Nr, wx, acc[3]);
    acc[4] = fma(Nr, wy, acc[4]);
    acc[5] = fma(Nr, wz, acc[5]);
    // P = S + N m m^T
    const double Nmx = N * mx, Nmy = N * my, Nmz = N * mz;
    const double p00 = fma(Nmx, mx, S00), p01 = fma(Nmx, my, S01), p02 = fma(Nmx, mz, S02);
    const double p11 = fma(Nmy, my, S11), p12 = fma(Nmy, mz, S12), p22 = fma(Nmz, mz, S22);
    // B = [w]x P  (rows: b_r = (w x P_col)...), computed as columns c of P: w x P[:, c]
    const double b00 = wy * p02 - wz * p01, b10 = wz * p00 - wx * p02, b20 = wx * p01 - wy * p00;
    const double b01 = wy * p12 - wz * p11, b11 = wz * p01 - wx * p12, b21 = wx * p11 - wy * p01;
    const double b02 = wy * p22 - wz * p12, b12 = wz * p02 - wx * p22;
    // B [w]x^T into the rotation block; [w]x rows: (0,-wz,wy), (wz,0,-wx), (-wy,wx,0)
    acc[6] = fma(wy, b02, fma(-wz, b01, acc[6]));
    acc[7] = fma(wz, b00, fma(-wx, b02, acc[7]));
    acc[8] = fma(wx, b01, fma(-wy, b00, acc[8]));
    acc[12] = fma(wz, b10, fma(-wx, b12, acc[12]));
    acc[13] = fma(wx, b11, fma(-wy, b10, acc[13]));
    acc[17] = fma(wx, b21, fma(-wy, b20, acc[17]));
    if (!gn) {
      // exact term sym(w m'^T) - (w . m') I: the off-diagonal halves go into
      // the sums here, the diagonal products into sums of their own (the trace
      // is taken off once per scan, as the term is linear)
      const double hx = 0.5 * mpx, hy = 0.5 * mpy, hz = 0.5 * mpz;
      acc[7] = fma(wx, hy, fma(hx, wy, acc[7]));
      acc[8] = fma(wx, hz, fma(hx, wz, acc[8]));
      acc[13] = fma(wy, hz, fma(hy, wz, acc[13]));
      acc[27] = fma(wx, mpx, acc[27]);
      acc[28] = fma(wy, mpy, acc[28]);
      acc[29] = fma(wz, mpz, acc[29]);
    }
    // rotation-translation block: N (m x w) w^T
    const double cx = Nmy * wz - Nmz * wy, cy = Nmz * wx - Nmx * wz, cz = Nmx * wy - Nmy * wx;
    acc[9] += cx * wx;
    acc[10] += cx * wy;
    acc[11] += cx * wz;
    acc[14] += cy * wx;
    acc[15] += cy * wy;
    acc[16] += cy * wz;
    acc[18] += cz * wx;
    acc[19] += cz * wy;
    acc[20] += cz * wz;
    // translation block: N w w^T
    const double Nwx = N * wx, Nwy = N * wy;
    acc[21] += Nwx * wx;
    acc[22] += Nwx * wy;
    acc[23] += Nwx * wz;
    acc[24] += Nwy * wy;
    acc[25] += Nwy * wz;
    acc[26] += N * wz * wz;
  }
  // Deterministic block reduction, then the rotation to the world frame, one
  // output entry per lane of warp 0.  On the FP64 pipe these cost what their
  // warp instructions are, however few lanes they hold: 31 + 3 additions and
  // ~20 operations of the rotation (a butterfly per sum and one thread's
  // rotation of the whole 6x6, ~1,000 instructions a scan, were 16% of the
  // pass at 1,500 observations a scan and most of it at 100: 3.43 -> 2.88 ms
  // at 10,000 scans of 1,500, 31 -> 16 us at 40 scans of 120).
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  warp_reduce_scatter32(acc);
  red[w][l] = acc[0];
  __syncthreads();
  if (w != 0) return;
  double tot = red[0][l];
#pragma unroll
  for (int q = 1; q < kScanThreads / 32; ++q) tot += red[q][l];
  __syncwarp();
  red[0][l] = tot;
  if (l < 9) red[1][l] = P[l];
  __syncwarp();
  const double* a = red[0];
  const double* R = red[1];
  double* out = gH + (int64_t)j * kGH;
  if (l < 6) {
    const int b = l / 3, r = l % 3;
    out[l] = fma(R[3 * r], a[3 * b], fma(R[3 * r + 1], a[3 * b + 1], R[3 * r + 2] * a[3 * b + 2]));
  } else if (l < kGH) {
    // entry (r, c) of the upper triangle: its 3x3 block B of the scan frame's 6x6 as R B R^T
    int r = 0, rem = l - 6;
    while (rem >= 6 - r) {
      rem -= 6 - r;
      ++r;
    }
    const int c = r + rem;
    const int br = r / 3, bc = c / 3, rr = r % 3, cc = c % 3;
    const double tr = br + bc == 0 ? a[27] + a[28] + a[29] : 0.0;
    double v = 0.0;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      double t = 0.0;
#pragma unroll
      for (int y = 0; y < 3; ++y) {
        int i = 3 * br + x, k = 3 * bc + y;
        if (i > k) {
          const int s = i;
          i = k;
          k = s;
        }
        double h = a[6 + 6 * i - i * (i - 1) / 2 + (k - i)];
        if (x == y && br + bc == 0) h += a[27 + x] - tr;
        t = fma(h, R[3 * cc + y], t);
      }
      v = fma(R[3 * rr + x], t, v);
    }
    out[l] = v;
  }
}

__global__ void __launch_bounds__(kScanThreads) scan_pass_f64_kernel(DevLayout L, const double* poses2,
                                                                    const double* planes2, double* gH,
                                                                    const DevState* st, int force, int order) {
  __shared__ double red[kScanThreads / 32][32];
  scan_pass_f64_body(L, poses2, planes2, gH, st, force, order, blockIdx.x, red);
}

__global__ void __launch_bounds__(kScanThreads) scan_pass_f64_batch_kernel(const __grid_constant__ JobGroup G,
                                                                          int order) {
  __shared__ double red[kScanThreads / 32][32];
  const int job = find_job(G.sblk, G.n_jobs, blockIdx.x);
  const JobView& J = G.jobs[job];
  scan_pass_f64_body(J.L, J.poses2, J.planes2, J.gH, J.st, 0, order, (int64_t)blockIdx.x - G.sblk[job], red);
}

// ---------------------------------------------------------------------------
// Solver: A = H + mu diag(H), A delta = -g by LDL^T, trial pose
// R' = Exp(dphi) R, t' = t + dt, and the scan's share of the predicted
// reduction -(g^T delta + delta^T H delta / 2).  The fixed scan and scans
// without observations keep their pose.
//
// Bound by the number of FP64 instructions of a warp (64 cycles of its SM
// sub-partition each, whatever the lanes): one thread per scan takes 310 for
// 32 scans, eight lanes per scan 120 for 4.  With fewer warps than
// sub-partitions the shorter one wins, with several to each the one with less
// work in all: solve_lanes.
// ---------------------------------------------------------------------------
// Coefficients in th^2, th = |dphi| < 0.1, of sin(th)/th, (1 - cos th)/th^2,
// cos(th/2) and sin(th/2)/th: the Taylor series to th^8 (the first dropped
// term is below 1e-17).
__device__ const double kExpSeries[4][5] = {
    {1.0, -1.0 / 6, 1.0 / 120, -1.0 / 5040, 1.0 / 362880},
    {0.5, -1.0 / 24, 1.0 / 720, -1.0 / 40320, 1.0 / 3628800},
    {1.0, -1.0 / 8, 1.0 / 384, -1.0 / 46080, 1.0 / 10321920},
    {0.5, -1.0 / 48, 1.0 / 3840, -1.0 / 645120, 1.0 / 185794560},
};

// The two forms do the same arithmetic in the same order (products and sums that
// the compiler could contract differently are written out), so a scan's step
// and a block's sums have the same bits in both.
//
// c0 + th^2 (c1 + ..) of one of the series, or its function beyond 0.1 rad
__device__ __forceinline__ double exp_coef(int which, const double* series, double th2) {
  if (!(th2 < 0.01)) {
    const double th = sqrt(th2);
    double sh, ch;
    sincos(0.5 * th, &sh, &ch);
    return which == 0 ? sin(th) / th : which == 1 ? 2.0 * sh * sh / th2 : which == 2 ? ch : sh / th;
  }
  double v = fma(th2, series[4], series[3]);
#pragma unroll
  for (int k = 2; k >= 0; --k) v = fma(th2, v, series[k]);
  return v;
}
// |dphi|^2
__device__ __forceinline__ double phi_sq(const double* d) { return fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2])); }
// a column p of R moved by Exp(dphi): p + a (phi x p) + b phi x (phi x p), the
// increment first (one rounding at the size of p)
__device__ __forceinline__ void exp_column(const double* d, double ca, double cb, const double* p, double* n) {
  const double u0 = fma(d[1], p[2], -(d[2] * p[1])), u1 = fma(d[2], p[0], -(d[0] * p[2])),
               u2 = fma(d[0], p[1], -(d[1] * p[0]));
  const double w0 = fma(d[1], u2, -(d[2] * u1)), w1 = fma(d[2], u0, -(d[0] * u2)), w2 = fma(d[0], u1, -(d[1] * u0));
  n[0] = __dadd_rn(p[0], fma(ca, u0, __dmul_rn(cb, w0)));
  n[1] = __dadd_rn(p[1], fma(ca, u1, __dmul_rn(cb, w1)));
  n[2] = __dadd_rn(p[2], fma(ca, u2, __dmul_rn(cb, w2)));
}
// component i of (cc, cs dphi) times the quaternion whose components i, i ^ 1,
// i ^ 2, i ^ 3 are q, q1, q2, q3 (the signs of the Hamilton product)
__device__ __forceinline__ double exp_quat(int i, const double* d, double cc, double cs, double q, double q1, double q2,
                                           double q3) {
  const double s1 = (i & 1) ? q1 : -q1, s2 = i == 1 || i == 2 ? q2 : -q2, s3 = (i & 2) ? q3 : -q3;
  return fma(cc, q, __dmul_rn(cs, fma(d[0], s1, fma(d[1], s2, __dmul_rn(d[2], s3)))));
}
// a row's term of -(g^T x + x^T H x / 2), with half the row's share of H x
__device__ __forceinline__ double pred_term(double x, double g, double hx) { return __dmul_rn(-x, __dadd_rn(g, hx)); }

// One thread per scan.  *stepped = false: the pose is kept (fixed scan, no
// observation, failed factorisation); otherwise dlt holds the increment.
__device__ inline double solve_scan(const DevLayout& L, int j, const double* P, double* Pt, const double* gH,
                                    DevState* st, double* dlt, bool* stepped) {
  *stepped = false;
  const double* a = gH + (int64_t)j * kGH;
  // a scan nobody observes keeps its pose: no observation in this handle's
  // layout, or, for a voxel-sharded solve (g, H totals over all shards), an
  // all-zero total Hessian diagonal (an observation always makes it nonzero)
  const bool unseen = st->shard ? (a[6] == 0.0 && a[12] == 0.0 && a[17] == 0.0 && a[21] == 0.0 && a[24] == 0.0 &&
                                   a[26] == 0.0)
                                : L.scan_off[j + 1] == L.scan_off[j];
  if (j == L.fixed_scan || unseen) {
    for (int k = 0; k < 12; ++k) Pt[k] = P[k];
    return 0.0;
  }
  double g[6], H[36], A[36], b[6];
  for (int k = 0; k < 6; ++k) g[k] = a[k];
  int idx = 6;
  for (int r = 0; r < 6; ++r)
    for (int c = r; c < 6; ++c) {
      H[6 * r + c] = a[idx];
      H[6 * c + r] = a[idx];
      ++idx;
    }
  const double mu = st->mu;
  for (int k = 0; k < 36; ++k) A[k] = H[k];
  for (int k = 0; k < 6; ++k) {
    A[7 * k] = fma(mu, H[7 * k], H[7 * k]);
    b[k] = -g[k];
  }
  if (!ldlt6_solve(A, b, dlt)) {
    atomicOr(&st->solve_fail_flag, 1);
    for (int k = 0; k < 12; ++k) Pt[k] = P[k];
    return 0.0;
  }
  // the quadratic form from H's upper triangle, the rows' terms summed as the
  // lanes' shuffles do
  double t[6];
#pragma unroll
  for (int r = 0; r < 6; ++r) {
    double hx = __dmul_rn(0.5 * H[7 * r], dlt[r]);
#pragma unroll
    for (int c = r + 1; c < 6; ++c) hx = fma(H[6 * r + c], dlt[c], hx);
    t[r] = pred_term(dlt[r], g[r], hx);
  }
  const double th2 = phi_sq(dlt);
  const double ca = exp_coef(0, kExpSeries[0], th2), cb = exp_coef(1, kExpSeries[1], th2);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double p[3] = {P[c], P[3 + c], P[6 + c]};
    double n[3];
    exp_column(dlt, ca, cb, p, n);
    Pt[c] = n[0];
    Pt[3 + c] = n[1];
    Pt[6 + c] = n[2];
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) Pt[9 + k] = __dadd_rn(P[9 + k], dlt[3 + k]);
  *stepped = true;
  return ((t[0] + t[1]) + (t[2] + t[3])) + (t[4] + t[5]);
}

// Eight lanes per scan.  Lane r < 6 holds row r of [A | -g] and eliminates it
// by the pivot rows' broadcasts; the substitution runs up the rows' kept
// factors.  The rotation's columns go to lanes 0..2 (p + a (phi x p) +
// b phi x (phi x p), the Exp map on a column), the translation to 3..5, the
// four series and the quaternion's components to 0..3.  Returns this lane's
// term of the predicted reduction.
__device__ __forceinline__ double solve_scan_lanes(const DevLayout& L, int64_t j, double* poses2, const double* gH,
                                                   DevState* st, const double* sref, float* stab2,
                                                   const double (&series)[5]) {
  constexpr unsigned kAll = 0xffffffffu;
  const int r = threadIdx.x & 7, row = r < 6 ? r : 5;
  const unsigned group = 0xffu << (threadIdx.x & 24);
  const bool live = j < L.n_scans;
  if (!live) j = L.n_scans - 1;  // computed and not written
  const int cur = st->cur;
  const double mu = st->mu;
  const double* P = poses2 + ((int64_t)cur * L.n_scans + j) * 12;
  double* Pt = poses2 + ((int64_t)(1 - cur) * L.n_scans + j) * 12;
  const double* h27 = gH + j * kGH;
  double h[6], a[7], p[3], q = 0.0, ref = 0.0;
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const int i = row < c ? row : c, k = row < c ? c : row;
    h[c] = h27[6 + 6 * i - i * (i - 1) / 2 + (k - i)];
  }
  const double g = h27[row];
  const int pc = r < 3 ? r : 9 + (row - 3);  // a column of R, or an entry of t
#pragma unroll
  for (int k = 0; k < 3; ++k) p[k] = P[r < 3 ? pc + 3 * k : pc];
  double* sq2 = stab2 ? after_wait(sq2_of(sref, L.n_scans)) : nullptr;
  if (stab2) {
    q = sq2[((int64_t)cur * L.n_scans + j) * 4 + (r & 3)];
    ref = sref[12 * j + 9 + (r < 3 ? r : row - 3)];
  }
  // a scan nobody observes keeps its pose (see solve_scan)
  double hd = 0.0;
#pragma unroll
  for (int c = 0; c < 6; ++c) hd = row == c ? h[c] : hd;
  const bool none = (__ballot_sync(kAll, hd != 0.0) & group) == 0;
  const bool unseen = st->shard ? none : L.scan_off[j + 1] == L.scan_off[j];
  const bool held = j == L.fixed_scan || unseen;

#pragma unroll
  for (int c = 0; c < 6; ++c) a[c] = row == c ? fma(mu, h[c], h[c]) : h[c];
  a[6] = -g;
  bool ok = true;
  double inv_row = 0.0, f[6];  // f: the row of L
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double d = __shfl_sync(kAll, a[k], k, 8);
    ok = ok && d > 0.0 && isfinite(d);
    const double inv = recip_pivot(d);
    if (row == k) inv_row = inv;
    if (k == 5) break;
    // the lower triangle: entry (row, c) takes column k's entry of row c, the
    // right-hand side the pivot row's
    const double l = row > k ? __dmul_rn(a[k], inv) : 0.0;
    f[k] = l;
    const double y = __shfl_sync(kAll, a[6], k, 8);
#pragma unroll
    for (int c = k + 1; c < 6; ++c) a[c] = fma(-l, __shfl_sync(kAll, a[k], c, 8), a[c]);
    a[6] = fma(-l, y, a[6]);
  }
  double x = __dmul_rn(a[6], inv_row);
#pragma unroll
  for (int k = 5; k >= 1; --k) {
    // row k of L to the lanes below: lane i takes its entry i
    double lk = 0.0;
#pragma unroll
    for (int i = 0; i < k; ++i) {
      const double v = __shfl_sync(kAll, f[i], k, 8);
      lk = row == i ? v : lk;
    }
    x = fma(-lk, __shfl_sync(kAll, x, k, 8), x);
  }
  const unsigned lost = __ballot_sync(kAll, !isfinite(x));  // by every lane, ok or not
  ok = ok && (lost & group) == 0;
  const bool stepped = ok && !held;
  if (live && !held && !ok && r == 0) atomicOr(&st->solve_fail_flag, 1);

  double dlt[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) dlt[c] = __shfl_sync(kAll, x, c, 8);
  // this row's term of the predicted reduction, H's upper triangle only
  double hx = __dmul_rn(0.5 * hd, x);
#pragma unroll
  for (int c = 1; c < 6; ++c) hx = fma(c > row ? h[c] : 0.0, dlt[c], hx);
  const double pred = live && stepped && r < 6 ? pred_term(x, g, hx) : 0.0;
  const double th2 = phi_sq(dlt);
  const double v = exp_coef(r & 3, series, th2);  // uniform branch over the scan's lanes
  __syncwarp();
  const double ca = __shfl_sync(kAll, v, 0, 8), cb = __shfl_sync(kAll, v, 1, 8);
  if (live) {
    if (r < 3) {
      double n[3];
      exp_column(dlt, ca, cb, p, n);
#pragma unroll
      for (int k = 0; k < 3; ++k) Pt[3 * k + r] = stepped ? n[k] : p[k];
    } else if (r < 6) {
      p[0] = stepped ? __dadd_rn(p[0], x) : p[0];
      Pt[6 + r] = p[0];
    }
  }
  if (stab2) {
    // the step's quaternion times the current one
    const double cc = __shfl_sync(kAll, v, 2, 8), cs = __shfl_sync(kAll, v, 3, 8);
    const int i = r & 3;
    const double q1 = __shfl_xor_sync(kAll, q, 1), q2 = __shfl_xor_sync(kAll, q, 2), q3 = __shfl_xor_sync(kAll, q, 3);
    double qn = exp_quat(i, dlt, cc, cs, q, q1, q2, q3);
    qn = stepped ? qn : q;
    const double w = __shfl_sync(kAll, qn, 0, 8);
    const double t = r < 3 ? 0.0 : p[0] - ref;
    if (live) {
      if (r < 4) sq2[((int64_t)(1 - cur) * L.n_scans + j) * 4 + r] = qn;
      // the FP32 table entry (scan_table_from_quat)
      float* out = stab2 + ((int64_t)(1 - cur) * L.n_scans + j) * kTab;
      if (r < 4) out[r] = f64_to_f32(w < 0.0 ? -qn : qn);
      if (r >= 3 && r < 6) out[1 + r] = f64_to_f32(t);
      if (r < 3) out[7 + r] = f64_to_f32(ref);
      if (r >= 6) out[4 + r] = 0.0f;
    }
  }
  return pred;
}

// With stab2 given (mixed precision) the trial scan's FP32 table entry is
// written too, from the trial pose and the scan's reference pose.  Block blk
// takes kSolveThreads / kLanes consecutive scans; the sum of the predicted
// reductions of every kPredScans scans goes to pred_part, in a fixed order.
template <int kLanes>
__device__ __forceinline__ void solve_f64_body(const DevLayout& L, double* poses2, const double* gH,
                                               double* pred_part, DevState* st, const double* sref, float* stab2,
                                               int64_t blk, double* red) {
  static_assert(kLanes == 1 || (kLanes == 8 && kSolveThreads == 8 * kPredScans && kPredScans == 8), "shuffle widths");
  double series[5];
  if (kLanes == 8) {
#pragma unroll
    for (int k = 0; k < 5; ++k) series[k] = kExpSeries[threadIdx.x & 3][k];
  }
  grid_wait();
  grid_launch_next();
  st = after_wait(st);
  gH = after_wait(gH);
  poses2 = after_wait(poses2);
  if (st->honor_stop && st->stop) return;  // uniform over the block
  if (kLanes == 8) {
    // rows, then scans, in pairs, fours and eights
    double v = solve_scan_lanes(L, blk * kPredScans + threadIdx.x / 8, poses2, gH, st, sref, stab2, series);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) pred_part[blk] = __dadd_rn(red[0], red[1]);
    return;
  }
  const int64_t j = blk * kSolveThreads + threadIdx.x;
  double pred = 0.0;
  if (j < L.n_scans) {
    const int cur = st->cur;
    const double* P = poses2 + ((int64_t)cur * L.n_scans + j) * 12;
    double* Pt = poses2 + ((int64_t)(1 - cur) * L.n_scans + j) * 12;
    double dlt[6];
    bool stepped;
    pred = solve_scan(L, (int)j, P, Pt, gH, st, dlt, &stepped);
    if (stab2) {
      // FP64 quaternion of the trial dR: the step's Exp composed onto the
      // current one (no matrix-to-quaternion conversion per step)
      double* sq2 = after_wait(sq2_of(sref, L.n_scans));
      const double* qc = sq2 + ((int64_t)cur * L.n_scans + j) * 4;
      double* qt = sq2 + ((int64_t)(1 - cur) * L.n_scans + j) * 4;
      const double q[4] = {qc[0], qc[1], qc[2], qc[3]};
      double qn[4];
      if (stepped) {
        const double th2 = phi_sq(dlt);
        const double cc = exp_coef(2, kExpSeries[2], th2), cs = exp_coef(3, kExpSeries[3], th2);
#pragma unroll
        for (int i = 0; i < 4; ++i) qn[i] = exp_quat(i, dlt, cc, cs, q[i], q[i ^ 1], q[i ^ 2], q[i ^ 3]);
      } else {
        for (int k = 0; k < 4; ++k) qn[k] = q[k];
      }
      for (int k = 0; k < 4; ++k) qt[k] = qn[k];
      scan_table_from_quat(qn, Pt, sref + 12 * (int64_t)j, stab2 + ((int64_t)(1 - cur) * L.n_scans + j) * kTab);
    }
  }
#pragma unroll
  for (int o = 1; o < kPredScans; o <<= 1) pred = __dadd_rn(pred, __shfl_xor_sync(0xffffffffu, pred, o));
  const int64_t part = (blk * kSolveThreads + threadIdx.x) / kPredScans;
  if (threadIdx.x % kPredScans == 0 && part < pred_parts(L.n_scans)) pred_part[part] = pred;
}

template <int kLanes>
__global__ void __launch_bounds__(kSolveThreads) solve_f64_kernel(DevLayout L, double* poses2, const double* gH,
                                                                 double* pred_part, DevState* st, const double* sref,
                                                                 float* stab2) {
  __shared__ double red[kSolveThreads / 32];
  solve_f64_body<kLanes>(L, poses2, gH, pred_part, st, sref, stab2, blockIdx.x, red);
}

template <int kLanes>
__global__ void __launch_bounds__(kSolveThreads) solve_f64_batch_kernel(const __grid_constant__ JobGroup G) {
  __shared__ double red[kSolveThreads / 32];
  const int job = find_job(G.oblk, G.n_jobs, blockIdx.x);
  const JobView& J = G.jobs[job];
  solve_f64_body<kLanes>(J.L, J.poses2, J.gH, J.pred_part, J.st, J.X.sref, J.X.stab2,
                         (int64_t)blockIdx.x - G.oblk[job], red);
}

__global__ void __launch_bounds__(kDecideThreads) decide_kernel(const double* __restrict__ cost_part, int64_t n_cost,
                                                               const double* __restrict__ pred_part, int64_t n_pred,
                                                               DevState* st, int mode) {
  __shared__ double red[kDecideThreads / 32];
  decide_body<kDecideThreads>(cost_part, n_cost, pred_part, n_pred, st, mode, red);
}

// Voxel-sharded solve: this handle's part of the trial cost (its cost
// partials summed in the decision's fixed order) ...
__global__ void __launch_bounds__(kDecideThreads) shard_cost_kernel(const double* __restrict__ cost_part, int64_t n_cost,
                                                                   double* __restrict__ out) {
  __shared__ double red[kDecideThreads / 32];
  const double csum = block_sum<kDecideThreads>(strided_sum<kDecideThreads>(cost_part, n_cost), red);
  if (threadIdx.x == 0) *out = csum;
}

// ... and the decision from the trial cost summed over every shard (the
// predicted reduction comes from the total g, H, so every shard has it whole)
__global__ void __launch_bounds__(kDecideThreads) shard_decide_kernel(const double* __restrict__ pred_part,
                                                                     int64_t n_pred, DevState* st, double trial_total) {
  __shared__ double red[kDecideThreads / 32];
  const double psum = block_sum<kDecideThreads>(strided_sum<kDecideThreads>(pred_part, n_pred), red);
  if (threadIdx.x == 0) decide_apply(st, trial_total, psum);
}

// ---- launchers ---------------------------------------------------------------

cudaError_t launch_voxel_pass_f64(const DevLayout& L, const double* poses2, double* planes2, double* full_out,
                                  double* cost_part, const double* pred_part, DevState* st, int use_trial,
                                  int decide_mode, cudaStream_t stream, bool dependent) {
  const bool whole = voxel_pass_f64_rows(L.n_voxels, L.n_obs) == 1;
  const auto kernel = full_out ? (whole ? voxel_pass_f64_kernel<true, true> : voxel_pass_f64_kernel<true, false>)
                               : (whole ? voxel_pass_f64_kernel<false, true> : voxel_pass_f64_kernel<false, false>);
  return launch_dependent(kernel, voxel_pass_f64_blocks(L.n_voxels, L.n_obs), kVoxelThreads, stream, dependent, L,
                          poses2, planes2, full_out, cost_part, pred_part, st, use_trial, decide_mode);
}

cudaError_t launch_scan_pass_f64(const DevLayout& L, const double* poses2, const double* planes2, double* gH,
                                 const DevState* st, int force, cudaStream_t stream, bool dependent,
                                 bool next_early) {
  if (L.n_scans == 0) return cudaSuccess;
  return launch_dependent(scan_pass_f64_kernel, L.n_scans, kScanThreads, stream, dependent, L, poses2, planes2, gH, st,
                          force, (dependent ? kWaits : 0) | (next_early ? kFreesNext : 0));
}

cudaError_t launch_shard_cost(const double* cost_part, int64_t n_cost, double* out, cudaStream_t stream) {
  shard_cost_kernel<<<1, kDecideThreads, 0, stream>>>(cost_part, n_cost, out);
  return cudaGetLastError();
}

cudaError_t launch_shard_decide(const DevLayout& L, const double* pred_part, DevState* st, double trial_total,
                                cudaStream_t stream) {
  shard_decide_kernel<<<1, kDecideThreads, 0, stream>>>(pred_part, pred_parts(L.n_scans), st, trial_total);
  return cudaGetLastError();
}

cudaError_t launch_solve_f64(const DevLayout& L, double* poses2, const double* gH, double* pred_part, DevState* st,
                             const double* sref, float* stab2, cudaStream_t stream, bool dependent) {
  const int lanes = solve_lanes(L.n_scans);
  return launch_dependent(lanes == 8 ? solve_f64_kernel<8> : solve_f64_kernel<1>, solve_blocks(L.n_scans, lanes),
                          kSolveThreads, stream, dependent, L, poses2, gH, pred_part, st, sref, stab2);
}

cudaError_t launch_decide(const double* cost_part, int64_t n_cost, const double* pred_part, int64_t n_pred,
                          DevState* st, int mode, cudaStream_t stream) {
  decide_kernel<<<1, kDecideThreads, 0, stream>>>(cost_part, n_cost, pred_part, n_pred, st, mode);
  return cudaGetLastError();
}

cudaError_t launch_batch_solve(const JobGroup& T, int64_t n_blocks, cudaStream_t stream) {
  return launch_dependent(T.solve_lanes == 8 ? solve_f64_batch_kernel<8> : solve_f64_batch_kernel<1>, n_blocks,
                          kSolveThreads, stream, false, T);
}

cudaError_t launch_batch_voxel_pass_f64(const JobGroup& T, int64_t n_blocks, int use_trial, cudaStream_t stream) {
  return launch_dependent(T.whole_voxels ? voxel_pass_f64_batch_kernel<true> : voxel_pass_f64_batch_kernel<false>,
                          n_blocks, kVoxelThreads, stream,
                          early_voxel_pass_f64(n_blocks) || T.sblk[T.n_jobs] >= 3 * kSMs, T, use_trial);
}

cudaError_t launch_batch_scan_pass_f64(const JobGroup& T, int64_t n_blocks, cudaStream_t stream) {
  const bool early = early_scan_pass_f64(n_blocks, T.vblk[T.n_jobs]);
  return launch_dependent(scan_pass_f64_batch_kernel, n_blocks, kScanThreads, stream, early, T, early ? kWaits : 0);
}

}  // namespace mmba
