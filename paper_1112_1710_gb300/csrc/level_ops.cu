// level_ops.cu -- per-level operations that feed the patch advance: the CFL
// time-step reduction, the list-driven ghost fill and the FP64 conservation
// sums.  Built with --fmad=false (the CFL candidate is compared bit for bit).
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"
#include "launch.h"
#include "physics.cuh"

namespace mhd {

// ---------------------------------------------------------------- CFL dt
// Per interior cell: t = min_d dx_d / (|v_d| + c_f,d), in the patch's
// arithmetic type.  The block minimum of t (warp shuffles, then shared
// memory; a block lies in one patch) becomes the candidate (cfl * t) * scale
// in FP64 once per block, and one atomicMin on its IEEE bits (positive, so
// integer order is value order) reduces over blocks.  x -> (cfl x) scale is
// monotone, so this equals the minimum of the per-cell candidates.
template <typename R>
__global__ void __launch_bounds__(kThreads) k_cfl(const DPatch* __restrict__ P,
                                                  const BlockTask* __restrict__ T, double gamma_d,
                                                  double cfl, unsigned long long* out,
                                                  int* status) {
  const BlockTask t = T[blockIdx.x];
  const DPatch& p = P[t.patch];
  const int e = t.start + threadIdx.x;
  const R inf = R(1) / R(0);
  R m = inf;
  if (e < p.n[0] * p.n[1] * p.n[2]) {
    int i, j, k;
    if (p.n[0] * p.n[1] * p.n[2] < (1 << 24)) {
      int ri, rj;
      const int q = divmod24(e, p.n[0], ri);
      k = divmod24(q, p.n[1], rj);
      i = ri;
      j = rj;
    } else {
      i = e % p.n[0];
      j = (e / p.n[0]) % p.n[1];
      k = e / (p.n[0] * p.n[1]);
    }
    const int64_t x = (int64_t)(p.g + i) + (int64_t)(p.g + j) * p.s1 + (int64_t)(p.g + k) * p.s2;
    const R gamma = (R)gamma_d, gm1 = gamma - R(1);
    R u[8], w[8];
#pragma unroll
    for (int q = 0; q < 5; ++q) u[q] = ((const R*)p.U[q])[x];
    u[5] = Tr<R>::half(((const R*)p.B[0])[x] + ((const R*)p.B[0])[x + 1]);
    u[6] = Tr<R>::half(((const R*)p.B[1])[x] + ((const R*)p.B[1])[x + p.s1]);
    u[7] = Tr<R>::half(((const R*)p.B[2])[x] + ((const R*)p.B[2])[x + p.s2]);
    cons2prim(u, gm1, w);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int t1 = (d + 1) % 3, t2 = (d + 2) % 3;
      R cf = fast_speed(w[0], w[4], w[5 + d], w[5 + t1], w[5 + t2], gamma);
      R tt = Tr<R>::div(dx_of<R>(p, d), Tr<R>::abs(w[1 + d]) + cf);
      m = rmin(m, tt);
    }
    if (!(w[0] > R(0)) || !(w[4] > R(0))) raise_status(status, -4);
  }
  for (int o = 16; o > 0; o >>= 1) {
    R u2 = __shfl_down_sync(0xffffffffu, m, o);
    m = (u2 < m) ? u2 : m;
  }
  __shared__ R red[kThreads / 32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = (threadIdx.x < kThreads / 32) ? red[threadIdx.x] : inf;
    for (int o = 16; o > 0; o >>= 1) {
      R u2 = __shfl_down_sync(0xffffffffu, m, o);
      m = (u2 < m) ? u2 : m;
    }
    if (threadIdx.x == 0) {
      const double v = (cfl * (double)m) * p.cfl_scale;
      if (v == v) atomicMin(out, (unsigned long long)__double_as_longlong(v));
    }
  }
}

__global__ void k_set_inf(unsigned long long* out) {
  *out = 0x7FF0000000000000ULL;
}

cudaError_t cfl_dt_launch(int dtype, const DPatch* patches, const BlockTask* tasks, int nblocks,
                          double gamma, double cfl, double* d_out, int* d_status,
                          const KernelTimer* tm, cudaStream_t s) {
  MHD_TIMED(tm, K_CFL, s, (k_set_inf<<<1, 1, 0, s>>>((unsigned long long*)d_out)));
  if (nblocks > 0) {
    if (dtype == 0)
      MHD_TIMED(tm, K_CFL, s, (k_cfl<double><<<nblocks, kThreads, 0, s>>>(
                                  patches, tasks, gamma, cfl, (unsigned long long*)d_out, d_status)));
    else
      MHD_TIMED(tm, K_CFL, s, (k_cfl<float><<<nblocks, kThreads, 0, s>>>(
                                  patches, tasks, gamma, cfl, (unsigned long long*)d_out, d_status)));
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------- sums
// Two passes with a fixed reduction tree, so the result is reproducible: per
// block the values x dV of 256 cells are added pairwise, cell t and t + 128,
// then + 64 and so on, and the blocks' sums in order, 256 chains of them side
// by side and then the same tree.
//
// A warp takes a block of cells, eight per lane 32 apart, so that the first
// three levels of the tree are a lane's own additions and nothing waits on a
// barrier; below 32 cells a warp holds several of the eight sums.  The FP64
// pipe (one warp instruction per SM every 16 cycles) carries the additions
// alone, 65 instructions per 256 cells: FP32 values are widened in integers,
// and the multiplication by dV is an addition to the exponent where dV is a
// power of two (a base grid of 2^k cells on the unit box).  The second pass
// takes one block per sum and coalesced rows of partial sums.  Measured on
// 200 patches of 8^3-64^3 cells (4.0 M cells, FP32), both passes: 295 -> 100
// us with dx = 1/256, 157 us with dx = 0.01; one thread per cell with the tree in shared memory took 180 us (259 us
// with the upper half of the warps leaving at each level).
__device__ __noinline__ double times(double x, double y) { return x * y; }

// x 2^k, exactly as the multiplication gives it
__device__ __forceinline__ double scaled(double x, int k) {
  const uint64_t u = i64::bits(x);
  const int e = (int)(u >> 52) & 0x7ff;
  if ((u << 1) == 0 || e == 0x7ff) return x;
  if (e == 0 || e + k < 1 || e + k > 0x7fe) return times(x, i64::value((uint64_t)(1023 + k) << 52));
  return i64::value(u + ((uint64_t)(int64_t)k << 52));
}

// x 2^k for an FP32 x (-1022 <= k <= 1023): a normal x widened and scaled in
// one addition to its exponent field
__device__ __forceinline__ double scaled(float x, int k) {
  const uint32_t f = __float_as_uint(x), e = (f >> 23) & 0xffu;
  if (e - 1u < 0xfeu && k >= -800 && k <= 800)
    return i64::value(((uint64_t)((f & 0x80000000u) | (((f & 0x7fffffffu) >> 3) + ((uint32_t)(896 + k) << 20))) << 32) |
                      (uint64_t)(f << 29));
  return (f << 1) == 0 ? i64::value((uint64_t)f << 32) : scaled(i64::widen(x), k);
}
__device__ __forceinline__ double widened(float x) { return i64::widen(x); }
__device__ __forceinline__ double widened(double x) { return x; }

template <typename R>
__global__ void __launch_bounds__(kThreads) k_sums(const DPatch* __restrict__ P,
                                                   const BlockTask* __restrict__ T, int ntasks,
                                                   double* partials) {
  const int task = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (task >= ntasks) return;
  const BlockTask t = T[task];
  const DPatch& p = P[t.patch];
  const int nc = p.n[0] * p.n[1] * p.n[2];
  const bool small = nc < (1 << 24);
  const uint64_t bdv = i64::bits(p.dv);
  const int edv = (int)(bdv >> 52) & 0x7ff;
  const bool pow2 = (bdv & 0xfffffffffffffull) == 0 && edv != 0 && edv != 0x7ff;
  int64_t x[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int e = t.start + lane + 32 * c;
    x[c] = -1;
    if (e < nc) {
      int i, j, k;
      if (small) {
        k = divmod24(divmod24(e, p.n[0], i), p.n[1], j);
      } else {
        i = e % p.n[0];
        j = (e / p.n[0]) % p.n[1];
        k = e / (p.n[0] * p.n[1]);
      }
      x[c] = (int64_t)(p.g + i) + (int64_t)(p.g + j) * p.s1 + (int64_t)(p.g + k) * p.s2;
    }
  }
  // a rolled loop: unrolled, the eight sums' code overflows the instruction cache
  __shared__ double part[kThreads / 32][8][32];
  double (*mine)[32] = part[threadIdx.x >> 5];
#pragma unroll 1
  for (int q = 0; q < 8; ++q) {
    const R* a = (const R*)(q < 5 ? p.U[q] : p.B[q - 5]);
    R raw[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) raw[c] = x[c] >= 0 ? a[x[c]] : R(0);
    double s[8];
#pragma unroll
    for (int c = 0; c < 8; ++c)
      s[c] = x[c] < 0 ? 0.0 : (pow2 ? scaled(raw[c], edv - 1023) : times(widened(raw[c]), p.dv));
#pragma unroll
    for (int w = 4; w > 0; w >>= 1)
#pragma unroll
      for (int c = 0; c < w; ++c) s[c] = s[c] + s[c + w];
    mine[q][lane] = s[0];
  }
  double v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = mine[q][lane];  // this lane's own
  // 32 cells x 8 sums left: at each step a lane keeps half of its sums and
  // gives the others to its partner, which holds their other cells
#pragma unroll
  for (int w = 16, n = 4; w >= 4; w >>= 1, n >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int q = 0; q < n; ++q) {
      const double give = up ? v[2 * q] : v[2 * q + 1], keep = up ? v[2 * q + 1] : v[2 * q];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, give, w);
    }
  }
  v[0] = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 2);
  v[0] = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
  const int q = ((lane >> 4) & 1) | ((lane >> 2) & 2) | (lane & 4);  // the sum this lane holds
  if ((lane & 3) == 0) partials[(int64_t)q * ntasks + task] = v[0];
}

__global__ void __launch_bounds__(kThreads) k_sums_final(const double* __restrict__ partials, int nblocks,
                                                         double* out) {
  __shared__ double sh[kThreads];
  const double* row = partials + (int64_t)blockIdx.x * nblocks;
  double v = 0.0;
#pragma unroll 8
  for (int b = threadIdx.x; b < nblocks; b += kThreads) v = v + row[b];
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] = sh[threadIdx.x] + sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = sh[0];
}

cudaError_t sums_launch(int dtype, const DPatch* patches, const BlockTask* tasks, int nblocks,
                        double* partials, double* d_out8, const KernelTimer* tm, cudaStream_t s) {
  if (nblocks > 0) {
    if (dtype == 0)
      MHD_TIMED(tm, K_SUMS, s, (k_sums<double><<<(nblocks + 7) / 8, kThreads, 0, s>>>(patches, tasks, nblocks, partials)));
    else
      MHD_TIMED(tm, K_SUMS, s, (k_sums<float><<<(nblocks + 7) / 8, kThreads, 0, s>>>(patches, tasks, nblocks, partials)));
  }
  MHD_TIMED(tm, K_SUMS, s, (k_sums_final<<<8, kThreads, 0, s>>>(partials, nblocks, d_out8)));
  return cudaGetLastError();
}

}  // namespace mhd
