// Device helpers shared by the sweep kernels: what a sweep does with a row of A x (epilogues) and
// the block's partial sum of |r|^2.
#pragma once
#include <cstdint>

#include "hhg_internal.h"
#include "hhg_launch.h"

namespace hhg {
namespace {

template <typename T>
__device__ __forceinline__ void block_sum_store(double v, double* out) {
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int tid = threadIdx.x + blockDim.x * threadIdx.y;
  const int nw = (blockDim.x * blockDim.y + 31) / 32;
  if ((tid & 31) == 0) red[tid >> 5] = v;
  __syncthreads();
  if (tid < 32) {
    double s = tid < nw ? red[tid] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (tid == 0) *out = s;
  }
}

template <typename T, int OP>
__device__ __forceinline__ void epilogue(const SweepArgs<T>& a, int64_t e, int64_t E, T ax, T ay, T az, T dgx, T dgy,
                                         T dgz, T x0, T y0, T z0, double& r2) {
  if (OP == OP_APPLY) {
    a.out[e] = ax;
    a.out[e + E] = ay;
    a.out[e + 2 * E] = az;
  } else if (OP == OP_DIAG) {
    a.out[e] = dgx;
    a.out[e + E] = dgy;
    a.out[e + 2 * E] = dgz;
  } else {
    const T rx = a.f[e] - ax, ry = a.f[e + E] - ay, rz = a.f[e + 2 * E] - az;
    if (OP == OP_RESID) {
      a.out[e] = rx;
      a.out[e + E] = ry;
      a.out[e + 2 * E] = rz;
      r2 += (double)rx * rx + (double)ry * ry + (double)rz * rz;
    } else if (OP == OP_JACOBI) {
      const T om = (T)a.omega;
      a.out[e] = x0 + om * rx / dgx;
      a.out[e + E] = y0 + om * ry / dgy;
      a.out[e + 2 * E] = z0 + om * rz / dgz;
    } else if (OP == OP_CHEBY) {
      const T r1 = (T)a.rho1, r2c = (T)a.rho2;
      const T ux = (a.d ? r1 * a.d[e] : (T)0) + r2c * rx / dgx;
      const T uy = (a.d ? r1 * a.d[e + E] : (T)0) + r2c * ry / dgy;
      const T uz = (a.d ? r1 * a.d[e + 2 * E] : (T)0) + r2c * rz / dgz;
      a.dout[e] = ux;
      a.dout[e + E] = uy;
      a.dout[e + 2 * E] = uz;
      a.out[e] = x0 + ux;
      a.out[e + E] = y0 + uy;
      a.out[e + 2 * E] = z0 + uz;
    }
  }
}

// Stokes epilogue (apply / residual) for one copy: velocity rows (identity on
// velocity-Dirichlet nodes) and the pressure row.
template <typename T, int OP>
__device__ __forceinline__ void stokes_epilogue(const SweepArgs<T>& a, int64_t e, int64_t E, T ax, T ay, T az, T yp,
                                                T x0, T y0, T z0, bool vdir, double& r2) {
  if (OP == OP_APPLY) {
    a.out[e] = vdir ? x0 : ax;
    a.out[e + E] = vdir ? y0 : ay;
    a.out[e + 2 * E] = vdir ? z0 : az;
    a.out[e + 3 * E] = yp;
  } else {
    const T rx = vdir ? (T)0 : a.f[e] - ax, ry = vdir ? (T)0 : a.f[e + E] - ay, rz = vdir ? (T)0 : a.f[e + 2 * E] - az;
    const T rp = a.f[e + 3 * E] - yp;
    a.out[e] = rx;
    a.out[e + E] = ry;
    a.out[e + 2 * E] = rz;
    a.out[e + 3 * E] = rp;
    r2 += (double)rx * rx + (double)ry * ry + (double)rz * rz + (double)rp * rp;
  }
}

}  // namespace
}  // namespace hhg
