// Device helpers shared by the sweep and transfer kernels: the numbering of a slice's interior points,
// what a sweep does with a row of A x (epilogues), the block's partial sum of |r|^2.
#pragma once
#include <cstdint>

#include "hhg_internal.h"
#include "hhg_launch.h"

namespace hhg {
namespace {

// (j, i) of the t-th interior point of a slice with M = n-1-k: rows j = 1..M-1 hold
// M-j points; C(j) = (j-1)(2M-j)/2 points precede row j.
__device__ __forceinline__ void slice_decode(int M, int t, int& j, int& i) {
  const float b = (float)(2 * M - 1);
  int u = (int)floorf(0.5f * (b - sqrtf(fmaxf(b * b - 8.0f * (float)t, 0.0f))));
  u = max(0, min(u, M - 2));
  // exact correction: C(u+1) <= t < C(u+2)
  if (((u + 1) * (2 * M - u - 2)) / 2 <= t) ++u;
  if ((u * (2 * M - u - 1)) / 2 > t) --u;
  j = u + 1;
  i = t - (u * (2 * M - u - 1)) / 2 + 1;
}

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

// What an epilogue reads of entry e besides the row: f and, for a Chebyshev step, the last correction d.
// Constructed before the row, so that the loads are in flight meanwhile.
template <typename T, int OP, int STK>
struct Rhs {
  static constexpr bool F = OP == OP_RESID || OP == OP_JACOBI || OP == OP_CHEBY;
  T f[3], fp, d[3];
  __device__ __forceinline__ Rhs(const SweepArgs<T>& a, int64_t e, int64_t E) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (F) f[c] = a.f[e + c * E];
      if (OP == OP_CHEBY) d[c] = a.d ? a.d[e + c * E] : (T)0;
    }
    if (F && STK) fp = a.f[e + 3 * E];
  }
};

template <typename T, int OP>
__device__ __forceinline__ void epilogue(const SweepArgs<T>& a, const Rhs<T, OP, 0>& rhs, int64_t e, int64_t E,
                                         T ax, T ay, T az, T dgx, T dgy, T dgz, T x0, T y0, T z0, double& r2) {
  if (OP == OP_APPLY) {
    a.out[e] = ax;
    a.out[e + E] = ay;
    a.out[e + 2 * E] = az;
  } else if (OP == OP_DIAG) {
    a.out[e] = dgx;
    a.out[e + E] = dgy;
    a.out[e + 2 * E] = dgz;
  } else {
    const T rx = rhs.f[0] - ax, ry = rhs.f[1] - ay, rz = rhs.f[2] - az;
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
      const T ux = r1 * rhs.d[0] + r2c * rx / dgx;
      const T uy = r1 * rhs.d[1] + r2c * ry / dgy;
      const T uz = r1 * rhs.d[2] + r2c * rz / dgz;
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
__device__ __forceinline__ void stokes_epilogue(const SweepArgs<T>& a, const Rhs<T, OP, 1>& rhs, int64_t e,
                                                int64_t E, T ax, T ay, T az, T yp, T x0, T y0, T z0, bool vdir, double& r2) {
  if (OP == OP_APPLY) {
    a.out[e] = vdir ? x0 : ax;
    a.out[e + E] = vdir ? y0 : ay;
    a.out[e + 2 * E] = vdir ? z0 : az;
    a.out[e + 3 * E] = yp;
  } else {
    const T rx = vdir ? (T)0 : rhs.f[0] - ax, ry = vdir ? (T)0 : rhs.f[1] - ay, rz = vdir ? (T)0 : rhs.f[2] - az;
    const T rp = rhs.fp - yp;
    a.out[e] = rx;
    a.out[e + E] = ry;
    a.out[e + 2 * E] = rz;
    a.out[e + 3 * E] = rp;
    r2 += (double)rx * rx + (double)ry * ry + (double)rz * rz + (double)rp * rp;
  }
}

// the same with the loads at the end of the row
template <typename T, int OP>
__device__ __forceinline__ void epilogue(const SweepArgs<T>& a, int64_t e, int64_t E, T ax, T ay, T az, T dgx, T dgy,
                                         T dgz, T x0, T y0, T z0, double& r2) {
  epilogue<T, OP>(a, Rhs<T, OP, 0>(a, e, E), e, E, ax, ay, az, dgx, dgy, dgz, x0, y0, z0, r2);
}
template <typename T, int OP>
__device__ __forceinline__ void stokes_epilogue(const SweepArgs<T>& a, int64_t e, int64_t E, T ax, T ay, T az, T yp,
                                                T x0, T y0, T z0, bool vdir, double& r2) {
  stokes_epilogue<T, OP>(a, Rhs<T, OP, 1>(a, e, E), e, E, ax, ay, az, yp, x0, y0, z0, vdir, r2);
}

}  // namespace
}  // namespace hhg
