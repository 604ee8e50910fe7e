// Macro-interior sweeps that march along a lattice direction (k_march): the default for every
// operator epilogue of the scaled-stencil variants and for the Stokes saddle operator.
//
// A thread takes a short column of points p, p + d2, p + 2 d2, ... along stencil direction 2, the
// lattice vector (0, -1, 1).  Along it c = j + k is constant, so
//   - the columns of a macro fill rectangles: for every c the points i = 1 .. n - 1 - c, k = 1 ..
//     c - 1; neighbouring lanes take neighbouring i (coalesced) and march equally far, whatever the
//     tetrahedron's shape;
//   - the offsets of the rows above and below (n + 1 - c and -(n + 2 - c) entries) stay the same,
//     and the stencil's 15 points lie in seven columns, each of which contributes one new point per
//     step: 28 loads (x, y, z, k) per point instead of 60;
//   - the block of the edge (p, p + d2) serves both its ends: khat (x_{p+d2} - x_p) and the
//     correction w x (x_{p+d2} - x_p) are kept for the next point, where they enter with the
//     opposite and the same sign (S_ji = S_ij^T).
// The correction stencils of a six-element edge are linearly dependent: with the ring nodes r_0 ..
// r_5 in cyclic order and s_q the axial vector of the pair (r_q, r_{q+3}), s_1 = s_0 + s_2 (the
// correction of an element is proportional to the vector between its other two vertices, and s_q
// to r_{q+1} - r_{q-1}), so w = (e_0 + e_1) s_0 + (e_1 + e_2) s_2 with e_q = k_{r_q} - k_{r_{q+3}}.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "hhg_internal.h"
#include "hhg_launch.h"
#include "hhg_rows.cuh"

namespace hhg {

namespace {

constexpr int MARCH_BLOCK = ROWS_BLOCK;

// the constants of one macro in shared memory, as 16-byte words: per direction pair S (6 values),
// s_0 and s_2 (s_0 and s_1 of a four-element edge), and for Stokes B, G, C and a pad
template <int STK>
constexpr int MARCH_C = STK ? 20 : 12;

template <typename T, int N>
__device__ __forceinline__ void load_shared(const T* p, T (&v)[N]) {
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int q = 0; q < N; q += 4) {
      const float4 f = *reinterpret_cast<const float4*>(p + q);
      v[q] = f.x;
      v[q + 1] = f.y;
      v[q + 2] = f.z;
      v[q + 3] = f.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < N; q += 2) {
      const double2 f = *reinterpret_cast<const double2*>(p + q);
      v[q] = f.x;
      v[q + 1] = f.y;
    }
  }
}

// a point in the order of evaluation that needs these values
__device__ __forceinline__ void keep(float& x, float& y, float& z) { asm volatile("" : "+f"(x), "+f"(y), "+f"(z)); }
__device__ __forceinline__ void keep(double& x, double& y, double& z) { asm volatile("" : "+d"(x), "+d"(y), "+d"(z)); }

// values of one lattice point
template <typename T, int STK>
struct Node {
  T x, y, z, k;
};
template <typename T>
struct Node<T, 1> {
  T x, y, z, k, p;
};

// columns of the march around the thread's own (offsets at equal k): own, i + 1, i - 1, the row
// above (j + 1) at i and i - 1, the row below at i and i + 1
enum { CP, CR, CUL, CU, CL, CD, CDR };

template <typename T, int OP, int GEN, int STK>
struct March {
  static constexpr bool DIAG = OP == OP_JACOBI || OP == OP_CHEBY || OP == OP_DIAG;
  using N = Node<T, STK>;
  const T* __restrict__ X;
  const T* __restrict__ K;
  int64_t E;
  int up, down;  // entries from a point to the one above / below it (j + 1, j - 1)
  // slices k and k + 1 of the columns whose next point the current point needs, and k and k - 1 of
  // the others
  N a[2][4], b[2][3];
  T kprev;           // coefficient of the column's previous point
  T tx, ty, tz;      // khat (x_{p+d2} - x_p) of the previous point's edge
  T hx, hy, hz;      // w x (x_{p+d2} - x_p) of it
  T kh2;             // khat of it
  T ux, uy, uz;      // (Stokes) x_{p+d2} - x_p of it

  __device__ __forceinline__ N load(int q) const {
    N v;
    v.x = __ldg(X + q);
    v.y = __ldg(X + E + q);
    v.z = __ldg(X + 2 * E + q);
    v.k = __ldg(K + q);
    if constexpr (STK) v.p = __ldg(X + 3 * E + q);
    return v;
  }
  __device__ __forceinline__ void load_a(N (&v)[4], int p) const {
    v[CP] = load(p);
    v[CR] = load(p + 1);
    v[CUL] = load(p + up - 1);
    v[CU] = load(p + up);
  }
  __device__ __forceinline__ void load_b(N (&v)[3], int p) const {
    v[CL - CL] = load(p - 1);
    v[CD - CL] = load(p + down);
    v[CDR - CL] = load(p + down + 1);
  }
  // neighbour in direction d
  __device__ __forceinline__ const N& nb(int d) const {
    switch (d) {
      case 0: return a[0][CR];
      case 1: return a[0][CUL];
      case 2: return a[1][CP];
      case 3: return a[0][CU];
      case 4: return a[1][CUL];
      case 5: return a[1][CR];
      case 6: return a[1][CU];
      case 7: return b[0][CL - CL];
      case 8: return b[0][CDR - CL];
      case 10: return b[0][CD - CL];
      case 11: return b[1][CDR - CL];
      case 12: return b[1][CL - CL];
      default: return b[1][CD - CL];  // 13; direction 9 is only asked for its coefficient
    }
  }
  __device__ __forceinline__ T kk(int d) const {
    return d == 9 ? kprev : nb(d).k;
  }
  // khat and w of direction d's edge (e: d or its negative) from the constants c of the pair
  __device__ __forceinline__ void edge(int d, bool negative, const T (&c)[MARCH_C<STK>], const OpFlags& fl, T& kh,
                                       T& wx, T& wy, T& wz) const {
    const bool physical = GEN ? fl.physical != 0 : true;
    const bool khat_edge = GEN ? fl.khat_edge != 0 : false;
    const T k0 = a[0][CP].k, kd = kk(negative ? d + 7 : d);
    T e[3], rs;
    const int nr = dir_red(d) ? 3 : 2;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      if (q >= nr) break;
      const int ra = ring_cyc(d, q), rb = ring_cyc(d, q + nr);
      const T ka = kk(negative ? dir_neg(ra) : ra), kb = kk(negative ? dir_neg(rb) : rb);
      const T sum = ka + kb;
      rs = q == 0 ? sum : rs + sum;
      e[q] = ka - kb;
    }
    if (khat_edge)
      kh = (T)0.5 * (k0 + kd);
    else
      kh = fma(dir_red(d) ? (T)(1.0 / 12.0) : (T)0.125, rs, fma((T)0.25, kd, (T)0.25 * k0));
    if (physical) {
      const T f0 = dir_red(d) ? e[0] + e[1] : e[0], f1 = dir_red(d) ? e[2] + e[1] : e[1];
      wx = fma(f1, c[9], f0 * c[6]);
      wy = fma(f1, c[10], f0 * c[7]);
      wz = fma(f1, c[11], f0 * c[8]);
    } else {
      wx = wy = wz = 0;
    }
  }

  // the row of the point; leaves the edge (p, p + d2) for the next point
  __device__ __forceinline__ void row(const T* __restrict__ cst, const OpFlags& fl, T& ax, T& ay, T& az, T& dgx, T& dgy,
                                      T& dgz, T& yp) {
    const bool physical = GEN ? fl.physical != 0 : true;
    ax = ay = az = dgx = dgy = dgz = yp = 0;
    const unsigned act = __activemask();
    int zero = 0;
    const N& o = a[0][CP];
#pragma unroll
    for (int d = 0; d < 7; ++d) {
      // the constants are read again for every point, direction by direction (the __syncwarp keeps
      // the scheduler from reading all of them first): held in registers they would spill
      asm volatile("" : "+r"(zero));
      __syncwarp(act);
      T c[MARCH_C<STK>];
      load_shared(cst + zero + d * MARCH_C<STK>, c);
      T khp, khm, wx, wy, wz, vx, vy, vz;
      edge(d, false, c, fl, khp, wx, wy, wz);
      const N& np = nb(d);
      const T px = np.x - o.x, py = np.y - o.y, pz = np.z - o.z;
      T mx, my, mz;
      if (d == 2) {
        khm = kh2;
        const T sx = khp * px, sy = khp * py, sz = khp * pz;
        vx = sx - tx;
        vy = sy - ty;
        vz = sz - tz;
        tx = sx;
        ty = sy;
        tz = sz;
        kh2 = khp;
        if (physical) {
          const T gx = fma(wy, pz, -(wz * py)), gy = fma(wz, px, -(wx * pz)), gz = fma(wx, py, -(wy * px));
          ax += gx + hx;
          ay += gy + hy;
          az += gz + hz;
          hx = gx;
          hy = gy;
          hz = gz;
        }
        mx = -ux;
        my = -uy;
        mz = -uz;
        ux = px;
        uy = py;
        uz = pz;
      } else {
        if (physical) {
          ax = fma(wy, pz, ax);
          ax = fma(-wz, py, ax);
          ay = fma(wz, px, ay);
          ay = fma(-wx, pz, ay);
          az = fma(wx, py, az);
          az = fma(-wy, px, az);
        }
        edge(d, true, c, fl, khm, wx, wy, wz);
        const N& nm = nb(d + 7);
        mx = nm.x - o.x;
        my = nm.y - o.y;
        mz = nm.z - o.z;
        if (physical) {
          ax = fma(wy, mz, ax);
          ax = fma(-wz, my, ax);
          ay = fma(wz, mx, ay);
          ay = fma(-wx, mz, ay);
          az = fma(wx, my, az);
          az = fma(-wy, mx, az);
        }
        vx = fma(khp, px, khm * mx);
        vy = fma(khp, py, khm * my);
        vz = fma(khp, pz, khm * mz);
      }
      ax = fma(c[0], vx, ax);
      ax = fma(c[3], vy, ax);
      ax = fma(c[4], vz, ax);
      ay = fma(c[3], vx, ay);
      ay = fma(c[1], vy, ay);
      ay = fma(c[5], vz, ay);
      az = fma(c[4], vx, az);
      az = fma(c[5], vy, az);
      az = fma(c[2], vz, az);
      if (DIAG) {
        const T ks = khp + khm;
        dgx = fma(-ks, c[0], dgx);
        dgy = fma(-ks, c[1], dgy);
        dgz = fma(-ks, c[2], dgz);
      }
      if constexpr (STK) {
        // B_{-d} = -B_d, G_{-d} = -G_d, C_{-d} = C_d
        const T pm = d == 2 ? pprev : nb(d + 7).p;
        const T dp = np.p - pm;
        ax = fma(c[15], dp, ax);
        ay = fma(c[16], dp, ay);
        az = fma(c[17], dp, az);
        yp = fma(c[12], px - mx, yp);
        yp = fma(c[13], py - my, yp);
        yp = fma(c[14], pz - mz, yp);
        yp = fma(c[18], (np.p - o.p) + (pm - o.p), yp);
      }
    }
  }
  T pprev;  // (Stokes) pressure of the column's previous point
};

// A block of columns of one macro (LevelDev::columns, FP64); cst: 7 MARCH_C values.
template <typename T, int OP, int GEN, int STK>
__device__ __forceinline__ void march_block(const LevelDev& L, const MacroConsts<T>* __restrict__ mc, const int macro,
                                            const int block, const OpFlags& fl, const SweepArgs<T>& a, T* cst,
                                            double* partial) {
  for (int q = threadIdx.x; q < 7 * MARCH_C<STK>; q += MARCH_BLOCK) {
    const int d = q / MARCH_C<STK>, r = q - d * MARCH_C<STK>;
    cst[q] = __ldg(&mc[macro].mar[d][r]);
  }
  __syncthreads();
  const int t = block * MARCH_BLOCK + threadIdx.x;
  double r2 = 0.0;
  if (t < L.ncolumns[1]) {
    const int32_t col = L.columns[1][t];
    const int n = L.n;
    const int c = col >> 20, i = col & 0x3FF;
    int k = (col >> 10) & 0x3FF;
    const int kend = min(k + L.column_len[1], c);
    March<T, OP, GEN, STK> M;
    const int64_t base = (int64_t)macro * L.nt;
    M.E = L.entries;
    M.X = a.x + base;
    M.K = a.k + base;
    M.up = n + 1 - c;
    M.down = -(n + 2 - c);
    int p = lattice_index32(n, i, c - k, k);
    // the point before the column and the edge from it (whose ring lies in the two slices)
    {
      const int pp = p - ((n - k + 1) * (n - k + 2)) / 2;
      M.a[0][CP] = M.load(pp);
      M.load_b(M.b[0], pp);
      M.load_a(M.a[1], p);
      const auto o = M.a[0][CP];
      const auto& q = M.a[1][CP];
      T cc[MARCH_C<STK>];
      load_shared(cst + 2 * MARCH_C<STK>, cc);
      T wx, wy, wz;
      M.edge(2, false, cc, fl, M.kh2, wx, wy, wz);
      M.ux = q.x - o.x;
      M.uy = q.y - o.y;
      M.uz = q.z - o.z;
      M.tx = M.kh2 * M.ux;
      M.ty = M.kh2 * M.uy;
      M.tz = M.kh2 * M.uz;
      M.hx = fma(wy, M.uz, -(wz * M.uy));
      M.hy = fma(wz, M.ux, -(wx * M.uz));
      M.hz = fma(wx, M.uy, -(wy * M.ux));
      M.kprev = o.k;
      if constexpr (STK) M.pprev = o.p;
#pragma unroll
      for (int r = 0; r < 4; ++r) M.a[0][r] = M.a[1][r];
#pragma unroll
      for (int r = 0; r < 3; ++r) M.b[1][r] = M.b[0][r];
      M.load_b(M.b[0], p);
    }
    T ax, ay, az, dgx, dgy, dgz, yp;
    const int k0 = k;
    while (true) {
      int pn = p + ((n - k) * (n - k + 1)) / 2;
      asm volatile("" : "+r"(pn));  // the step's loads stay behind the last step's arithmetic (registers)
      M.load_a(M.a[1], pn);
      if (k > k0) M.load_b(M.b[0], p);
      const Rhs<T, OP, STK> rhs(a, base + p, M.E);
      M.row(cst, fl, ax, ay, az, dgx, dgy, dgz, yp);
      asm volatile("" : "+r"(p));
      keep(ax, ay, az);
      const auto& o = M.a[0][CP];
      if constexpr (STK) {
        stokes_epilogue<T, OP>(a, rhs, base + p, M.E, ax, ay, az, yp, o.x, o.y, o.z, false, r2);
        M.pprev = o.p;
      } else {
        epilogue<T, OP>(a, rhs, base + p, M.E, ax, ay, az, dgx, dgy, dgz, o.x, o.y, o.z, r2);
      }
      if (++k >= kend) break;
      M.kprev = o.k;
#pragma unroll
      for (int q = 0; q < 4; ++q) M.a[0][q] = M.a[1][q];
#pragma unroll
      for (int q = 0; q < 3; ++q) M.b[1][q] = M.b[0][q];
      p = pn;
    }
  }
  if (OP == OP_RESID && partial != nullptr) block_sum_store<T>(r2, partial);
}

// ---------------------------------------------------------------------------
// FP32: both directions of a pair (d, -d) in the two lanes of packed FP32 arithmetic
// (fma.rn.f32x2 and friends).  The pair's constants, patch means, corrections and cross products
// are the same sums over point-reflected neighbours, so every packed instruction serves both.  Along
// the march the pairs need no moves: with A the columns ahead (i + 1; j + 1; j + 1, i - 1) and B
// their reflections (i - 1; j - 1; j - 1, i + 1), the point of slice k pairs (A_k, B_k) and
// (A_{k+1}, B_{k-1}), and the next one (A_{k+1}, B_{k+1}) and (A_{k+2}, B_k): the new values overwrite
// the lanes of the two old pairs that are no longer needed.
// ---------------------------------------------------------------------------
struct F2 {
  float2 v;
  __device__ __forceinline__ F2() {}
  __device__ __forceinline__ F2(float2 a) : v(a) {}
  __device__ __forceinline__ F2(float a, float b) : v(make_float2(a, b)) {}
};
__device__ __forceinline__ F2 dup(float a) { return F2(a, a); }
__device__ __forceinline__ F2 swapped(F2 a) { return F2(a.v.y, a.v.x); }
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return F2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return F2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) { return F2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
  unsigned long long r;
  const unsigned long long x = *reinterpret_cast<const unsigned long long*>(&a.v);
  const unsigned long long y = *reinterpret_cast<const unsigned long long*>(&b.v);
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return F2(*reinterpret_cast<const float2*>(&r));
}
__device__ __forceinline__ float sum(F2 a) { return a.v.x + a.v.y; }
__device__ __forceinline__ float diff(F2 a) { return a.v.x - a.v.y; }

// constants of a direction pair in shared memory: S (6 values and a pad), then the lane pairs (s, s)
// of the two axial vectors and, for Stokes, of B, G, C
template <int STK>
constexpr int MARCH2_C = 8 + 2 * (6 + (STK ? 8 : 0));

// fields of a lattice point: x, y, z, k and, for Stokes, p
template <int OP, int GEN, int STK, int KB>
struct March2 {
  static constexpr bool DIAG = OP == OP_JACOBI || OP == OP_CHEBY || OP == OP_DIAG;
  static constexpr int NF = STK ? 5 : 4;
  static constexpr int FK = 3, FP = 4;
  const float* __restrict__ X;
  const float* __restrict__ K;
  const uint16_t* __restrict__ K16;
  int64_t E;
  int up, down;
  // q[s][c][f]: column pair c (0: i + 1 | i - 1; 1: j + 1, i - 1 | its reflection; 2: j + 1 | j - 1);
  // s = 0: (A_k, B_k), 1: (A_{k+1}, B_{k-1})
  F2 q[2][3][NF];
  F2 ce[NF];      // (k + 1, k - 1) of the thread's own column
  float o[NF];    // its point of slice k

  __device__ __forceinline__ float load(int f, int at) const {
    if (f == FK) {
      if constexpr (KB)
        return __uint_as_float((uint32_t)__ldg(K16 + at) << 16);
      else
        return __ldg(K + at);
    }
    return __ldg(X + (f == FP ? 3 : f) * E + at);
  }
  // lane x (A) / y (B) of the column pairs from the slice whose own point is at `at`
  __device__ __forceinline__ void load_a(F2 (&v)[3][NF], int at) const {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      v[0][f].v.x = load(f, at + 1);
      v[1][f].v.x = load(f, at + up - 1);
      v[2][f].v.x = load(f, at + up);
    }
  }
  __device__ __forceinline__ void load_b(F2 (&v)[3][NF], int at) const {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      v[0][f].v.y = load(f, at - 1);
      v[1][f].v.y = load(f, at + down + 1);
      v[2][f].v.y = load(f, at + down);
    }
  }
  // field f of the neighbours (d, -d), d < 7
  __device__ __forceinline__ F2 pairof(int d, int f) const {
    switch (d) {
      case 0: return q[0][0][f];
      case 1: return q[0][1][f];
      case 3: return q[0][2][f];
      case 2: return ce[f];
      case 4: return q[1][1][f];
      case 5: return q[1][0][f];
      default: return q[1][2][f];
    }
  }
  // coefficients of the neighbours (e, -e), e < 14
  __device__ __forceinline__ F2 kk(int e) const {
    return e < 7 ? pairof(e, FK) : swapped(pairof(e - 7, FK));
  }

  __device__ __forceinline__ void row(const float* __restrict__ cst, const OpFlags& fl, float& ax, float& ay, float& az,
                                      float& dgx, float& dgy, float& dgz, float& yp) const {
    const unsigned act = __activemask();
    const bool physical = GEN ? fl.physical != 0 : true;
    const bool khat_edge = GEN ? fl.khat_edge != 0 : false;
    ax = ay = az = dgx = dgy = dgz = yp = 0.0f;
    // cross products: sums of w_y d_z, w_z d_x, w_x d_y and of w_z d_y, w_x d_z, w_y d_x
    F2 cx = dup(0.0f), cy = cx, cz = cx, nx = cx, ny = cx, nz = cx;
    F2 gx = cx, gy = cx, gz = cx, bd = cx, cp = cx;
    const F2 x0 = dup(o[0]), y0 = dup(o[1]), z0 = dup(o[2]), k0q = dup(0.25f * o[FK]);
    int zero = 0;
#pragma unroll
    for (int d = 0; d < 7; ++d) {
      // the constants are read again for every point, direction by direction (the __syncwarp keeps
      // the scheduler from reading all of them first): held in registers they would spill
      asm volatile("" : "+r"(zero));
      __syncwarp(act);
      const float* cd = cst + zero + d * MARCH2_C<STK>;
      const float4 s0 = *reinterpret_cast<const float4*>(cd), s1 = *reinterpret_cast<const float4*>(cd + 4);
      float4 w[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) w[r] = *reinterpret_cast<const float4*>(cd + 8 + 4 * r);
      const F2 dx = pairof(d, 0) - x0, dy = pairof(d, 1) - y0, dz = pairof(d, 2) - z0;
      F2 e[3], rs;
      const int nr = dir_red(d) ? 3 : 2;
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        if (r >= nr) break;
        const F2 ka = kk(ring_cyc(d, r)), kb = kk(ring_cyc(d, r + nr));
        rs = r == 0 ? ka + kb : (rs + ka) + kb;
        e[r] = ka - kb;
      }
      const F2 kd = pairof(d, FK);
      const F2 kh = khat_edge ? fma2(dup(0.5f), kd, k0q + k0q)
                              : fma2(dup(dir_red(d) ? (float)(1.0 / 12.0) : 0.125f), rs, fma2(dup(0.25f), kd, k0q));
      if (physical) {
        const F2 f0 = dir_red(d) ? e[0] + e[1] : e[0], f1 = dir_red(d) ? e[2] + e[1] : e[1];
        const F2 wx = fma2(f1, F2(w[1].z, w[1].w), f0 * F2(w[0].x, w[0].y));
        const F2 wy = fma2(f1, F2(w[2].x, w[2].y), f0 * F2(w[0].z, w[0].w));
        const F2 wz = fma2(f1, F2(w[2].z, w[2].w), f0 * F2(w[1].x, w[1].y));
        cx = fma2(wy, dz, cx);
        nx = fma2(wz, dy, nx);
        cy = fma2(wz, dx, cy);
        ny = fma2(wx, dz, ny);
        cz = fma2(wx, dy, cz);
        nz = fma2(wy, dx, nz);
      }
      const float vx = sum(kh * dx), vy = sum(kh * dy), vz = sum(kh * dz);
      ax = fmaf(s0.x, vx, ax);
      ax = fmaf(s0.w, vy, ax);
      ax = fmaf(s1.x, vz, ax);
      ay = fmaf(s0.w, vx, ay);
      ay = fmaf(s0.y, vy, ay);
      ay = fmaf(s1.y, vz, ay);
      az = fmaf(s1.x, vx, az);
      az = fmaf(s1.y, vy, az);
      az = fmaf(s0.z, vz, az);
      if (DIAG) {
        const float ks = sum(kh);
        dgx = fmaf(-ks, s0.x, dgx);
        dgy = fmaf(-ks, s0.y, dgy);
        dgz = fmaf(-ks, s0.z, dgz);
      }
      if constexpr (STK) {
        // B_{-d} = -B_d, G_{-d} = -G_d, C_{-d} = C_d
        float4 u[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) u[r] = *reinterpret_cast<const float4*>(cd + 20 + 4 * r);
        const F2 dp = pairof(d, FP) - dup(o[FP]);
        bd = fma2(F2(u[0].x, u[0].y), dx, bd);
        bd = fma2(F2(u[0].z, u[0].w), dy, bd);
        bd = fma2(F2(u[1].x, u[1].y), dz, bd);
        gx = fma2(F2(u[1].z, u[1].w), dp, gx);
        gy = fma2(F2(u[2].x, u[2].y), dp, gy);
        gz = fma2(F2(u[2].z, u[2].w), dp, gz);
        cp = fma2(F2(u[3].x, u[3].y), dp, cp);
      }
    }
    if (physical) {
      ax += sum(cx - nx);
      ay += sum(cy - ny);
      az += sum(cz - nz);
    }
    if constexpr (STK) {
      ax += diff(gx);
      ay += diff(gy);
      az += diff(gz);
      yp = diff(bd) + sum(cp);
    }
  }
};

// As march_block; cst: 7 MARCH2_C values, and with SHARE > 0 as many for each of the block's macros: it takes
// macros `macro` .. with all their columns, 2^SHARE threads each.
template <int OP, int GEN, int STK, int KB, int SHARE>
__device__ __forceinline__ void march2_block(const LevelDev& L, const MacroConsts<float>* __restrict__ mc,
                                             int macro, const int block, const OpFlags& fl,
                                             const SweepArgs<float>& a, float* cst, double* partial) {
  constexpr int NC = 7 * MARCH2_C<STK>;
  for (int r = threadIdx.x; r < (SHARE ? MARCH_BLOCK >> SHARE : 1) * NC; r += MARCH_BLOCK) {
    const int m = SHARE ? macro + r / NC : macro, d = (SHARE ? r % NC : r) / MARCH2_C<STK>;
    const int w = (SHARE ? r % NC : r) - d * MARCH2_C<STK>;
    if (SHARE && m >= L.nmacro) break;
    cst[r] = w < 8 ? (w < 6 ? __ldg(&mc[m].mar[d][w]) : 0.0f) : __ldg(&mc[m].mar[d][6 + (w - 8) / 2]);
  }
  __syncthreads();
  int t = block * MARCH_BLOCK + threadIdx.x;
  if constexpr (SHARE > 0) {
    const int part = threadIdx.x >> SHARE;
    macro += part;
    cst += part * NC;
    t = macro < L.nmacro ? threadIdx.x & ((1 << SHARE) - 1) : INT32_MAX;
  }
  double r2 = 0.0;
  if (t < L.ncolumns[0]) {
    const int32_t col = L.columns[0][t];
    const int n = L.n;
    const int c = col >> 20, i = col & 0x3FF;
    int k = (col >> 10) & 0x3FF;
    const int kend = min(k + L.column_len[0], c);
    March2<OP, GEN, STK, KB> M;
    constexpr int NF = STK ? 5 : 4;
    const int64_t base = (int64_t)macro * L.nt;
    M.E = L.entries;
    M.X = a.x + base;
    M.K = a.k + base;
    M.K16 = KB ? a.k16 + base : nullptr;
    M.up = n + 1 - c;
    M.down = -(n + 2 - c);
    int p = lattice_index32(n, i, c - k, k);
    int pn = p + ((n - k) * (n - k + 1)) / 2;
    {
      const int pp = p - ((n - k + 1) * (n - k + 2)) / 2;
      M.load_a(M.q[0], p);
      M.load_b(M.q[1], pp);
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        M.o[f] = M.load(f, p);
        M.ce[f].v.y = M.load(f, pp);
      }
    }
    float ax, ay, az, dgx, dgy, dgz, yp;
    do {
      asm volatile("" : "+r"(pn));  // the step's loads stay behind the last step's arithmetic (registers)
      M.load_a(M.q[1], pn);
      M.load_b(M.q[0], p);
#pragma unroll
      for (int f = 0; f < NF; ++f) M.ce[f].v.x = M.load(f, pn);
      const Rhs<float, OP, STK> rhs(a, base + p, M.E);
      M.row(cst, fl, ax, ay, az, dgx, dgy, dgz, yp);
      asm volatile("" : "+r"(p));
      keep(ax, ay, az);
      if constexpr (STK)
        stokes_epilogue<float, OP>(a, rhs, base + p, M.E, ax, ay, az, yp, M.o[0], M.o[1], M.o[2], false, r2);
      else
        epilogue<float, OP>(a, rhs, base + p, M.E, ax, ay, az, dgx, dgy, dgz, M.o[0], M.o[1], M.o[2], r2);
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        M.ce[f].v.y = M.o[f];
        M.o[f] = M.ce[f].v.x;
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) {
          const F2 t2 = M.q[0][cc][f];
          M.q[0][cc][f] = M.q[1][cc][f];
          M.q[1][cc][f] = t2;
        }
      }
      p = pn;
      ++k;
      pn += ((n - k) * (n - k + 1)) / 2;
    } while (k < kend);
  }
  if (OP == OP_RESID && partial != nullptr) block_sum_store<float>(r2, partial);
}

// ---------------------------------------------------------------------------
// A whole sweep in one launch: blocks of the macro interiors with the skeleton's blocks spread evenly
// between them.  One launch for latency's sake: on small levels it is one wave, where two launches on two
// streams followed one another, since either one's blocks fill the registers of every SM.  On large levels
// the parts add up all the same (FP32 apply on 257^3 nodes: interiors alone 330 us, rows alone 66, together
// 390): a row block waits for memory most of the time, in a slot that a march block could use.
// ---------------------------------------------------------------------------
template <typename T, int OP, int GEN, int STK, int KB, int SHARE = 0>
__global__ void __launch_bounds__(MARCH_BLOCK, sizeof(T) == 4 ? 4 : 2)
    k_sweep(const LevelDev L, const MacroConsts<T>* __restrict__ mc, const OpFlags fl, const SweepArgs<T> a,
            const int per_macro, const int rows) {
  constexpr int NC = 7 * (sizeof(T) == 4 ? MARCH2_C<STK> : MARCH_C<STK>);
  __shared__ union U {
    RowScratch<T> rows;
    float4 align;
    T cst[(SHARE ? MARCH_BLOCK >> SHARE : 1) * NC];
    __device__ U() {}
  } sh;
  // row blocks among the first b blocks: b rows / blocks
  const uint32_t b = blockIdx.x;
  const uint32_t r0 = (uint32_t)((uint64_t)b * (uint32_t)rows / gridDim.x);
  const uint32_t r1 = (uint32_t)((uint64_t)(b + 1) * (uint32_t)rows / gridDim.x);
  if (r1 != r0) {
    rows_block<T, OP, STK>(L, mc, fl, a, (int)r0, sh.rows, a.partial);
    return;
  }
  const int q = (int)(b - r0), macro = SHARE ? q * (MARCH_BLOCK >> SHARE) : q / per_macro;
  const int block = SHARE ? 0 : q - macro * per_macro;
  double* partial = a.partial ? a.partial + RowBlocks<T, STK>(L).partials() + q : nullptr;
  if constexpr (sizeof(T) == 4)
    march2_block<OP, GEN, STK, KB, SHARE>(L, mc, macro, block, fl, a, sh.cst, partial);
  else
    march_block<T, OP, GEN, STK>(L, mc, macro, block, fl, a, sh.cst, partial);
}

template <typename T, int OP, int STK>
int launch(const LevelDev& L, const MacroConsts<T>* mc, const OpFlags& fl, const SweepArgs<T>& a, cudaStream_t s,
           int64_t* partial_count) {
  const bool gen = !(fl.physical == 1 && fl.khat_edge == 0);
  const RowBlocks<T, STK> R(L);
  const int columns = L.ncolumns[sizeof(T) == 8];
  // Macros of up to 32 columns (4 or 8 intervals per edge) share blocks of four in FP32: a block each left one of
  // its warps busy (apply on 3072 macros of 4 / 8 intervals 105 / 123 us; so, and with build_rows' rule for
  // small faces and edges, 58 / 100).  Only with more macros
  // than SMs (fewer blocks all run at once), and not in FP64, where a warp's instructions fill an SM and the
  // rows are most of such a sweep (831 us against 891).  A kernel of its own, with the run-time flags and the
  // FP32 copy of a BF16 coefficient: the general index arithmetic cost the large sweeps 4 to 7 %.
  const bool share = sizeof(T) == 4 && L.nmacro > 152 && columns <= 32;
  const int per = std::max(1, (columns + MARCH_BLOCK - 1) / MARCH_BLOCK);
  const int64_t inner = columns == 0 ? 0 : share ? (L.nmacro + 3) / 4 : (int64_t)per * L.nmacro;
  if (partial_count) *partial_count = inner + R.partials();
  if (inner + R.total == 0) return 0;
  if (inner + R.total > INT32_MAX) return (int)cudaErrorInvalidValue;
  const unsigned g = (unsigned)(inner + R.total);
  if constexpr (sizeof(T) == 4) {
    if (share) {
      k_sweep<T, OP, 1, STK, 0, 5><<<g, MARCH_BLOCK, 0, s>>>(L, mc, fl, a, per, R.total);
      return (int)cudaGetLastError();
    }
  }
  // a kernel with the variant and khat rule folded in (FP64: 1.77 against 1.94 ms for a residual on
  // 129^3 nodes), but for FP32 Stokes, where the run-time flags do not show
  if constexpr (sizeof(T) == 4 && STK) {
    k_sweep<T, OP, 1, STK, 0><<<g, MARCH_BLOCK, 0, s>>>(L, mc, fl, a, per, R.total);
  } else {
    if (gen)
      k_sweep<T, OP, 1, STK, 0><<<g, MARCH_BLOCK, 0, s>>>(L, mc, fl, a, per, R.total);
    else if (sizeof(T) == 4 && a.k16)
      k_sweep<T, OP, 0, STK, (sizeof(T) == 4)><<<g, MARCH_BLOCK, 0, s>>>(L, mc, fl, a, per, R.total);
    else
      k_sweep<T, OP, 0, STK, 0><<<g, MARCH_BLOCK, 0, s>>>(L, mc, fl, a, per, R.total);
  }
  return (int)cudaGetLastError();
}

}  // namespace
}  // namespace hhg
