// Rows of nodes on the macro skeleton (faces, edges and vertices of the macro mesh, Sec. 2.2 of
// arXiv 1908.08666): device code of the skeleton part of a sweep, run by k_rows alone (hhg_rows_launch.cuh)
// and by k_sweep in blocks between those of the macro interiors.
//
// A lane takes one incidence of a node (the node seen from one of the macros that hold it) and
// evaluates that macro's part of the row; the parts are summed in an order that is the same for every
// copy of the node, and each lane writes its own copy.  In a macro the row of point p runs over the
// stencil directions d whose neighbour p + d lies in the macro:
//   - scaled block (Lemma 2.1) when p + d is macro-interior (symmetric interface rule),
//   - else nodal integration a_h over the macro's elements that hold the edge (p, p + d), which
//     are the pairs of cyclically consecutive ring nodes of the edge that both lie in the macro.
// Rows are in difference form: the centre block is minus the sum of the others.
//
// Nodes inside a macro face or edge: what depends on the direction is fixed by the kind of face or edge
// that the macro sees (prim_incidence, unrolled over the directions); a lane per node, all lanes of a warp
// in the same macro.  Vertices, with up to dozens of macros, and the few nodes of faces and edges on the
// coarsest level: incidence_lane, half a warp per macro, a lane per direction, the ring's coefficients by
// shuffles.
//
// What bounds them: latency, and on meshes of many macros instructions.  There are few such nodes (2 % of
// 129^3), but most of a face's or edge's neighbours lie in different rows.  FP32 apply on 384 macros at
// level 5, whole sweep: 209 us with an unrolled kernel per node kind (rows 93 + 62), 112 with this layout
// (160 with half a warp per incidence for the nodes of edges too).
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "hhg_internal.h"
#include "hhg_launch.h"
#include "hhg_row.cuh"

namespace hhg {

namespace {

constexpr int ROWS_BLOCK = 128;
constexpr int ROWS_WARPS = ROWS_BLOCK / 32;
constexpr int DIR_PER_THREAD = 4;  // Dirichlet entries a thread copies, their loads in flight together

// per direction d: its lattice offset, and its ring in cyclic order, closed
struct alignas(16) DirTable {
  int8_t d[3];
  uint8_t red;
  uint8_t cyc[7];
  uint8_t pad[5];
};
__constant__ DirTable c_dir[16];  // one copy per translation unit, filled by upload_direction_tables

// COUNT values of a constant table, in 16-byte words
template <typename T, int COUNT, int N>
__device__ __forceinline__ void load_values(const T* __restrict__ p, T (&v)[N]) {
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int q = 0; q < COUNT; q += 4) {
      const float4 f = __ldg(reinterpret_cast<const float4*>(p + q));
      v[q] = f.x;
      v[q + 1] = f.y;
      v[q + 2] = f.z;
      v[q + 3] = f.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < COUNT; q += 2) {
      const double2 f = __ldg(reinterpret_cast<const double2*>(p + q));
      v[q] = f.x;
      v[q + 1] = f.y;
    }
  }
}
// values of MacroConsts::el that the velocity rows need, and the Stokes rows
template <typename T, int STK>
constexpr int EL_COUNT = STK ? 16 : sizeof(T) == 4 ? 12 : 10;

template <typename T>
struct RowSum {
  T ax = 0, ay = 0, az = 0, dgx = 0, dgy = 0, dgz = 0, yp = 0;
};

// difference x_{p+d} - x_p of the velocity and of the pressure; pg = p_{p+d} + p_p / 3 (B^T: an
// element's four pressures, a third of the point's own on each of its three edges)
template <typename T>
struct EdgeDiff {
  T dx, dy, dz, dp, pg;
};

// an element's nodal-integration block, its nodal coefficients summing to ks
template <typename T, bool DIAG, int STK>
__device__ __forceinline__ void element_term(const T (&v)[16], T ks, bool vel, const EdgeDiff<T>& D, RowSum<T>& s) {
  if (vel) {
    const T kb = (T)0.25 * ks;
    s.ax = fma(kb, fma(v[0], D.dx, fma(v[1], D.dy, v[2] * D.dz)), s.ax);
    s.ay = fma(kb, fma(v[3], D.dx, fma(v[4], D.dy, v[5] * D.dz)), s.ay);
    s.az = fma(kb, fma(v[6], D.dx, fma(v[7], D.dy, v[8] * D.dz)), s.az);
    if (DIAG) {
      s.dgx = fma(-kb, v[0], s.dgx);
      s.dgy = fma(-kb, v[4], s.dgy);
      s.dgz = fma(-kb, v[8], s.dgz);
    }
  }
  if (STK) {
    s.yp = fma(v[9], D.dx, fma(v[10], D.dy, fma(v[11], D.dz, fma(v[15], D.dp, s.yp))));
    s.ax = fma(v[12], D.pg, s.ax);
    s.ay = fma(v[13], D.pg, s.ay);
    s.az = fma(v[14], D.pg, s.az);
  }
}

// the scaled block of a direction from its ring's coefficients kr in cyclic order
template <typename T, bool DIAG>
__device__ __forceinline__ void scaled_term(const T (&v)[16], bool red, T k0, T kd, const T (&kr)[6],
                                            const OpFlags& fl, const EdgeDiff<T>& D, RowSum<T>& s) {
  T rs = (kr[0] + kr[1]) + (kr[2] + kr[3]);
  T e0 = kr[0] - kr[2], e1 = kr[1] - kr[3], wx, wy, wz;
  if (red) {
    rs += kr[4] + kr[5];
    e0 = kr[0] - kr[3];
    e1 = kr[1] - kr[4];
    const T e2 = kr[2] - kr[5];
    wx = e2 * v[12];
    wy = e2 * v[13];
    wz = e2 * v[14];
  } else {
    wx = wy = wz = 0;
  }
  wx = fma(e0, v[6], fma(e1, v[9], wx));
  wy = fma(e0, v[7], fma(e1, v[10], wy));
  wz = fma(e0, v[8], fma(e1, v[11], wz));
  const T kh = fl.khat_edge ? (T)0.5 * (k0 + kd) : fma(red ? (T)(1.0 / 12.0) : (T)0.125, rs, (T)0.25 * (k0 + kd));
  const T vx = kh * D.dx, vy = kh * D.dy, vz = kh * D.dz;
  s.ax = fma(v[0], vx, fma(v[3], vy, fma(v[4], vz, s.ax)));
  s.ay = fma(v[3], vx, fma(v[1], vy, fma(v[5], vz, s.ay)));
  s.az = fma(v[4], vx, fma(v[5], vy, fma(v[2], vz, s.az)));
  if (fl.physical) {
    s.ax = fma(wy, D.dz, fma(-wz, D.dy, s.ax));
    s.ay = fma(wz, D.dx, fma(-wx, D.dz, s.ay));
    s.az = fma(wx, D.dy, fma(-wy, D.dx, s.az));
  }
  if (DIAG) {
    s.dgx = fma(-kh, v[0], s.dgx);
    s.dgy = fma(-kh, v[1], s.dgy);
    s.dgz = fma(-kh, v[2], s.dgz);
  }
}

// the Stokes blocks of a direction all of whose elements lie in the macro
template <typename T>
__device__ __forceinline__ void stokes_term(const T (&v)[8], const EdgeDiff<T>& D, RowSum<T>& s) {
  s.yp = fma(v[0], D.dx, fma(v[1], D.dy, fma(v[2], D.dz, fma(v[6], D.dp, s.yp))));
  s.ax = fma(v[3], D.pg, s.ax);
  s.ay = fma(v[4], D.pg, s.ay);
  s.az = fma(v[5], D.pg, s.az);
}

// One direction of one macro's part of a row: lanes 0 .. 13 and 16 .. 29 of a warp take the directions
// of two incidences (valid: the lane's incidence exists; all lanes call this together).
template <typename T, bool DIAG, int STK>
__device__ __forceinline__ void incidence_lane(const LevelDev& L, const MacroConsts<T>* __restrict__ mc,
                                               const OpFlags& fl, const SweepArgs<T>& a, const SkelInc& it, bool valid,
                                               bool vel, RowSum<T>& s) {
  const int lane = threadIdx.x & 31, d = lane & 15, half = lane & 16;
  const DirTable t = c_dir[d];
  const bool red = t.red;
  const int n = L.n;
  const int64_t E = L.entries;
  const T* __restrict__ px = a.x + (int64_t)it.macro * L.nt;
  const T* __restrict__ pk = a.k + (int64_t)it.macro * L.nt;
  const int qi = it.i + t.d[0], qj = it.j + t.d[1], qk = it.k + t.d[2], ql = n - qi - qj - qk;
  const bool in = valid && d < NDIR && (qi | qj | qk | ql) >= 0;
  const bool interior = qi >= 1 && qj >= 1 && qk >= 1 && ql >= 1;
  T k0 = 0, kd = 0, x0 = 0, y0 = 0, z0 = 0, p0 = 0;
  EdgeDiff<T> D{0, 0, 0, 0, 0};
  if (in) {
    const int c0 = lattice_index32(n, it.i, it.j, it.k), c1 = lattice_index32(n, qi, qj, qk);
    k0 = pk[c0];
    kd = pk[c1];
    x0 = px[c0];
    y0 = px[c0 + E];
    z0 = px[c0 + 2 * E];
    D.dx = px[c1] - x0;
    D.dy = px[c1 + E] - y0;
    D.dz = px[c1 + 2 * E] - z0;
    if (STK) {
      p0 = px[c0 + 3 * E];
      const T pd = px[c1 + 3 * E];
      D.dp = pd - p0;
      D.pg = fma((T)(1.0 / 3.0), p0, pd);
    }
  }
  const unsigned inside = __ballot_sync(0xffffffffu, in) >> half;
  T kr[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) kr[q] = __shfl_sync(0xffffffffu, kd, half + t.cyc[q]);
  if (!in) return;
  const MacroConsts<T>& C = mc[it.macro];
  if (interior && !fl.practical) {
    if (vel) {
      T v[16];
      load_values<T, 16>(&C.sc[d][0], v);
      scaled_term<T, DIAG>(v, red, k0, kd, kr, fl, D, s);
    }
    if (STK) {
      T v[8];
      load_values<T, 8>(&C.sb[d][0], v);
      stokes_term<T>(v, D, s);
    }
    return;
  }
  const T ke = k0 + kd;
  // elements whose constants are requested together
  constexpr int UE = sizeof(T) == 4 && !STK ? 6 : 3;
#pragma unroll
  for (int e0 = 0; e0 < 6; e0 += UE) {
    T v[UE][16];
    bool ok[UE];
#pragma unroll
    for (int e = 0; e < UE; ++e) {
      ok[e] = (e0 + e < 4 || red) && ((inside >> t.cyc[e0 + e]) & (inside >> t.cyc[e0 + e + 1]) & 1u);
      if (ok[e]) load_values<T, EL_COUNT<T, STK>>(&C.el[d][e0 + e][0], v[e]);
    }
#pragma unroll
    for (int e = 0; e < UE; ++e) {
      // a four-element ring is closed by its fifth entry
      const int q = e0 + e;
      const T kn = q == 5 || (q == 3 && !red) ? kr[0] : kr[q < 5 ? q + 1 : 0];
      if (ok[e]) element_term<T, DIAG, STK>(v[e], ke + (kr[q] + kn), vel, D, s);
    }
  }
}

// Primitives of a macro whose interiors hold the skeleton's nodes: faces 0 .. 3 (i + j + k = n, i = 0, j =
// 0, k = 0) and edges 4 .. 9, the meets of two faces (0 1, 0 2, 0 3, 1 2, 1 3, 2 3).  Which directions
// stay in the macro from a point inside the primitive, and which can end at a macro-interior point: the
// representative point on a lattice with 16 intervals decides, at compile time.  Only next to the
// primitive's ends an inward direction may end on the skeleton instead.
__device__ __forceinline__ constexpr bool prim_on_face(int F, int f) {
  return F < 4 ? F == f : F == 4 ? f < 2 : F == 5 ? f == 0 || f == 2 : F == 6 ? f == 0 || f == 3
                        : F == 7 ? f == 1 || f == 2 : F == 8 ? f == 1 || f == 3 : f >= 2;
}
__device__ __forceinline__ constexpr int prim_coord(int F, int c) {  // c: 0 n - i - j - k, 1 i, 2 j, 3 k
  return prim_on_face(F, c) ? 0 : F < 4 ? (c == (F == 0 ? 3 : 0) ? 6 : 5) : 8;
}
__device__ __forceinline__ bool prim_dir_valid(int F, int d) {
  return lattice_inside(16, prim_coord(F, 1) + dir_di(d), prim_coord(F, 2) + dir_dj(d), prim_coord(F, 3) + dir_dk(d));
}
__device__ __forceinline__ bool prim_dir_inward(int F, int d) {
  return lattice_interior(16, prim_coord(F, 1) + dir_di(d), prim_coord(F, 2) + dir_dj(d), prim_coord(F, 3) + dir_dk(d));
}

// Which form rows inside faces and edges take.  FP32: prim_incidence, unrolled.  FP64: loop_incidence, and two
// warps take a side of a face block.
template <typename T>
constexpr bool ROWS_UNROLLED = sizeof(T) == 4;
template <typename T>
constexpr int FACE_GROUPS = sizeof(T) == 8 ? 2 : 1;

// Scratch of the run-time form: neighbour coefficients and entries, a column per thread.
template <typename T>
struct RowColumns {
  T k[NDIR][ROWS_BLOCK];
  int at[NDIR][ROWS_BLOCK];
};

struct NoColumns {};
template <typename T>
struct RowScratch {
  T share[6 * ROWS_BLOCK];  // sums that warps exchange
  std::conditional_t<ROWS_UNROLLED<T>, NoColumns, RowColumns<T>> columns;
};

// The same sums as prim_incidence in a loop over the directions, with run-time ring indices.  FP64: a
// warp's FP64 instruction takes 64 cycles, so the loop's integer work hides behind it, and ten kinds of
// face and edge need not be unrolled.  groups > 1: only every groups-th direction, from `group` on (several
// warps share the points, since a row's chain of about 450 instructions is 15 us).
template <typename T, bool DIAG, int STK>
__device__ __forceinline__ void loop_incidence(const LevelDev& L, const MacroConsts<T>& C, const T* __restrict__ px,
                                               const T* __restrict__ pk, const OpFlags& fl, int i, int j, int k,
                                               bool vel, int group, int groups, RowColumns<T>& sh, RowSum<T>& s) {
  const int tid = threadIdx.x;
  const int n = L.n;
  const int64_t E = L.entries;
  const int l = n - i - j - k;
  const int c0 = lattice_index32(n, i, j, k);
  uint32_t inside = 0, interior = 0;
  {
    int nb[NDIR];
    lattice_neighbours(n, i, j, k, nb);
#pragma unroll
    for (int d = 0; d < NDIR; ++d) {
      const int di = dir_di(d), dj = dir_dj(d), dk = dir_dk(d), dl = -di - dj - dk;
      const int qi = i + di, qj = j + dj, qk = k + dk, ql = l + dl;
      const bool in = (qi | qj | qk | ql) >= 0;
      if (in) inside |= 1u << d;
      if (qi >= 1 && qj >= 1 && qk >= 1 && ql >= 1) interior |= 1u << d;
      const int q = in ? nb[d] : c0;
      sh.k[d][tid] = pk[q];
      sh.at[d][tid] = q;
    }
  }
  const T k0 = pk[c0], x0 = px[c0], y0 = px[c0 + E], z0 = px[c0 + 2 * E];
  const T p0 = STK ? px[c0 + 3 * E] : (T)0;
  const uint32_t scaled = fl.practical ? 0u : interior;
  // the neighbour's values are requested one direction ahead
  T xn, yn, zn, pn = 0;
  auto fetch = [&](int d) {
    const T* q = px + sh.at[d][tid];
    xn = q[0];
    yn = q[E];
    zn = q[2 * E];
    if (STK) pn = q[3 * E];
  };
  auto next = [&](int d, int steps) {  // the steps-th direction from d on that stays in the macro
    while (d < NDIR && (!((inside >> d) & 1u) || steps-- > 0)) ++d;
    return d;
  };
  int d = next(0, group);
  if (d < NDIR) fetch(d);
#pragma unroll 1
  while (d < NDIR) {
    EdgeDiff<T> D{xn - x0, yn - y0, zn - z0, pn - p0, STK ? fma((T)(1.0 / 3.0), p0, pn) : (T)0};
    const int dn = next(d + 1, groups - 1);
    if (dn < NDIR) fetch(dn);
    const DirTable t = c_dir[d];
    const bool red = t.red;
    const T kd = sh.k[d][tid];
    if ((scaled >> d) & 1u) {
      if (vel) {
        T v[16], kr[6];
        load_values<T, 16>(&C.sc[d][0], v);
#pragma unroll
        for (int q = 0; q < 6; ++q) kr[q] = sh.k[t.cyc[q]][tid];
        scaled_term<T, DIAG>(v, red, k0, kd, kr, fl, D, s);
      }
      if (STK) {
        T v[8];
        load_values<T, 8>(&C.sb[d][0], v);
        stokes_term<T>(v, D, s);
      }
    } else {
      const T ke = k0 + kd;
      const int ne = red ? 6 : 4;
#pragma unroll 2
      for (int e = 0; e < ne; ++e) {
        const int ra = t.cyc[e], rb = t.cyc[e + 1];
        if (!((inside >> ra) & (inside >> rb) & 1u)) continue;
        T v[16];
        load_values<T, EL_COUNT<T, STK>>(&C.el[d][e][0], v);
        element_term<T, DIAG, STK>(v, ke + (sh.k[ra][tid] + sh.k[rb][tid]), vel, D, s);
      }
    }
    d = dn;
  }
}

// One macro's part of the row of such a point (group G of its directions): six directions in the face (a_h over the half of the
// edge's elements that lies in the macro), four inward ones (the scaled block where they end at a
// macro-interior point, else, and with the practical rule or nodal integration, a_h over all of the
// edge's elements).  All lanes read the same constants.  near: points next to the face's edges.
template <typename T, int F, bool DIAG, int STK>
__device__ __forceinline__ void prim_incidence(const MacroConsts<T>& C, const T* __restrict__ px,
                                               const T* __restrict__ pk, int64_t E, int n, int i, int j, int k,
                                               const OpFlags& fl, bool vel, bool near, RowSum<T>& s) {
  int nb[NDIR];
  lattice_neighbours(n, i, j, k, nb);
  const int c0 = lattice_index32(n, i, j, k);
  T kv[NDIR], x[NDIR], y[NDIR], z[NDIR], p[STK ? NDIR : 1];
#pragma unroll
  for (int d = 0; d < NDIR; ++d) {
    kv[d] = 0;
    if (!prim_dir_valid(F, d)) continue;
    kv[d] = pk[nb[d]];
    x[d] = px[nb[d]];
    y[d] = px[nb[d] + E];
    z[d] = px[nb[d] + 2 * E];
    if (STK) p[STK ? d : 0] = px[nb[d] + 3 * E];
  }
  const T k0 = pk[c0], x0 = px[c0], y0 = px[c0 + E], z0 = px[c0 + 2 * E];
  const T p0 = STK ? px[c0 + 3 * E] : (T)0;
  const bool scaled = !fl.practical;
#pragma unroll
  for (int d = 0; d < NDIR; ++d) {
    if (!prim_dir_valid(F, d)) continue;
    EdgeDiff<T> D{x[d] - x0, y[d] - y0, z[d] - z0, 0, 0};
    if (STK) {
      D.dp = p[STK ? d : 0] - p0;
      D.pg = fma((T)(1.0 / 3.0), p0, p[STK ? d : 0]);
    }
    if (prim_dir_inward(F, d) && scaled &&
        (!near || lattice_interior(n, i + dir_di(d), j + dir_dj(d), k + dir_dk(d)))) {
      if (vel) {
        T v[16], kr[6];
        load_values<T, 16>(&C.sc[d][0], v);
#pragma unroll
        for (int q = 0; q < 6; ++q) kr[q] = kv[ring_cyc(d, q)];
        scaled_term<T, DIAG>(v, dir_red(d), k0, kv[d], kr, fl, D, s);
      }
      if (STK) {
        T v[8];
        load_values<T, 8>(&C.sb[d][0], v);
        stokes_term<T>(v, D, s);
      }
      continue;
    }
    const T ke = k0 + kv[d];
#pragma unroll
    for (int e = 0; e < 6; ++e) {
      if (e >= 4 && !dir_red(d)) break;
      if (!prim_dir_valid(F, ring_cyc(d, e)) || !prim_dir_valid(F, ring_cyc(d, e + 1))) continue;
      T v[16];
      load_values<T, EL_COUNT<T, STK>>(&C.el[d][e][0], v);
      element_term<T, DIAG, STK>(v, ke + (kv[ring_cyc(d, e)] + kv[ring_cyc(d, e + 1)]), vel, D, s);
    }
  }
}

// What a lane does with its node's sums: every copy receives the row.
template <typename T, int OP, int STK>
__device__ __forceinline__ void write_row(const SweepArgs<T>& a, int64_t e, int64_t E, const RowSum<T>& s, bool vdir,
                                          double& r2) {
  const T x0 = a.x[e], y0 = a.x[e + E], z0 = a.x[e + 2 * E];
  if constexpr (STK)
    stokes_epilogue<T, OP>(a, e, E, s.ax, s.ay, s.az, s.yp, x0, y0, z0, vdir, r2);
  else
    epilogue<T, OP>(a, e, E, s.ax, s.ay, s.az, s.dgx, s.dgy, s.dgz, x0, y0, z0, r2);
}

// A block of 32 face nodes, two (FP64: four) warps: warp q evaluates them from the macro on side q % 2,
// the sums are exchanged through shared memory (added in the same order in every warp) and each side's
// first warp writes its copies.  All threads of the launch's block call this together (b < 0: nothing
// to do).
template <typename T, int OP, int STK>
__device__ __forceinline__ double face_block(const LevelDev& L, const MacroConsts<T>* __restrict__ mc,
                                             const OpFlags& fl, const SweepArgs<T>& a, int b, RowScratch<T>& sh) {
  constexpr bool DIAG = OP == OP_JACOBI || OP == OP_CHEBY || OP == OP_DIAG;
  constexpr int G = FACE_GROUPS<T>;
  const int lane = threadIdx.x & 31, side = (threadIdx.x >> 5) & 1, group = G > 1 ? (threadIdx.x >> 6) % G : 0;
  FaceBlock B{{-1, -1}, {0, 0}, 0, 0, 0, 0};
  FacePoint P{0, 0, 0, 0};
  if (b >= 0) {
    B = L.face_blocks[STK][b];
    P = L.face_points[STK][64 * (int64_t)b + 32 * side + lane];
  }
  const int m = side == 0 ? B.macro[0] : B.macro[1];
  const bool valid = m >= 0 && lane < B.count;
  const bool vel = !STK || !B.vdir, near = B.near;
  RowSum<T> s;
  if (valid) {
    const T* px = a.x + (int64_t)m * L.nt;
    const T* pk = a.k + (int64_t)m * L.nt;
    const int64_t E = L.entries;
    if constexpr (!ROWS_UNROLLED<T>) {
      loop_incidence<T, DIAG, STK>(L, mc[m], px, pk, fl, P.i, P.j, P.k, vel, group, G, sh.columns, s);
    } else {
      switch (side == 0 ? B.face[0] : B.face[1]) {
        case 0: prim_incidence<T, 0, DIAG, STK>(mc[m], px, pk, E, L.n, P.i, P.j, P.k, fl, vel, near, s); break;
        case 1: prim_incidence<T, 1, DIAG, STK>(mc[m], px, pk, E, L.n, P.i, P.j, P.k, fl, vel, near, s); break;
        case 2: prim_incidence<T, 2, DIAG, STK>(mc[m], px, pk, E, L.n, P.i, P.j, P.k, fl, vel, near, s); break;
        default: prim_incidence<T, 3, DIAG, STK>(mc[m], px, pk, E, L.n, P.i, P.j, P.k, fl, vel, near, s); break;
      }
    }
  }
  T* share = sh.share;
  T* own = share + threadIdx.x;
  own[0] = s.ax;
  own[ROWS_BLOCK] = s.ay;
  own[2 * ROWS_BLOCK] = s.az;
  own[3 * ROWS_BLOCK] = STK ? s.yp : s.dgx;
  own[4 * ROWS_BLOCK] = s.dgy;
  own[5 * ROWS_BLOCK] = s.dgz;
  __syncthreads();
  double r2 = 0.0;
  if (valid && group == 0) {
    RowSum<T> r;
#pragma unroll
    for (int q = 0; q < 2 * G; ++q) {
      const T* p = share + (G > 1 ? 0 : threadIdx.x & ~63) + 32 * q + lane;
      r.ax += p[0];
      r.ay += p[ROWS_BLOCK];
      r.az += p[2 * ROWS_BLOCK];
      if (STK) r.yp += p[3 * ROWS_BLOCK];
      if (DIAG) {
        r.dgx += p[3 * ROWS_BLOCK];
        r.dgy += p[4 * ROWS_BLOCK];
        r.dgz += p[5 * ROWS_BLOCK];
      }
    }
    double tmp = 0.0;
    write_row<T, OP, STK>(a, (int64_t)m * L.nt + lattice_index32(L.n, P.i, P.j, P.k), L.entries, r, STK && B.vdir, tmp);
    if (side == 0) r2 = tmp;
  }
  return r2;
}

// A block of up to 32 nodes of one macro edge: warp w takes the macros w, w + 4, ... that hold the edge,
// the warps' sums are added in order, and each warp writes its macros' copies.
template <typename T, int OP, int STK>
__device__ __forceinline__ double edge_block(const LevelDev& L, const MacroConsts<T>* __restrict__ mc,
                                             const OpFlags& fl, const SweepArgs<T>& a, int b, RowScratch<T>& sh) {
  constexpr bool DIAG = OP == OP_JACOBI || OP == OP_CHEBY || OP == OP_DIAG;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const EdgeBlock B = L.edge_blocks[STK][b];
  const bool valid = lane < B.count, vel = !STK || !B.vdir;
  const int64_t E = L.entries;
  RowSum<T> s;
  for (int q = w; q < B.macros; q += ROWS_WARPS) {
    const EdgeSide S = L.edge_sides[STK][B.first + q];
    const int i = S.at[0] + lane * S.step[0], j = S.at[1] + lane * S.step[1], k = S.at[2] + lane * S.step[2];
    const T* px = a.x + (int64_t)S.macro * L.nt;
    const T* pk = a.k + (int64_t)S.macro * L.nt;
    const MacroConsts<T>& C = mc[S.macro];
    if (!valid) continue;
    if constexpr (!ROWS_UNROLLED<T>) {
      loop_incidence<T, DIAG, STK>(L, C, px, pk, fl, i, j, k, vel, 0, 1, sh.columns, s);
    } else {
      switch (S.edge) {
        case 4: prim_incidence<T, 4, DIAG, STK>(C, px, pk, E, L.n, i, j, k, fl, vel, true, s); break;
        case 5: prim_incidence<T, 5, DIAG, STK>(C, px, pk, E, L.n, i, j, k, fl, vel, true, s); break;
        case 6: prim_incidence<T, 6, DIAG, STK>(C, px, pk, E, L.n, i, j, k, fl, vel, true, s); break;
        case 7: prim_incidence<T, 7, DIAG, STK>(C, px, pk, E, L.n, i, j, k, fl, vel, true, s); break;
        case 8: prim_incidence<T, 8, DIAG, STK>(C, px, pk, E, L.n, i, j, k, fl, vel, true, s); break;
        default: prim_incidence<T, 9, DIAG, STK>(C, px, pk, E, L.n, i, j, k, fl, vel, true, s); break;
      }
    }
  }
  T* share = sh.share;
  T* own = share + threadIdx.x;
  own[0] = s.ax;
  own[ROWS_BLOCK] = s.ay;
  own[2 * ROWS_BLOCK] = s.az;
  own[3 * ROWS_BLOCK] = STK ? s.yp : s.dgx;
  own[4 * ROWS_BLOCK] = s.dgy;
  own[5 * ROWS_BLOCK] = s.dgz;
  __syncthreads();
  RowSum<T> r;
#pragma unroll
  for (int q = 0; q < ROWS_WARPS; ++q) {
    const T* p = share + 32 * q + lane;
    r.ax += p[0];
    r.ay += p[ROWS_BLOCK];
    r.az += p[2 * ROWS_BLOCK];
    if (STK) r.yp += p[3 * ROWS_BLOCK];
    if (DIAG) {
      r.dgx += p[3 * ROWS_BLOCK];
      r.dgy += p[4 * ROWS_BLOCK];
      r.dgz += p[5 * ROWS_BLOCK];
    }
  }
  double r2 = 0.0;
  for (int q = w; q < B.macros && valid; q += ROWS_WARPS) {
    const EdgeSide S = L.edge_sides[STK][B.first + q];
    const int i = S.at[0] + lane * S.step[0], j = S.at[1] + lane * S.step[1], k = S.at[2] + lane * S.step[2];
    double tmp = 0.0;
    write_row<T, OP, STK>(a, (int64_t)S.macro * L.nt + lattice_index32(L.n, i, j, k), E, r, STK && B.vdir, tmp);
    if (q == 0) r2 = tmp;
  }
  return r2;
}

// A block of macro vertices (EvWarp): the sums of a warp by a butterfly, those of a
// node's warps in order, and the node's threads write its copies.
template <typename T, int OP, int STK>
__device__ __forceinline__ double ev_block(const LevelDev& L, const MacroConsts<T>* __restrict__ mc, const OpFlags& fl,
                                           const SweepArgs<T>& a, int b, RowScratch<T>& sh) {
  constexpr bool DIAG = OP == OP_JACOBI || OP == OP_CHEBY || OP == OP_DIAG;
  const EvWarp W = L.ev_warps[STK][ROWS_WARPS * b + (threadIdx.x >> 5)];
  RowSum<T> s;
  if (W.first >= 0) {
    const int half = (threadIdx.x >> 4) & 1;
    for (int q0 = 2 * W.w; q0 < W.count; q0 += 2 * W.warps) {
      const bool valid = q0 + half < W.count;
      incidence_lane<T, DIAG, STK>(L, mc, fl, a, L.skel_inc[W.first + (valid ? q0 + half : q0)], valid, !(STK && W.vdir),
                                   s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s.ax += __shfl_xor_sync(0xffffffffu, s.ax, o);
      s.ay += __shfl_xor_sync(0xffffffffu, s.ay, o);
      s.az += __shfl_xor_sync(0xffffffffu, s.az, o);
      if (DIAG) {
        s.dgx += __shfl_xor_sync(0xffffffffu, s.dgx, o);
        s.dgy += __shfl_xor_sync(0xffffffffu, s.dgy, o);
        s.dgz += __shfl_xor_sync(0xffffffffu, s.dgz, o);
      }
      if (STK) s.yp += __shfl_xor_sync(0xffffffffu, s.yp, o);
    }
  }
  T* share = sh.share;
  if ((threadIdx.x & 31) == 0) {
    T* p = share + 8 * (threadIdx.x >> 5);
    p[0] = s.ax;
    p[1] = s.ay;
    p[2] = s.az;
    p[3] = STK ? s.yp : s.dgx;
    p[4] = s.dgy;
    p[5] = s.dgz;
  }
  __syncthreads();
  double r2 = 0.0;
  if (W.first >= 0) {
    RowSum<T> r;
    for (int q = W.w0; q < W.w0 + W.warps; ++q) {
      const T* p = share + 8 * q;
      r.ax += p[0];
      r.ay += p[1];
      r.az += p[2];
      if (STK) r.yp += p[3];
      if (DIAG) {
        r.dgx += p[3];
        r.dgy += p[4];
        r.dgz += p[5];
      }
    }
    for (int q = 32 * W.w + (threadIdx.x & 31); q < W.count; q += 32 * W.warps) {
      const SkelInc I = L.skel_inc[W.first + q];
      double tmp = 0.0;
      write_row<T, OP, STK>(a, (int64_t)I.macro * L.nt + lattice_index32(L.n, I.i, I.j, I.k), L.entries, r,
                            STK && W.vdir, tmp);
      if (q == 0) r2 = tmp;
    }
  }
  return r2;
}

// Blocks of the skeleton part of a sweep, in this order: macro vertices, macro edges, face
// blocks (two a block, FP64 one), Dirichlet entries (identity rows, every copy; not in the Stokes lists).
template <typename T, int STK>
struct RowBlocks {
  static constexpr int FACES = ROWS_WARPS / (2 * FACE_GROUPS<T>);  // face blocks per block
  int nfaces, ev_blocks, edge_blocks, face_blocks, total;
  __host__ __device__ explicit RowBlocks(const LevelDev& L)
      : nfaces(L.nface_blocks[STK]),
        ev_blocks(L.nev_blocks[STK]),
        edge_blocks(L.nedge_blocks[STK]),
        face_blocks((nfaces + FACES - 1) / FACES),
        total(ev_blocks + edge_blocks + face_blocks +
              (STK ? 0 : (int)((L.ndir_entries + ROWS_BLOCK * DIR_PER_THREAD - 1) / (ROWS_BLOCK * DIR_PER_THREAD)))) {}
  // blocks that hold rows with a residual
  __host__ __device__ int partials() const { return ev_blocks + edge_blocks + face_blocks; }
};

// Block b of them; its partial sum of |r|^2 goes to partial[b].
template <typename T, int OP, int STK>
__device__ __forceinline__ void rows_block(const LevelDev& L, const MacroConsts<T>* __restrict__ mc, const OpFlags& fl,
                                           const SweepArgs<T>& a, int b, RowScratch<T>& sh, double* partial) {
  const RowBlocks<T, STK> R(L);
  const int64_t E = L.entries;
  if (b >= R.partials()) {
    if (STK) return;
    const int64_t t = (int64_t)(b - R.partials()) * ROWS_BLOCK * DIR_PER_THREAD + threadIdx.x;
#pragma unroll
    for (int q = 0; q < DIR_PER_THREAD; ++q) {
      if (t + q * ROWS_BLOCK >= L.ndir_entries) break;
      const int64_t e = L.dir_entries[t + q * ROWS_BLOCK];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        a.out[e + c * E] = OP == OP_RESID ? (T)0 : OP == OP_DIAG ? (T)1 : __ldg(a.x + e + c * E);
        if (OP == OP_CHEBY) a.dout[e + c * E] = 0;
      }
    }
    return;
  }
  double r2;
  if (b >= R.ev_blocks + R.edge_blocks) {
    const int f = (b - R.ev_blocks - R.edge_blocks) * R.FACES + (R.FACES > 1 ? threadIdx.x >> 6 : 0);
    r2 = face_block<T, OP, STK>(L, mc, fl, a, f < R.nfaces ? f : -1, sh);
  } else if (b >= R.ev_blocks) {
    r2 = edge_block<T, OP, STK>(L, mc, fl, a, b - R.ev_blocks, sh);
  } else {
    r2 = ev_block<T, OP, STK>(L, mc, fl, a, b, sh);
  }
  if (OP == OP_RESID && partial != nullptr) block_sum_store<T>(r2, partial + b);
}

// fills this translation unit's ring tables used with run-time direction indices
inline int upload_tables() {
  DirTable t[16] = {};
  for (int d = 0; d < 16; ++d) {
    const int e = d < NDIR ? d : 0;
    t[d].d[0] = (int8_t)dir_di(e);
    t[d].d[1] = (int8_t)dir_dj(e);
    t[d].d[2] = (int8_t)dir_dk(e);
    t[d].red = dir_red(e);
    for (int q = 0; q < 7; ++q) t[d].cyc[q] = (uint8_t)ring_cyc(e, q);
  }
  cudaError_t e = cudaMemcpyToSymbol(c_dir, t, sizeof(t));
  // the copy may still be landing on the legacy stream, which library streams do not wait for
  if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);
  return (int)e;
}

}  // namespace
}  // namespace hhg
