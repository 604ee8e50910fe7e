// Rows of nodes on the macro skeleton (faces, edges and vertices of the macro mesh, Sec. 2.2 of
// arXiv 1908.08666): device code of the skeleton part of a sweep, run by k_rows alone and by k_sweep
// in blocks between those of the macro interiors.
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
// Nodes in the interior of a macro face have one or two incidences, and what depends on the direction
// is fixed by the face's type: face_incidence, unrolled over the directions, one lane per node and
// side, all lanes of a warp on the same face.  Nodes on macro edges and vertices: incidence, a short
// loop over the directions with run-time ring indices (unrolled it would be tens of KB, and a small
// launch spends its time fetching instructions); the incidences of a node lie in lanes of one warp a
// power of two apart and are summed by a butterfly.
#pragma once
#include <cuda_runtime.h>

#include "hhg_internal.h"
#include "hhg_launch.h"
#include "hhg_row.cuh"

namespace hhg {

namespace {

constexpr int ROWS_BLOCK = 128;
constexpr int ROWS_WARPS = ROWS_BLOCK / 32;
constexpr int DIR_PER_THREAD = 4;  // Dirichlet entries a thread copies, their loads in flight together

// per direction d: ring pairs (ring_a, ring_b), then the ring in cyclic order, closed
struct alignas(16) DirTable {
  uint8_t ring[3][2];
  uint8_t cyc[7];
  uint8_t pad[3];
};
__constant__ DirTable c_dir[NDIR];  // one copy per translation unit, filled by upload_direction_tables

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

// the scaled block of a direction from its ring's coefficients (pairs ka[c], kb[c])
template <typename T, bool DIAG>
__device__ __forceinline__ void scaled_term(const T (&v)[16], bool red, T k0, T kd, const T (&ka)[3], const T (&kb)[3],
                                            const OpFlags& fl, const EdgeDiff<T>& D, RowSum<T>& s) {
  T rs = 0, wx = 0, wy = 0, wz = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (c == 2 && !red) break;
    rs += ka[c] + kb[c];
    const T dk = ka[c] - kb[c];
    wx = fma(dk, v[6 + 3 * c], wx);
    wy = fma(dk, v[7 + 3 * c], wy);
    wz = fma(dk, v[8 + 3 * c], wz);
  }
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

// Scratch of the lane-per-incidence rows: neighbour entries and coefficients, a column per thread.
template <typename T>
struct RowScratch {
  T k[NDIR][ROWS_BLOCK];
  int at[NDIR][ROWS_BLOCK];
};

// One macro's part of the row of the point of `it`.
template <typename T, bool DIAG, int STK>
__device__ __forceinline__ void incidence(const LevelDev& L, const MacroConsts<T>* __restrict__ mc, const OpFlags& fl,
                                          const SweepArgs<T>& a, const RowLane& it, RowScratch<T>& sh, RowSum<T>& s) {
  const int tid = threadIdx.x;
  const int n = L.n;
  const int64_t E = L.entries;
  const int64_t base = (int64_t)it.macro * L.nt;
  const T* __restrict__ px = a.x + base;
  const T* __restrict__ pk = a.k + base;
  const int i = it.i, j = it.j, k = it.k, l = n - i - j - k;
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
  const bool vel = !STK || !(it.flags & ROW_VDIR);
  // directions with the scaled block
  const uint32_t scaled = fl.practical ? 0u : interior;
  const MacroConsts<T>& C = mc[it.macro];
  // elements whose constants are in flight at a time
  constexpr int UE = sizeof(T) == 4 ? 3 : 2;
  // the neighbour's values are requested one direction ahead
  T xn, yn, zn, pn = 0;
  auto fetch = [&](int d) {
    const T* q = px + sh.at[d][tid];
    xn = q[0];
    yn = q[E];
    zn = q[2 * E];
    if (STK) pn = q[3 * E];
  };
  fetch(0);
#pragma unroll 1
  for (int d = 0; d < NDIR; ++d) {
    EdgeDiff<T> D{xn - x0, yn - y0, zn - z0, pn - p0, STK ? fma((T)(1.0 / 3.0), p0, pn) : (T)0};
    if (d + 1 < NDIR) fetch(d + 1);
    if (!((inside >> d) & 1u)) continue;
    const DirTable t = c_dir[d];
    const int e7 = d < 7 ? d : d - 7;
    const bool red = e7 < 3 || e7 == 6;
    const T kd = sh.k[d][tid];
    if ((scaled >> d) & 1u) {
      if (vel) {
        T v[16], ka[3], kb[3];
        load_values<T, 16>(&C.sc[d][0], v);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          ka[c] = sh.k[t.ring[c][0]][tid];
          kb[c] = sh.k[t.ring[c][1]][tid];
        }
        scaled_term<T, DIAG>(v, red, k0, kd, ka, kb, fl, D, s);
      }
      if (STK) {
        T v[8];
        load_values<T, 8>(&C.sb[d][0], v);
        stokes_term<T>(v, D, s);
      }
      continue;
    }
    const T ke = k0 + kd;
#pragma unroll
    for (int e0 = 0; e0 < 6; e0 += UE) {
      if (e0 >= 4 && !red) break;
      T v[UE][16], ks[UE];
#pragma unroll
      for (int e = 0; e < UE; ++e) {
        const int ra = t.cyc[e0 + e], rb = t.cyc[e0 + e + 1];
        const bool ok = (inside >> ra) & (inside >> rb) & (red || e0 + e < 4) & 1u;
        ks[e] = ke + (sh.k[ra][tid] + sh.k[rb][tid]);
#pragma unroll
        for (int q = 0; q < 16; ++q) v[e][q] = 0;
        if (ok) load_values<T, EL_COUNT<T, STK>>(&C.el[d][e0 + e][0], v[e]);
      }
#pragma unroll
      for (int e = 0; e < UE; ++e) element_term<T, DIAG, STK>(v[e], ks[e], vel, D, s);
    }
  }
}

// Which directions stay in the macro from a point inside its face F, and which can end at a
// macro-interior point: the representative point on a lattice with 16 intervals decides, at compile
// time.  Only next to the face's edges an inward direction may end on another face instead.
__device__ __forceinline__ constexpr int face_coord(int F, int c) {  // c: i, j, k
  return F == 0 ? (c == 2 ? 6 : 5) : F == c + 1 ? 0 : 5;
}
__device__ __forceinline__ bool face_dir_valid(int F, int d) {
  return lattice_inside(16, face_coord(F, 0) + dir_di(d), face_coord(F, 1) + dir_dj(d), face_coord(F, 2) + dir_dk(d));
}
__device__ __forceinline__ bool face_dir_inward(int F, int d) {
  return lattice_interior(16, face_coord(F, 0) + dir_di(d), face_coord(F, 1) + dir_dj(d), face_coord(F, 2) + dir_dk(d));
}

// One macro's part of the row of such a point: six directions in the face (a_h over the half of the
// edge's elements that lies in the macro), four inward ones (the scaled block where they end at a
// macro-interior point, else, and with the practical rule or nodal integration, a_h over all of the
// edge's elements).  All lanes read the same constants.  near: points next to the face's edges.
template <typename T, int F, bool DIAG, int STK>
__device__ __forceinline__ void face_incidence(const MacroConsts<T>& C, const T* __restrict__ px,
                                               const T* __restrict__ pk, int64_t E, int n, int i, int j, int k,
                                               const OpFlags& fl, bool vel, bool near, RowSum<T>& s) {
  int nb[NDIR];
  lattice_neighbours(n, i, j, k, nb);
  const int c0 = lattice_index32(n, i, j, k);
  T kv[NDIR], x[NDIR], y[NDIR], z[NDIR], p[STK ? NDIR : 1];
#pragma unroll
  for (int d = 0; d < NDIR; ++d) {
    kv[d] = 0;
    if (!face_dir_valid(F, d)) continue;
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
    if (!face_dir_valid(F, d)) continue;
    EdgeDiff<T> D{x[d] - x0, y[d] - y0, z[d] - z0, 0, 0};
    if (STK) {
      D.dp = p[STK ? d : 0] - p0;
      D.pg = fma((T)(1.0 / 3.0), p0, p[STK ? d : 0]);
    }
    if (face_dir_inward(F, d) && scaled &&
        (!near || lattice_interior(n, i + dir_di(d), j + dir_dj(d), k + dir_dk(d)))) {
      if (vel) {
        T v[16], ka[3], kb[3];
        load_values<T, 16>(&C.sc[d][0], v);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          ka[c] = c < ring_count(d) ? kv[ring_a(d, c)] : (T)0;
          kb[c] = c < ring_count(d) ? kv[ring_b(d, c)] : (T)0;
        }
        scaled_term<T, DIAG>(v, dir_red(d), k0, kv[d], ka, kb, fl, D, s);
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
      if (!face_dir_valid(F, ring_cyc(d, e)) || !face_dir_valid(F, ring_cyc(d, e + 1))) continue;
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

// A block of 32 face nodes, two warps: warp q evaluates them from the macro on side q, the sums are
// exchanged through shared memory (side 0 + side 1 in both warps) and each warp writes its own copies.
// All threads of the launch's block call this together (b < 0: nothing to do).
template <typename T, int OP, int STK>
__device__ __forceinline__ double face_block(const LevelDev& L, const MacroConsts<T>* __restrict__ mc,
                                             const OpFlags& fl, const SweepArgs<T>& a, int b, T* share) {
  constexpr bool DIAG = OP == OP_JACOBI || OP == OP_CHEBY || OP == OP_DIAG;
  const int lane = threadIdx.x & 31, side = (threadIdx.x >> 5) & 1;
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
    switch (side == 0 ? B.face[0] : B.face[1]) {
      case 0: face_incidence<T, 0, DIAG, STK>(mc[m], px, pk, E, L.n, P.i, P.j, P.k, fl, vel, near, s); break;
      case 1: face_incidence<T, 1, DIAG, STK>(mc[m], px, pk, E, L.n, P.i, P.j, P.k, fl, vel, near, s); break;
      case 2: face_incidence<T, 2, DIAG, STK>(mc[m], px, pk, E, L.n, P.i, P.j, P.k, fl, vel, near, s); break;
      default: face_incidence<T, 3, DIAG, STK>(mc[m], px, pk, E, L.n, P.i, P.j, P.k, fl, vel, near, s); break;
    }
  }
  double r2 = 0.0;
  T* own = share + threadIdx.x;
  const T* oth = share + (threadIdx.x ^ 32);
  own[0] = s.ax;
  own[ROWS_BLOCK] = s.ay;
  own[2 * ROWS_BLOCK] = s.az;
  own[3 * ROWS_BLOCK] = STK ? s.yp : s.dgx;
  own[4 * ROWS_BLOCK] = s.dgy;
  own[5 * ROWS_BLOCK] = s.dgz;
  __syncthreads();
  s.ax += oth[0];
  s.ay += oth[ROWS_BLOCK];
  s.az += oth[2 * ROWS_BLOCK];
  if (STK) s.yp += oth[3 * ROWS_BLOCK];
  if (DIAG) {
    s.dgx += oth[3 * ROWS_BLOCK];
    s.dgy += oth[4 * ROWS_BLOCK];
    s.dgz += oth[5 * ROWS_BLOCK];
  }
  if (valid) {
    double tmp = 0.0;
    write_row<T, OP, STK>(a, (int64_t)m * L.nt + lattice_index32(L.n, P.i, P.j, P.k), L.entries, s, STK && B.vdir, tmp);
    if (side == 0) r2 = tmp;
  }
  return r2;
}

// Blocks of the skeleton part of a sweep, in this order: warps of row_lanes (ROWS_WARPS a block; a
// node with more than 32 incidences takes several rounds of its warp), face blocks (two a block),
// Dirichlet entries (identity rows, every copy; not in the Stokes lists).
template <int STK>
struct RowBlocks {
  const RowLane* lanes;
  const int32_t* warps;
  int nwarps, nfaces, row_blocks, face_blocks, total;
  __host__ __device__ explicit RowBlocks(const LevelDev& L)
      : lanes(STK ? L.row_lanes_stk : L.row_lanes),
        warps(STK ? L.row_warps_stk : L.row_warps),
        nwarps(STK ? L.nrow_stk : L.nrow_skel),
        nfaces(L.nface_blocks[STK]),
        row_blocks((nwarps + ROWS_WARPS - 1) / ROWS_WARPS),
        face_blocks((nfaces + ROWS_WARPS / 2 - 1) / (ROWS_WARPS / 2)),
        total(row_blocks + face_blocks + (STK ? 0 : (int)((L.ndir_entries + ROWS_BLOCK * DIR_PER_THREAD - 1) / (ROWS_BLOCK * DIR_PER_THREAD)))) {}
  // blocks that hold rows with a residual
  __host__ __device__ int partials() const { return row_blocks + face_blocks; }
};

// Block b of them; its partial sum of |r|^2 goes to partial[b].
template <typename T, int OP, int STK>
__device__ __forceinline__ void rows_block(const LevelDev& L, const MacroConsts<T>* __restrict__ mc, const OpFlags& fl,
                                           const SweepArgs<T>& a, int b, RowScratch<T>& sh, double* partial) {
  constexpr bool DIAG = OP == OP_JACOBI || OP == OP_CHEBY || OP == OP_DIAG;
  const RowBlocks<STK> R(L);
  const int64_t E = L.entries;
  if (b >= R.row_blocks + R.face_blocks) {
    if (STK) return;
    const int64_t t = (int64_t)(b - R.row_blocks - R.face_blocks) * ROWS_BLOCK * DIR_PER_THREAD + threadIdx.x;
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
  double r2 = 0.0;
  if (b >= R.row_blocks) {
    const int f = (b - R.row_blocks) * (ROWS_WARPS / 2) + (threadIdx.x >> 6);
    r2 = face_block<T, OP, STK>(L, mc, fl, a, f < R.nfaces ? f : -1, &sh.k[0][0]);
  } else if (const int w = b * ROWS_WARPS + (threadIdx.x >> 5); w < R.nwarps) {
    const RowLane* row = R.lanes + (int64_t)R.warps[w] * 32 + (threadIdx.x & 31);
    const int rounds = row->flags >> ROW_ROUNDS_SHIFT, lg = row->flags & ROW_LG;  // the same in the whole warp
    RowSum<T> s;
#pragma unroll 1
    for (int r = 0; r < rounds; ++r) {
      const RowLane it = row[32 * r];
      if (it.macro >= 0) incidence<T, DIAG, STK>(L, mc, fl, a, it, sh, s);
    }
#pragma unroll 1
    for (int o = 32 >> lg; o < 32; o <<= 1) {
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
#pragma unroll 1
    for (int r = 0; r < rounds; ++r) {
      const RowLane it = row[32 * r];
      if (it.macro < 0) continue;
      double tmp = 0.0;
      write_row<T, OP, STK>(a, (int64_t)it.macro * L.nt + lattice_index32(L.n, it.i, it.j, it.k), E, s,
                            it.flags & ROW_VDIR, tmp);
      if (it.flags & ROW_FIRST) r2 = tmp;
    }
  }
  if (OP == OP_RESID && partial != nullptr) block_sum_store<T>(r2, partial + b);
}

// fills this translation unit's ring tables used with run-time direction indices
inline int upload_tables() {
  DirTable t[NDIR] = {};
  for (int d = 0; d < NDIR; ++d) {
    for (int c = 0; c < 3; ++c) {
      t[d].ring[c][0] = (uint8_t)(c < ring_count(d) ? ring_a(d, c) : 0);
      t[d].ring[c][1] = (uint8_t)(c < ring_count(d) ? ring_b(d, c) : 0);
    }
    for (int q = 0; q < 7; ++q) t[d].cyc[q] = (uint8_t)ring_cyc(d, q);
  }
  cudaError_t e = cudaMemcpyToSymbol(c_dir, t, sizeof(t));
  // the copy may still be landing on the legacy stream, which library streams do not wait for
  if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);
  return (int)e;
}

}  // namespace
}  // namespace hhg
