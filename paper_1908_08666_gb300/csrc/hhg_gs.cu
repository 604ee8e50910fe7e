// Gauss-Seidel passes of the hybrid smoother over the macro interiors (Sec. 5 of arXiv 1908.08666):
// eight colours by the parities of (i, j, k), in place, every point with its neighbours' newest values.
//
// What bounds them: FP64 (the smoother's precision in the paper's solver), about 560 FP64 instructions
// per point at 2 lanes per SM and clock, and on coarse levels the latency of one row's chain.
//   - k_gs_colour: a launch per colour, one thread per point.  Points come from a list per colour, so
//     every lane has one (a chunk of a lattice row per warp left 17 of 32 lanes busy on 129^3 nodes,
//     8 on macros of 32 intervals); blocks of two warps, so that a pass spreads evenly over the SMs.
//   - k_gs_macro: all colours in one launch.  During the passes the skeleton is fixed, so the macros
//     do not depend on each other: a cluster of blocks takes one macro and meets at a barrier after
//     every colour.  Eight lanes share a point, one direction pair each, so that a row's chain is a
//     seventh as long; 95 instead of 70 FP64 instructions per four points, so it serves the levels
//     where latency and launches count.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "hhg_internal.h"
#include "hhg_launch.h"

namespace hhg {

namespace {

constexpr int GS_BLOCK = 64;
constexpr int GSM_BLOCK = 256;
constexpr int GS_C = 12;  // constants per direction pair (MacroConsts::mar): S, s_0, s_2

// khat and w of an edge from its end points' coefficients and its ring's (pairs ka[q], kb[q] in cyclic
// order; see hhg_march.cuh for the dependency of a six-element edge's three axial vectors)
template <typename T, int GEN>
__device__ __forceinline__ void edge_block(bool red, T k0, T kd, const T (&ka)[3], const T (&kb)[3], const T (&c)[GS_C],
                                           const OpFlags& fl, T& kh, T& wx, T& wy, T& wz) {
  const bool physical = GEN ? fl.physical != 0 : true;
  const bool khat_edge = GEN ? fl.khat_edge != 0 : false;
  T rs = (ka[0] + kb[0]) + (ka[1] + kb[1]);
  const T e0 = ka[0] - kb[0], e1 = ka[1] - kb[1];
  T f0 = e0, f1 = e1;
  if (red) {
    rs += ka[2] + kb[2];
    f0 = e0 + e1;
    f1 = (ka[2] - kb[2]) + e1;
  }
  if (khat_edge)
    kh = (T)0.5 * (k0 + kd);
  else
    kh = fma(red ? (T)(1.0 / 12.0) : (T)0.125, rs, fma((T)0.25, kd, (T)0.25 * k0));
  if (physical) {
    wx = fma(f1, c[9], f0 * c[6]);
    wy = fma(f1, c[10], f0 * c[7]);
    wz = fma(f1, c[11], f0 * c[8]);
  } else {
    wx = wy = wz = 0;
  }
}

template <typename T>
struct GsSum {
  T ax = 0, ay = 0, az = 0, dgx = 0, dgy = 0, dgz = 0;
};

// A direction pair's part of the row: differences p (d) and m (-d) to the point
template <typename T, int GEN>
__device__ __forceinline__ void pair_part(bool red, T k0, T kp, T km, const T (&pa)[3], const T (&pb)[3],
                                          const T (&ma)[3], const T (&mb)[3], const T (&p)[3], const T (&m)[3],
                                          const T (&c)[GS_C], const OpFlags& fl, GsSum<T>& s) {
  T khp, khm, wx, wy, wz;
  edge_block<T, GEN>(red, k0, kp, pa, pb, c, fl, khp, wx, wy, wz);
  s.ax = fma(wy, p[2], fma(-wz, p[1], s.ax));
  s.ay = fma(wz, p[0], fma(-wx, p[2], s.ay));
  s.az = fma(wx, p[1], fma(-wy, p[0], s.az));
  edge_block<T, GEN>(red, k0, km, ma, mb, c, fl, khm, wx, wy, wz);
  s.ax = fma(wy, m[2], fma(-wz, m[1], s.ax));
  s.ay = fma(wz, m[0], fma(-wx, m[2], s.ay));
  s.az = fma(wx, m[1], fma(-wy, m[0], s.az));
  const T vx = fma(khp, p[0], khm * m[0]), vy = fma(khp, p[1], khm * m[1]), vz = fma(khp, p[2], khm * m[2]);
  s.ax = fma(c[0], vx, fma(c[3], vy, fma(c[4], vz, s.ax)));
  s.ay = fma(c[3], vx, fma(c[1], vy, fma(c[5], vz, s.ay)));
  s.az = fma(c[4], vx, fma(c[5], vy, fma(c[2], vz, s.az)));
  const T ks = khp + khm;
  s.dgx = fma(-ks, c[0], s.dgx);
  s.dgy = fma(-ks, c[1], s.dgy);
  s.dgz = fma(-ks, c[2], s.dgz);
}

template <typename T>
__device__ __forceinline__ void load_constants(const T* __restrict__ p, T (&c)[GS_C]) {
#pragma unroll
  for (int q = 0; q < GS_C; ++q) c[q] = p[q];
}

// One colour: the points packed (k << 20) | (j << 10) | i of the list at `points`; grid: blocks x
// macros macro0 ...
template <typename T, int GEN>
__global__ void __launch_bounds__(GS_BLOCK) k_gs_colour(const LevelDev L, const MacroConsts<T>* __restrict__ mc,
                                                        const int macro0, const OpFlags fl, const T* __restrict__ f,
                                                        const T* __restrict__ kc, T* x,
                                                        const int32_t* __restrict__ points, const int count) {
  __shared__ T cst[7 * GS_C];
  const int macro = macro0 + blockIdx.y;
  for (int q = threadIdx.x; q < 7 * GS_C; q += GS_BLOCK) cst[q] = __ldg(&mc[macro].mar[q / GS_C][q % GS_C]);
  __syncthreads();
  const int t = blockIdx.x * GS_BLOCK + threadIdx.x;
  if (t >= count) return;
  const int32_t pt = points[t];
  const int i = pt & 0x3FF, j = (pt >> 10) & 0x3FF, k = pt >> 20;
  const int64_t E = L.entries;
  const int64_t base = (int64_t)macro * L.nt;
  int nb[NDIR];
  lattice_neighbours(L.n, i, j, k, nb);
  const int c0 = nb[0] - 1;
  // neighbours are points of other colours: nothing that this launch writes is read through here
  const T* __restrict__ X = x + base;
  const T* __restrict__ K = kc + base;
  T kk[NDIR], d[NDIR][3];
  const T k0 = __ldg(K + c0);
  const T o[3] = {X[c0], X[c0 + E], X[c0 + 2 * E]};
#pragma unroll
  for (int q = 0; q < NDIR; ++q) {
    kk[q] = __ldg(K + nb[q]);
#pragma unroll
    for (int r = 0; r < 3; ++r) d[q][r] = __ldg(X + nb[q] + r * E) - o[r];
  }
  GsSum<T> s;
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    T c[GS_C], pa[3], pb[3], ma[3], mb[3];
    load_constants(cst + q * GS_C, c);
    const int nr = dir_red(q) ? 3 : 2;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int ra = ring_cyc(q, r < nr ? r : 0), rb = ring_cyc(q, r < nr ? r + nr : 0);
      pa[r] = kk[ra];
      pb[r] = kk[rb];
      ma[r] = kk[dir_neg(ra)];
      mb[r] = kk[dir_neg(rb)];
    }
    pair_part<T, GEN>(dir_red(q), k0, kk[q], kk[q + 7], pa, pb, ma, mb, d[q], d[q + 7], c, fl, s);
  }
  const int64_t e = base + c0;
  x[e] = o[0] + (__ldg(f + e) - s.ax) / s.dgx;
  x[e + E] = o[1] + (__ldg(f + e + E) - s.ay) / s.dgy;
  x[e + 2 * E] = o[2] + (__ldg(f + e + 2 * E) - s.az) / s.dgz;
}

// lattice offsets (i, j, k) of a direction and of its ring's first half, in cyclic order
struct GsPair {
  int8_t d[3], ra[3][3], rb[3][3];
  int8_t red;
};
__constant__ GsPair c_pair[8];

// All colours of one macro per cluster (grid: clusters x macros macro0 ..); lane group of 8: direction
// pairs 0 .. 6 of one point.
template <typename T, int GEN>
__global__ void __launch_bounds__(GSM_BLOCK) k_gs_macro(const LevelDev L, const MacroConsts<T>* __restrict__ mc,
                                                        const int macro0, const OpFlags fl, const T* __restrict__ f,
                                                        const T* __restrict__ kc, T* x) {
  namespace cg = cooperative_groups;
  const cg::cluster_group cluster = cg::this_cluster();
  const int parts = gridDim.x;  // blocks of the cluster
  const int macro = macro0 + blockIdx.y;
  const int pair = threadIdx.x & 7;
  const GsPair D = c_pair[pair];
  const bool red = D.red;
  T c[GS_C];
#pragma unroll
  for (int q = 0; q < GS_C; ++q) c[q] = pair < 7 ? __ldg(&mc[macro].mar[pair][q]) : (T)0;
  const int64_t E = L.entries;
  const int64_t base = (int64_t)macro * L.nt;
  T* X = x + base;
  const T* __restrict__ K = kc + base;
  const int n = L.n;
  for (int col = 0; col < 8; ++col) {
    const int first = L.gs_ptr[col], count = L.gs_ptr[col + 1] - first;
    if (count == 0) continue;
    const int stride = parts * (GSM_BLOCK / 8);
    // whole warps go round together (the shuffles below): lanes past the end take the last point
    for (int t0 = blockIdx.x * (GSM_BLOCK / 8) + (threadIdx.x >> 5) * 4; t0 < count; t0 += stride) {
      const int t = t0 + ((threadIdx.x & 31) >> 3);
      const bool valid = t < count;
      const int32_t pt = L.gs_points[first + min(t, count - 1)];
      const int i = pt & 0x3FF, j = (pt >> 10) & 0x3FF, k = pt >> 20;
      const int c0 = lattice_index32(n, i, j, k);
      auto at = [&](const int8_t (&o)[3], int sign) {
        return lattice_index32(n, i + sign * o[0], j + sign * o[1], k + sign * o[2]);
      };
      const int ip = at(D.d, 1), im = at(D.d, -1);
      const T k0 = __ldg(K + c0), kp = __ldg(K + ip), km = __ldg(K + im);
      T o[3], p[3], m[3], pa[3], pb[3], ma[3], mb[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        // other blocks of the cluster write x: past the L1 cache
        o[r] = __ldcg(X + c0 + r * E);
        p[r] = __ldcg(X + ip + r * E) - o[r];
        m[r] = __ldcg(X + im + r * E) - o[r];
        pa[r] = __ldg(K + at(D.ra[r], 1));
        pb[r] = __ldg(K + at(D.rb[r], 1));
        ma[r] = __ldg(K + at(D.ra[r], -1));
        mb[r] = __ldg(K + at(D.rb[r], -1));
      }
      const int comp = pair < 3 ? pair : 0;
      const T fv = __ldg(f + base + c0 + comp * E);
      GsSum<T> s;
      pair_part<T, GEN>(red, k0, kp, km, pa, pb, ma, mb, p, m, c, fl, s);
      if (pair == 7) s = GsSum<T>();
      // sum over the 8 lanes, one of the six sums per lane: halve the sums held three times
      T v[8] = {s.ax, s.ay, s.az, 0, s.dgx, s.dgy, s.dgz, 0};
#pragma unroll
      for (int h = 4; h >= 1; h >>= 1) {
        const bool up = pair & h;
#pragma unroll
        for (int q = 0; q < h; ++q) {
          const T send = up ? v[q] : v[q + h], keep = up ? v[q + h] : v[q];
          v[q] = keep + __shfl_xor_sync(0xffffffffu, send, h);
        }
      }
      // lane q holds the sum of index q: 0..2 the row, 4..6 the diagonal
      const T dg = __shfl_xor_sync(0xffffffffu, v[0], 4);
      if (valid && pair < 3) X[c0 + comp * E] = (comp == 0 ? o[0] : comp == 1 ? o[1] : o[2]) + (fv - v[0]) / dg;
    }
    if (parts > 1) {
      __threadfence();
      cluster.sync();
    } else {
      __syncthreads();
    }
  }
}

constexpr int GS_MAX_MACROS = 65535;  // grid.y

// Which form.  k_gs_macro takes parts * GSM_BLOCK / 8 points of a macro at a time, in rounds that follow one
// another, so it takes the levels whose colours fit a few rounds, and of those the ones that do not fill
// the chip (95 against 70 FP64 instructions per four points).  A smoothing step (skeleton rows and 8 colours)
// in FP64 / FP32, us, in one launch and in eight:
//   rounds  macros x intervals per edge        one launch    eight launches
//   1       48 x 8 (10 points a colour)        74 / 27       204 / 62
//   2       48 x 16 (84)                       124 / 39      216 / 64
//   3       6 x 32 (680)                       207 / 59      199 / 62
//   3       96 x 16 (84)                       193 / 45      251 / 66
//   6       24 x 32 (680)                      345 / 86      236 / 63
//   22      1 x 64 (5456)                      1125 / 251    175 / 60
constexpr int GS_MACRO_MAX_ROUNDS = 3;
constexpr int64_t GS_MACRO_MAX_POINTS = 12000;

}  // namespace

// Tables of k_gs_macro: pairs beyond a four-element edge's two ring pairs and pair 7 point at the
// centre's own first ring node (loaded, not used).
int upload_gs_tables() {
  GsPair t[8] = {};
  for (int d = 0; d < 7; ++d) {
    t[d].d[0] = (int8_t)dir_di(d);
    t[d].d[1] = (int8_t)dir_dj(d);
    t[d].d[2] = (int8_t)dir_dk(d);
    t[d].red = dir_red(d);
    const int nr = dir_red(d) ? 3 : 2;
    for (int r = 0; r < 3; ++r) {
      const int ra = ring_cyc(d, r < nr ? r : 0), rb = ring_cyc(d, r < nr ? r + nr : 0);
      t[d].ra[r][0] = (int8_t)dir_di(ra);
      t[d].ra[r][1] = (int8_t)dir_dj(ra);
      t[d].ra[r][2] = (int8_t)dir_dk(ra);
      t[d].rb[r][0] = (int8_t)dir_di(rb);
      t[d].rb[r][1] = (int8_t)dir_dj(rb);
      t[d].rb[r][2] = (int8_t)dir_dk(rb);
    }
  }
  t[7] = t[0];
  cudaError_t e = cudaMemcpyToSymbol(c_pair, t, sizeof(t));
  // the copy may still be landing on the legacy stream, which library streams do not wait for
  if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);
  return (int)e;
}

template <typename T>
int launch_gs(const LevelDev& L, const MacroConsts<T>* mc, const OpFlags& fl, const T* f, const T* k, T* x,
              void* stream) {
  const int total = L.gs_ptr[8];
  if (total == 0 || L.nmacro == 0) return 0;
  cudaStream_t s = (cudaStream_t)stream;
  const bool gen = !(fl.physical == 1 && fl.khat_edge == 0);
  int most = 0;
  for (int c = 0; c < 8; ++c) most = std::max(most, L.gs_ptr[c + 1] - L.gs_ptr[c]);
  for (int m0 = 0; m0 < L.nmacro; m0 += GS_MAX_MACROS) {
    const int nm = std::min(GS_MAX_MACROS, L.nmacro - m0);
    // blocks per macro: enough for the largest colour, no more than share the SMs, a power of two up
    // to 8 (three blocks per macro were slower than two: 118 against 73 us on 48 macros)
    int parts = 1;
    while (parts < 8 && parts * (GSM_BLOCK / 8) < most && 2 * parts * L.nmacro <= 152) parts *= 2;
    if (most <= GS_MACRO_MAX_ROUNDS * parts * (GSM_BLOCK / 8) && (int64_t)most * L.nmacro <= GS_MACRO_MAX_POINTS) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(parts, nm);
      cfg.blockDim = dim3(GSM_BLOCK);
      cfg.stream = s;
      cudaLaunchAttribute at = {};
      at.id = cudaLaunchAttributeClusterDimension;
      at.val.clusterDim.x = parts;
      at.val.clusterDim.y = 1;
      at.val.clusterDim.z = 1;
      cfg.attrs = &at;
      cfg.numAttrs = 1;
      const cudaError_t e = gen ? cudaLaunchKernelEx(&cfg, k_gs_macro<T, 1>, L, mc, m0, fl, f, k, x)
                                : cudaLaunchKernelEx(&cfg, k_gs_macro<T, 0>, L, mc, m0, fl, f, k, x);
      if (e != cudaSuccess) return (int)e;
      continue;
    }
    for (int c = 0; c < 8; ++c) {
      const int count = L.gs_ptr[c + 1] - L.gs_ptr[c];
      if (count == 0) continue;
      const dim3 g((count + GS_BLOCK - 1) / GS_BLOCK, nm);
      const int32_t* pts = L.gs_points + L.gs_ptr[c];
      if (gen)
        k_gs_colour<T, 1><<<g, GS_BLOCK, 0, s>>>(L, mc, m0, fl, f, k, x, pts, count);
      else
        k_gs_colour<T, 0><<<g, GS_BLOCK, 0, s>>>(L, mc, m0, fl, f, k, x, pts, count);
    }
  }
  return (int)cudaGetLastError();
}
template int launch_gs<float>(const LevelDev&, const MacroConsts<float>*, const OpFlags&, const float*, const float*,
                              float*, void*);
template int launch_gs<double>(const LevelDev&, const MacroConsts<double>*, const OpFlags&, const double*,
                               const double*, double*, void*);

}  // namespace hhg
