// The skeleton part of a sweep as a launch of its own (k_rows): beside the interior kernels of the
// nodal-integration and stored-stencil variants and of hhg_set_interior_kernel, and in the hybrid
// Gauss-Seidel smoother.  The device code is in hhg_rows.cuh; a translation unit per precision, since they
// compile long.
#pragma once
#include "hhg_rows.cuh"

namespace hhg {

namespace {

template <typename T, int OP, int STK>
__global__ void __launch_bounds__(ROWS_BLOCK) k_rows(const LevelDev L, const MacroConsts<T>* __restrict__ mc,
                                                     const OpFlags fl, const SweepArgs<T> a) {
  __shared__ RowScratch<T> sh;
  rows_block<T, OP, STK>(L, mc, fl, a, blockIdx.x, sh, a.partial);
}

}  // namespace

template <typename T>
int launch_rows(const LevelDev& L, const MacroConsts<T>* mc, OpKind op, const OpFlags& fl, const SweepArgs<T>& a,
                void* stream, int64_t partial_offset, int64_t* partial_count) {
  cudaStream_t s = (cudaStream_t)stream;
  const RowBlocks<T, 0> R(L);
  if (partial_count) *partial_count = R.partials();
  if (R.total == 0) return 0;
  SweepArgs<T> am = a;
  if (a.partial) am.partial = a.partial + partial_offset;
  switch (op) {
    case OP_APPLY: k_rows<T, OP_APPLY, 0><<<R.total, ROWS_BLOCK, 0, s>>>(L, mc, fl, am); break;
    case OP_RESID: k_rows<T, OP_RESID, 0><<<R.total, ROWS_BLOCK, 0, s>>>(L, mc, fl, am); break;
    case OP_JACOBI: k_rows<T, OP_JACOBI, 0><<<R.total, ROWS_BLOCK, 0, s>>>(L, mc, fl, am); break;
    case OP_CHEBY: k_rows<T, OP_CHEBY, 0><<<R.total, ROWS_BLOCK, 0, s>>>(L, mc, fl, am); break;
    case OP_DIAG: k_rows<T, OP_DIAG, 0><<<R.total, ROWS_BLOCK, 0, s>>>(L, mc, fl, am); break;
  }
  return (int)cudaGetLastError();
}

template <typename T>
int launch_rows_stokes(const LevelDev& L, const MacroConsts<T>* mc, OpKind op, const OpFlags& fl,
                       const SweepArgs<T>& a, void* stream, int64_t partial_offset, int64_t* partial_count) {
  if (op != OP_APPLY && op != OP_RESID) return (int)cudaErrorInvalidValue;
  cudaStream_t s = (cudaStream_t)stream;
  const RowBlocks<T, 1> R(L);
  if (partial_count) *partial_count = R.partials();
  if (R.total == 0) return 0;
  SweepArgs<T> am = a;
  if (a.partial) am.partial = a.partial + partial_offset;
  if (op == OP_APPLY)
    k_rows<T, OP_APPLY, 1><<<R.total, ROWS_BLOCK, 0, s>>>(L, mc, fl, am);
  else
    k_rows<T, OP_RESID, 1><<<R.total, ROWS_BLOCK, 0, s>>>(L, mc, fl, am);
  return (int)cudaGetLastError();
}

}  // namespace hhg
