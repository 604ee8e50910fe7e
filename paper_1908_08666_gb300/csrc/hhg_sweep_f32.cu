// Sweeps of the scaled-stencil variants in one launch, FP32.
#include "hhg_march.cuh"

namespace hhg {

int upload_tables_f32() { return upload_tables(); }

template <typename T>
int launch_sweep(const LevelDev& L, const MacroConsts<T>* mc, OpKind op, const OpFlags& fl, const SweepArgs<T>& a,
                 void* stream, int64_t* partial_count) {
  cudaStream_t s = (cudaStream_t)stream;
  switch (op) {
    case OP_APPLY: return launch<T, OP_APPLY, 0>(L, mc, fl, a, s, partial_count);
    case OP_RESID: return launch<T, OP_RESID, 0>(L, mc, fl, a, s, partial_count);
    case OP_JACOBI: return launch<T, OP_JACOBI, 0>(L, mc, fl, a, s, partial_count);
    case OP_CHEBY: return launch<T, OP_CHEBY, 0>(L, mc, fl, a, s, partial_count);
    case OP_DIAG: return launch<T, OP_DIAG, 0>(L, mc, fl, a, s, partial_count);
  }
  return (int)cudaErrorInvalidValue;
}
template int launch_sweep<float>(const LevelDev&, const MacroConsts<float>*, OpKind, const OpFlags&, const SweepArgs<float>&, void*,
                                 int64_t*);

}  // namespace hhg
