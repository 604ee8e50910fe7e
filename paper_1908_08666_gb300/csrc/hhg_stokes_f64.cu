// Sweeps of the Stokes saddle operator in one launch, FP64.
#include "hhg_march.cuh"

namespace hhg {

int upload_tables_stokes_f64() { return upload_tables(); }

template <typename T>
int launch_sweep_stokes(const LevelDev& L, const MacroConsts<T>* mc, OpKind op, const OpFlags& fl,
                        const SweepArgs<T>& a, void* stream, int64_t* partial_count) {
  if (op == OP_APPLY) return launch<T, OP_APPLY, 1>(L, mc, fl, a, (cudaStream_t)stream, partial_count);
  if (op == OP_RESID) return launch<T, OP_RESID, 1>(L, mc, fl, a, (cudaStream_t)stream, partial_count);
  return (int)cudaErrorInvalidValue;
}
template int launch_sweep_stokes<double>(const LevelDev&, const MacroConsts<double>*, OpKind, const OpFlags&,
                                        const SweepArgs<double>&, void*, int64_t*);

}  // namespace hhg
