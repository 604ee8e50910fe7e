// Sweeps of the Stokes saddle operator in one launch, FP32.
#include "hhg_march.cuh"

namespace hhg {

int upload_tables_stokes_f32() { return upload_tables(); }

template <typename T>
int launch_sweep_stokes(const LevelDev& L, const MacroConsts<T>* mc, OpKind op, const OpFlags& fl,
                        const SweepArgs<T>& a, void* stream, int64_t* partial_count) {
  if (op == OP_APPLY) return launch<T, OP_APPLY, 1>(L, mc, fl, a, (cudaStream_t)stream, partial_count);
  if (op == OP_RESID) return launch<T, OP_RESID, 1>(L, mc, fl, a, (cudaStream_t)stream, partial_count);
  return (int)cudaErrorInvalidValue;
}
template int launch_sweep_stokes<float>(const LevelDev&, const MacroConsts<float>*, OpKind, const OpFlags&,
                                        const SweepArgs<float>&, void*, int64_t*);

}  // namespace hhg
