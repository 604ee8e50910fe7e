// Skeleton rows in a launch of their own, FP64.
#include "hhg_rows_launch.cuh"

namespace hhg {

template int launch_rows<double>(const LevelDev&, const MacroConsts<double>*, OpKind, const OpFlags&, const SweepArgs<double>&,
                                void*, int64_t, int64_t*);
template int launch_rows_stokes<double>(const LevelDev&, const MacroConsts<double>*, OpKind, const OpFlags&,
                                       const SweepArgs<double>&, void*, int64_t, int64_t*);

int upload_tables_rows_f64() { return upload_tables(); }

}  // namespace hhg
