// Skeleton rows in a launch of their own, FP32.
#include "hhg_rows_launch.cuh"

namespace hhg {

template int launch_rows<float>(const LevelDev&, const MacroConsts<float>*, OpKind, const OpFlags&, const SweepArgs<float>&,
                                void*, int64_t, int64_t*);
template int launch_rows_stokes<float>(const LevelDev&, const MacroConsts<float>*, OpKind, const OpFlags&,
                                       const SweepArgs<float>&, void*, int64_t, int64_t*);

int upload_direction_tables() {
  int e = upload_tables();
  if (e == 0) e = upload_tables_rows_f64();
  if (e == 0) e = upload_tables_f32();
  if (e == 0) e = upload_tables_f64();
  if (e == 0) e = upload_tables_stokes_f32();
  if (e == 0) e = upload_tables_stokes_f64();
  return e;
}

}  // namespace hhg
