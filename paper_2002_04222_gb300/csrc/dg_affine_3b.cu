// Instances of the axis-aligned residual (DG_INSTANCES_3B).
#include "dg_affine.cuh"

namespace dg {
#define DG_INST(D_, P_, Q_) \
  template dg_status launch_fix<D_, P_, Q_>(dg_mesh_s*, const EvalArgs&, cudaStream_t);
DG_INSTANCES_3B(DG_INST)
#undef DG_INST
}  // namespace dg
