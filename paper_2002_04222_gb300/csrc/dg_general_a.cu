// Instances of the residual on general elements.
#include "dg_general.cuh"

namespace dg {
#define DG_INST(D_, P_, Q_)                                                        \
  template dg_status launch_gen<D_, P_, Q_>(dg_mesh_s*, const EvalArgs&, cudaStream_t); \
  template dg_status launch_minv_exp<D_, P_, Q_>(dg_mesh_s*, cudaStream_t);
DG_INST(2, 2, 4) DG_INST(2, 3, 5) DG_INST(3, 1, 3) DG_INST(3, 2, 5)
#undef DG_INST
}  // namespace dg
