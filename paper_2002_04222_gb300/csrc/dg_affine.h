// The residual on axis-aligned elements (kernels in dg_affine.cuh), one
// instance per (dim, P, Q), compiled in dg_affine_*.cu.
#pragma once
#include "dg_internal.h"

// (dim, P, Q) instances built into the library, in groups of one translation
// unit's work
#define DG_INSTANCES_2D(X) \
  X(2, 1, 3) X(2, 2, 3) X(2, 2, 4) X(2, 3, 5) X(2, 4, 6) X(2, 5, 7) X(2, 6, 8)
#define DG_INSTANCES_3A(X) X(3, 1, 3) X(3, 2, 4) X(3, 2, 5) X(3, 3, 5)
#define DG_INSTANCES_3B(X) X(3, 3, 6) X(3, 4, 6)
#define DG_INSTANCES_3C(X) X(3, 4, 8)
#define DG_INSTANCES(X) DG_INSTANCES_2D(X) DG_INSTANCES_3A(X) DG_INSTANCES_3B(X) DG_INSTANCES_3C(X)

namespace dg {

template <int DIM, int P, int Q>
dg_status launch_fix(dg_mesh_s* m, const EvalArgs& a, cudaStream_t s);
// general elements (dg_general.cuh; the instances of DG_CURVED_INSTANCES)
template <int DIM, int P, int Q>
dg_status launch_gen(dg_mesh_s* m, const EvalArgs& a, cudaStream_t s);
template <int DIM, int P, int Q>
dg_status launch_minv_exp(dg_mesh_s* m, cudaStream_t s);

}  // namespace dg
