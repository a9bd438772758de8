// The residual's kernels as the dispatch sees them: on axis-aligned elements
// (dg_affine.cuh), one instance per (dim, P, Q), compiled in dg_affine_*.cu, and
// on general ones (dg_general.cuh).
#pragma once
#include "dg_internal.h"
#include "dg_sumfact.cuh"

// (dim, P, Q) instances built into the library, in groups of one translation
// unit's work
#define DG_INSTANCES_2D(X) \
  X(2, 1, 3) X(2, 2, 3) X(2, 2, 4) X(2, 3, 5) X(2, 4, 6) X(2, 5, 7) X(2, 6, 8)
#define DG_INSTANCES_3A(X) X(3, 1, 3) X(3, 2, 4) X(3, 2, 5) X(3, 3, 5)
#define DG_INSTANCES_3B(X) X(3, 3, 6) X(3, 4, 6)
#define DG_INSTANCES_3C(X) X(3, 4, 8)
#define DG_INSTANCES(X) DG_INSTANCES_2D(X) DG_INSTANCES_3A(X) DG_INSTANCES_3B(X) DG_INSTANCES_3C(X)

namespace dg {

// Layout and shared memory of the axis-aligned kernels
template <int DIM, int P, int Q>
struct Aff {
  using C = Cfg<DIM, P, Q>;
  static constexpr int N = P + 1, NV = DIM + 2, NM = C::NM, NQ = C::NQ, NF = C::NF;
  // rows along direction 0 padded to an odd length: lines along it start in
  // different shared-memory banks
  static constexpr int RQ = Q | 1;
  static constexpr int Q2 = DIM == 3 ? Q : 1, N2 = DIM == 3 ? N : 1;
  static constexpr int VP = RQ * Q * Q2;      // padded volume array of one variable
  static constexpr int LQ = NF;               // lines of one direction on the Gauss grid
  // volume kernel, per element: DIM + 1 arrays
  static constexpr int VOL_EL = (DIM + 1) * NV * VP;
  // face kernel, per face: two regions used in turn
  static constexpr int NT = DIM == 3 ? N * N : N;   // coefficients of a face
  static constexpr int KK = DIM + 2;                // trace fields: both values, d_n, d_t
  static constexpr int imax(int a, int b) { return a > b ? a : b; }
  static constexpr int FX = imax(2 * NV * NM, DIM == 3 ? 4 * NV * N * RQ : KK * NV * NF);
  static constexpr int FY = imax(4 * NV * NT, DIM == 3 ? KK * NV * NF : 0);
  // shared memory in bytes of `e` elements / `f` faces per block
  static constexpr size_t vol_bytes(int e) {
    return (size_t)e * (8 * VOL_EL + 2 * DIM * 32 + 4 * NV * 4);
  }
  static constexpr size_t face_bytes(int f) { return (size_t)f * (8 * (FX + FY) + 128 + 6 * NV * 4); }
};

// and of those on general elements
template <int DIM, int P, int Q>
struct Gen : Aff<DIM, P, Q> {
  using A = Aff<DIM, P, Q>;
  static constexpr int NFLD = 2 + 2 * DIM;  // trace fields: both values, both sides' derivatives
  static constexpr int GX = A::imax(2 * A::NV * A::NM, DIM == 3 ? 6 * A::NV * A::N * A::RQ
                                                                : NFLD * A::NV * A::NF);
  static constexpr int GY = A::imax(4 * A::NV * A::NT, DIM == 3 ? NFLD * A::NV * A::NF : 0);
  static constexpr size_t vol_bytes(int e) {
    return (size_t)e * (8 * A::VOL_EL + 2 * DIM * 4 + (5 * A::NV + 1) * 4 + 16) + 4 * A::NM;
  }
  static constexpr size_t face_bytes(int f) {
    return (size_t)f * (8 * (GX + GY) + 64 + (2 + 1 + 1 + 4) * A::NV * 4 + 16);
  }
};

// shared memory of a block; every launch shape the tuning admits stays below
constexpr size_t FIX_SMEM = 227 * 1024;

template <int DIM, int P, int Q>
dg_status launch_fix(dg_mesh_s* m, const EvalArgs& a, cudaStream_t s);
// general elements (dg_general.cuh; the instances of DG_CURVED_INSTANCES)
template <int DIM, int P, int Q>
dg_status launch_gen(dg_mesh_s* m, const EvalArgs& a, cudaStream_t s);
template <int DIM, int P, int Q>
dg_status launch_minv_exp(dg_mesh_s* m, cudaStream_t s);

}  // namespace dg
