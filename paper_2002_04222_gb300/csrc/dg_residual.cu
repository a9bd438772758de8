// DG residual R(u) = M^-1 L(u, t) of Sec. 3.1 (Eq. matrix-form-equations): the
// dispatch over (dim, P, Q) and geometry, launch shapes and their autotuning,
// the shock sensor, the L2 projection, and the FP64 traces that the
// preconditioner build differentiates.  The residual's own kernels are two per
// geometry kind (axis-aligned: dg_affine.cuh; general: dg_general.cuh): faces
// (traces, Riemann, interior-penalty and symmetric fluxes) and volume
// (BwdTrans, derivatives, fluxes, the lift of both, M^-1, and for the
// Jacobian-free product the finite-difference combination).  Their
// contractions run in 64-bit fixed point on the integer pipe (dg_fix.cuh),
// FP64 is left with the pointwise fluxes.
#include <cstdio>
#include <vector>
#include "dg_internal.h"
#include "dg_physics.cuh"
#include "dg_sumfact.cuh"
#include "dg_affine.h"

namespace dg {

// ---------------------------------------------------------------- shock sensor
// Artificial-viscosity factor f_e = mu_0 S_e h_e / P of element e (Sec. 3.1.2),
// by one warp: the density's modified-basis coefficients (in A, overwritten;
// B is scratch of the same size) go to Legendre coefficients c by the 1-D
// transform along each direction; the reference-element L2 norms are then
// sums of c^2 times the Legendre norms, and the part removed by the
// projection onto degree <= P-1 per direction is the set of modes with some
// index equal to P.  Lane 0 writes avf[e].
template <int DIM, int P, int Q, bool CV>
__device__ void sensor_element(const SensorTab& st, const Phys& ph,
                               const ElemGeo* __restrict__ geo, const GenGeo& gg, int e,
                               double* A, double* B, int lane, double* __restrict__ avf) {
  using C = Cfg<DIM, P, Q>;
  constexpr int N = C::N, NM = C::NM, NQ = C::NQ;
  double* src = A;
  double* dst = B;
  int stride = 1;
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    for (int mm = lane; mm < NM; mm += 32) {
      const int id = (mm / stride) % N;
      const int m0 = mm - id * stride;
      double a = 0.0;
#pragma unroll
      for (int k = 0; k < N; ++k) a = fma(st.T[id * N + k], src[m0 + k * stride], a);
      dst[mm] = a;
    }
    __syncwarp();
    double* tmp = src;
    src = dst;
    dst = tmp;
    stride *= N;
  }
  double num = 0.0, den = 0.0, vol = 0.0;
  for (int mm = lane; mm < NM; mm += 32) {
    int r = mm;
    double wgt = 1.0;
    bool top = false;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const int id = r % N;
      r /= N;
      wgt *= st.nrm[id];
      top = top || id == P;
    }
    const double c2 = src[mm] * src[mm] * wgt;
    den += c2;
    if (top) num += c2;
  }
  if constexpr (CV) {
    const double* wj = gg.vgeo + (long long)e * (DIM * DIM + 1) * NQ + DIM * DIM * NQ;
    for (int q = lane; q < NQ; q += 32) vol += wj[q];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, o);
    den += __shfl_xor_sync(0xffffffffu, den, o);
    vol += __shfl_xor_sync(0xffffffffu, vol, o);
  }
  if (lane != 0) return;
  // below the ramp (the common case) no logarithm, sine or root is taken
  double S = 0.0;
  if (num > 0.0 && den > 0.0 && num >= st.lo * den) {
    if (num > st.hi * den) {
      S = 1.0;
    } else {
      const double se = log10(num / den), s0 = -4.0 * log10((double)P), kap = ph.av_kappa;
      S = 0.5 * (1.0 + sin(3.14159265358979323846 * (se - s0) / (2.0 * kap)));
    }
  }
  if (S == 0.0) {
    avf[e] = 0.0;
    return;
  }
  if constexpr (!CV) vol = geo[e].detJ * (double)(1 << DIM);
  const double h = DIM == 2 ? sqrt(vol) : cbrt(vol);
  avf[e] = ph.av_mu0 * S * h / (double)P;
}

// The factor of every element at u (dg_av_factor, and before the face kernel of
// a residual with shock capturing).  One warp per element.
constexpr int SENSOR_WARPS = 8;
template <int DIM, int P, int Q, bool CV>
__global__ void __launch_bounds__(32 * SENSOR_WARPS) sensor_kernel(
    const __grid_constant__ SensorTab st, const __grid_constant__ Phys ph,
    const ElemGeo* __restrict__ geo, const __grid_constant__ GenGeo gg, int E,
    const double* __restrict__ u, const double* __restrict__ v, const double* __restrict__ epsp,
    double* __restrict__ avf) {
  using C = Cfg<DIM, P, Q>;
  constexpr int NV = C::NV, NM = C::NM;
  __shared__ double sA[SENSOR_WARPS][NM], sC[SENSOR_WARPS][NM];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int e = blockIdx.x * SENSOR_WARPS + w;
  if (e >= E) return;  // warp-uniform; the kernel has no block-wide barrier
  const long long base = (long long)e * NV * NM;  // variable 0: density
  for (int k = lane; k < NM; k += 32) sA[w][k] = v ? fma(epsp[0], v[base + k], u[base + k]) : u[base + k];
  __syncwarp();
  sensor_element<DIM, P, Q, CV>(st, ph, geo, gg, e, sA[w], sC[w], lane, avf);
}

// ---------------------------------------------------------------- FP64 traces
// Traces of Q and grad Q on every element's faces, [E][2 DIM][(1+DIM) NV][NF]:
// sum-factorised BwdTrans, collocation derivatives on the Gauss grid and
// Lagrange extrapolation along the normal, all in FP64.
template <int DIM, int P, int Q, bool CV>
__global__ void __launch_bounds__(256) trace_kernel(const __grid_constant__ Tables tab,
                                                    const ElemGeo* __restrict__ geo,
                                                    const __grid_constant__ GenGeo gg, int E,
                                                    const double* __restrict__ u,
                                                    double* __restrict__ tbuf) {
  using C = Cfg<DIM, P, Q>;
  constexpr int N = C::N, NV = C::NV, NM = C::NM, NQ = C::NQ, NF = C::NF;
  constexpr int Q2 = C::Q2, N2 = C::N2, EPB = C::EPB;
  extern __shared__ double sm[];
  double* sB = sm;
  double* sD = sB + Q * N;
  double* sl = sD + Q * Q;  // lm, lp
  double* sU = sm + C::TAB;            // [EPB][NV][NM]
  double* sQ = sU + EPB * NV * NM;     // [EPB][NV][NQ]
  double* sG = sQ + EPB * NV * NQ;     // DIM arrays [EPB][NV][NQ]
  double* sT = sG + EPB * DIM * NV * NQ;  // 2-D only: scratch
  const int e0 = blockIdx.x * EPB;
  const int nrep = EPB * NV;

  stage_tables<DIM, P, Q>(tab, sm);
  for (int i = threadIdx.x; i < EPB * NV * NM; i += blockDim.x) {
    const int eb = i / (NV * NM);
    sU[i] = e0 + eb < E ? u[(long long)e0 * NV * NM + i] : 0.0;
  }
  __syncthreads();
  // BwdTrans: contract direction 0, 1 (, 2) with B
  if (DIM == 2) {
    contract<N, N, 1, 0, Q, N, 1, false>(sU, sT, sB, nrep);
    __syncthreads();
    contract<Q, N, 1, 1, Q, N, 1, false>(sT, sQ, sB, nrep);
  } else {
    double* t1 = sG + EPB * NV * NQ;       // reuse gradient slots 1 and 2
    double* t2 = sG + 2 * EPB * NV * NQ;
    contract<N, N, N2, 0, Q, N, 1, false>(sU, t1, sB, nrep);
    __syncthreads();
    contract<Q, N, N2, 1, Q, N, 1, false>(t1, t2, sB, nrep);
    __syncthreads();
    contract<Q, Q, N2, 2, Q, N, 1, false>(t2, sQ, sB, nrep);
  }
  __syncthreads();
  // reference derivatives on the Gauss grid (exact for the degree-P expansion)
  contract<Q, Q, Q2, 0, Q, Q, 1, false>(sQ, sG, sD, nrep);
  contract<Q, Q, Q2, 1, Q, Q, 1, false>(sQ, sG + EPB * NV * NQ, sD, nrep);
  if (DIM == 3) contract<Q, Q, Q2, 2, Q, Q, 1, false>(sQ, sG + 2 * EPB * NV * NQ, sD, nrep);
  __syncthreads();
  // face traces of Q and grad Q by Lagrange extrapolation along the normal
  constexpr int NTR = 2 * DIM * (1 + DIM) * NV * NF;
  if constexpr (CV) {
    // general element: extrapolate the value and the DIM reference
    // derivatives (polynomials along the line), then map the derivatives with
    // the metric of the face point
    constexpr int NTV = 2 * DIM * NV * NF;
    for (int idx = threadIdx.x; idx < EPB * NTV; idx += blockDim.x) {
      const int eb = idx / NTV;
      int rem = idx - eb * NTV;
      const int e = e0 + eb;
      if (e >= E) continue;
      const int p = rem % NF;
      rem /= NF;
      const int vv = rem % NV;
      const int lf = rem / NV;
      const int r = lf >> 1;
      const double* lw = sl + (lf & 1) * Q;
      int c[3] = {0, 0, 0};
      if (DIM == 2) {
        c[1 - r] = p;
      } else {
        const int t0 = r == 0 ? 1 : 0, t1 = r == 2 ? 1 : 2;
        c[t0] = p % Q;
        c[t1] = p / Q;
      }
      const int base = c[0] + Q * c[1] + Q * Q * c[2];
      const int str = r == 0 ? 1 : (r == 1 ? Q : Q * Q);
      double ext[1 + DIM];
#pragma unroll
      for (int fld = 0; fld <= DIM; ++fld) {
        const double* src = fld == 0 ? sQ + (eb * NV + vv) * NQ
                                     : sG + (((fld - 1) * EPB + eb) * NV + vv) * NQ;
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < Q; ++k) acc = fma(lw[k], src[base + k * str], acc);
        ext[fld] = acc;
      }
      const double* gp = gg.fgeo + ((long long)e * 2 * DIM + lf) * DIM * DIM * NF + p;
      double* tb = tbuf + (long long)e * NTR + (lf * (1 + DIM) * NV + vv) * NF + p;
      tb[0] = ext[0];
#pragma unroll
      for (int j = 0; j < DIM; ++j) {
        double a = 0.0;
#pragma unroll
        for (int rr = 0; rr < DIM; ++rr) a = fma(gp[(rr * DIM + j) * NF], ext[1 + rr], a);
        tb[(1 + j) * NV * NF] = a;
      }
    }
    return;
  }
  for (int idx = threadIdx.x; idx < EPB * NTR; idx += blockDim.x) {
    const int eb = idx / NTR;
    int rem = idx - eb * NTR;
    const int e = e0 + eb;
    if (e >= E) continue;
    const int p = rem % NF;
    rem /= NF;
    const int vv = rem % NV;
    rem /= NV;
    const int fld = rem % (1 + DIM);
    const int lf = rem / (1 + DIM);
    const int r = lf >> 1;
    const double* lw = sl + (lf & 1) * Q;
    const double* src = fld == 0 ? sQ + (eb * NV + vv) * NQ
                                 : sG + (((fld - 1) * EPB + eb) * NV + vv) * NQ;
    // grid offset of the face point and stride along direction r
    int c[3] = {0, 0, 0};
    if (DIM == 2) {
      c[1 - r] = p;
    } else {
      const int t0 = r == 0 ? 1 : 0, t1 = r == 2 ? 1 : 2;
      c[t0] = p % Q;
      c[t1] = p / Q;
    }
    const int base = c[0] + Q * c[1] + Q * Q * c[2];
    const int str = r == 0 ? 1 : (r == 1 ? Q : Q * Q);
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < Q; ++k) acc = fma(lw[k], src[base + k * str], acc);
    if (fld > 0) acc *= geo[e].rh[fld - 1];
    tbuf[(long long)e * NTR + ((lf * (1 + DIM) + fld) * NV + vv) * NF + p] = acc;
  }
}

// B^T on G [EPB][NV][NQ] -> result in R [EPB][NV][NM] (general elements: the
// dense inverse mass matrix is applied by the caller)
template <int DIM, int P, int Q>
__device__ __forceinline__ void bt_only(double* sG, double* t1, double* t2, double* sR,
                                        const double* sB, int nrep) {
  using C = Cfg<DIM, P, Q>;
  constexpr int N = C::N, Q2 = C::Q2, N2 = C::N2;
  if (DIM == 2) {
    contract<Q, Q, 1, 1, N, 1, N, false>(sG, t1, sB, nrep);
    __syncthreads();
    contract<Q, N, 1, 0, N, 1, N, false>(t1, sR, sB, nrep);
  } else {
    contract<Q, Q, Q2, 2, N, 1, N, false>(sG, t1, sB, nrep);
    __syncthreads();
    contract<Q, Q, N2, 1, N, 1, N, false>(t1, t2, sB, nrep);
    __syncthreads();
    contract<Q, N, N2, 0, N, 1, N, false>(t2, sR, sB, nrep);
  }
  __syncthreads();
}

// out = M_e^-1 x for the coefficient vector x (NM values in shared memory)
template <int NM>
__device__ __forceinline__ double dense_minv_row(const double* __restrict__ Mi, int m,
                                                 const double* x) {
  double a = 0.0;
#pragma unroll 8
  for (int k = 0; k < NM; ++k) a = fma(Mi[(long long)k * NM + m], x[k], a);  // M^-1 symmetric
  return a;
}

// B^T then |J|^-1 (M1^-1)^(x)d on G [EPB][NV][NQ] -> result in R [EPB][NV][NM]
template <int DIM, int P, int Q>
__device__ __forceinline__ void bt_minv(double* sG, double* t1, double* t2, double* sR,
                                        const double* sB, const double* sMi, int nrep) {
  using C = Cfg<DIM, P, Q>;
  constexpr int N = C::N, Q2 = C::Q2, N2 = C::N2;
  if (DIM == 2) {
    contract<Q, Q, 1, 1, N, 1, N, false>(sG, t1, sB, nrep);
    __syncthreads();
    contract<Q, N, 1, 0, N, 1, N, false>(t1, t2, sB, nrep);
    __syncthreads();
    contract<N, N, 1, 0, N, N, 1, false>(t2, t1, sMi, nrep);
    __syncthreads();
    contract<N, N, 1, 1, N, N, 1, false>(t1, sR, sMi, nrep);
  } else {
    contract<Q, Q, Q2, 2, N, 1, N, false>(sG, t1, sB, nrep);
    __syncthreads();
    contract<Q, Q, N2, 1, N, 1, N, false>(t1, t2, sB, nrep);
    __syncthreads();
    contract<Q, N, N2, 0, N, 1, N, false>(t2, t1, sB, nrep);
    __syncthreads();
    contract<N, N, N2, 0, N, N, 1, false>(t1, t2, sMi, nrep);
    __syncthreads();
    contract<N, N, N2, 1, N, N, 1, false>(t2, t1, sMi, nrep);
    __syncthreads();
    contract<N, N, N2, 2, N, N, 1, false>(t1, sR, sMi, nrep);
  }
  __syncthreads();
}

// L2 projection of the analytic field (what = 0) or of the forcing (what = 1)
template <int DIM, int P, int Q, bool CV>
__global__ void __launch_bounds__(256) project_kernel(const __grid_constant__ Tables tab,
                                                      const __grid_constant__ Phys ph,
                                                      const ElemGeo* __restrict__ geo,
                                                      const __grid_constant__ GenGeo gg, int E,
                                                      int what, double t,
                                                      double* __restrict__ out) {
  using C = Cfg<DIM, P, Q>;
  constexpr int N = C::N, NV = C::NV, NM = C::NM, NQ = C::NQ, EPB = C::EPB;
  extern __shared__ double sm[];
  double* sB = sm;
  double* sl = sB + Q * N + Q * Q;
  double* sMi = sl + 2 * Q;
  double* sw = sMi + N * N;
  double* sH = sm + C::TAB;
  double* sG = sH + DIM * EPB * NV * NQ;
  double* t1 = sG + EPB * NV * NQ;
  double* t2 = t1 + EPB * NV * NQ;
  const int e0 = blockIdx.x * EPB;
  stage_tables<DIM, P, Q>(tab, sm);
  __syncthreads();
  for (int idx = threadIdx.x; idx < EPB * NQ; idx += blockDim.x) {
    const int eb = idx / NQ, q = idx - eb * NQ;
    const int e = e0 + eb;
    double U[NV];
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) U[vv] = 0.0;
    if (e < E) {
      double x[3] = {0, 0, 0};
      double wJ = 1.0;
      if constexpr (CV) {
        for (int r = 0; r < DIM; ++r) x[r] = gg.vx[((long long)e * DIM + r) * NQ + q];
        wJ = gg.vgeo[((long long)e * (DIM * DIM + 1) + DIM * DIM) * NQ + q];
      } else {
        const ElemGeo g = geo[e];
        int c[3];
        grid_coords<DIM, Q>(q, c);
        for (int r = 0; r < DIM; ++r) {
          x[r] = g.x0[r] + 0.5 * (tab.x[c[r]] + 1.0) * g.h[r];
          wJ *= sw[c[r]] * 0.5 * g.h[r];
        }
      }
      if (what == 0)
        exact_state(DIM, ph, x, t, U);
      else
        forcing(DIM, ph, x, U);
#pragma unroll
      for (int vv = 0; vv < NV; ++vv) U[vv] *= wJ;
    }
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) sG[(eb * NV + vv) * NQ + q] = U[vv];
  }
  __syncthreads();
  if constexpr (CV)
    bt_only<DIM, P, Q>(sG, t1, t2, sH, sB, EPB * NV);
  else
    bt_minv<DIM, P, Q>(sG, t1, t2, sH, sB, sMi, EPB * NV);
  for (int i = threadIdx.x; i < EPB * NV * NM; i += blockDim.x) {
    const int eb = i / (NV * NM);
    const int e = e0 + eb;
    if (e >= E) continue;
    double val;
    if constexpr (CV) {
      const int m = i % NM;
      val = dense_minv_row<NM>(gg.minv + (long long)e * NM * NM, m, sH + (i - m));
    } else {
      val = sH[i] * geo[e].idet;
    }
    out[(long long)e * NV * NM + (i - eb * NV * NM)] = val;
  }
}

// ---------------------------------------------------------------- launchers
template <int DIM, int P, int Q>
static dg_status run_sensor(dg_mesh_s* m, const double* u, const double* v, const double* eps,
                            double* out, cudaStream_t s);

template <int DIM, int P, int Q>
static dg_status run_residual(dg_mesh_s* m, const EvalArgs& a, cudaStream_t s) {
  // (with shock capturing the elements' artificial-viscosity factors first)
  if (!a.skip_face && m->phys.avf) DG_TRY((run_sensor<DIM, P, Q>(m, a.u, a.v, a.eps, m->avf, s)));
  if (m->curved) {
    if constexpr (has_curved<DIM, P, Q>()) return launch_gen<DIM, P, Q>(m, a, s);
    return DG_ERR_UNSUPPORTED;
  }
  return launch_fix<DIM, P, Q>(m, a, s);
}

// FP64 traces for the preconditioner build: its trace Jacobians are one-sided
// differences over 1e-8 steps, so they keep the arithmetic of the blocks' own
// FP64 state evaluation
template <int DIM, int P, int Q, bool CV>
static dg_status run_traces_g(dg_mesh_s* m, const double* u, cudaStream_t s) {
  using C = Cfg<DIM, P, Q>;
  if (m->phys.avf) DG_TRY((run_sensor<DIM, P, Q>(m, u, nullptr, nullptr, m->avf, s)));
  const size_t sm = sizeof(double) * C::VOL_SM;
  DG_CUDA(cudaFuncSetAttribute(trace_kernel<DIM, P, Q, CV>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  DG_PROF(K_TRACE, s, trace_kernel<DIM, P, Q, CV><<<(m->E + C::EPB - 1) / C::EPB, C::NT, sm, s>>>(
      m->tab, m->geo, gen_geo(m), m->E, u, m->tbuf));
  DG_LAUNCHED(1);
  return DG_OK;
}
template <int DIM, int P, int Q>
static dg_status run_traces(dg_mesh_s* m, const double* u, cudaStream_t s) {
  if (m->curved) {
    if constexpr (has_curved<DIM, P, Q>()) return run_traces_g<DIM, P, Q, true>(m, u, s);
    return DG_ERR_UNSUPPORTED;
  }
  return run_traces_g<DIM, P, Q, false>(m, u, s);
}

// Launch shapes before tuning.  Axis-aligned elements: blocks of about 128
// threads (several per SM, so that one block's contractions run beside another's
// fluxes; 16^3 P = 3 volume kernel: 270 us at 128 threads, 332 at 224) with up
// to 256 volume points or 224 face points, halved while the grid would leave
// SMs idle.
template <int DIM, int P, int Q>
static void default_tune(dg_mesh_s* m) {
  using C = Cfg<DIM, P, Q>;
  auto threads = [](int points, int most) {
    const int t = (points + 31) / 32 * 32;
    return t < 64 ? 64 : (t > most ? most : t);
  };
  int epb = 256 / C::NQ > 1 ? 256 / C::NQ : 1;
  if (DIM == 2 && epb > 8) epb = 8;
  while (epb > 1 && (m->E + epb - 1) / epb < 2 * 152) epb /= 2;
  m->tune.vol_epb = epb;
  m->tune.vol_threads = threads(epb * C::NQ, C::NQ > 256 ? 256 : 128);
  if (DIM == 3 && m->tune.vol_threads < 128) m->tune.vol_threads = 128;
  int fe = 224 / (C::NF * DIM) > 1 ? 224 / (C::NF * DIM) : 1;
  if (fe > 4) fe = 4;
  while (fe > 1 && (m->F + fe * DIM - 1) / (fe * DIM) < 2 * 152) fe /= 2;
  m->tune.lift_epb = fe;
  m->tune.lift_threads = threads(fe * DIM * C::NF, 224);
  if (DIM == 3 && m->tune.lift_threads < 128) m->tune.lift_threads = 128;
}

// candidate (elements per CTA, threads per CTA) launch shapes whose shared
// memory one CTA can have; lift: the face kernel's, DIM faces an element
template <int DIM, class A>
static void tune_candidates_of(std::vector<int2>& vol, std::vector<int2>& lift) {
  const int epbs3[] = {1, 2, 3, 4};
  const int epbs2[] = {1, 2, 4, 8, 16, 32};
  // every warp multiple up to the kernels' bound: a count just above the
  // Gauss points of one or more elements (224 for 216 at Q = 6) gives the
  // per-point flux stage one pass without idle lanes
  const int nts[] = {64, 96, 128, 160, 192, 224, 256};
  for (int e : (DIM == 3 ? std::vector<int>(epbs3, epbs3 + 4) : std::vector<int>(epbs2, epbs2 + 6)))
    for (int t : nts) {
      if (DIM == 3 && t < 128) continue;
      if (A::vol_bytes(e) <= FIX_SMEM) vol.push_back(make_int2(e, t));
      if (A::face_bytes(e * DIM) <= FIX_SMEM) lift.push_back(make_int2(e, t));
    }
}
template <int DIM, int P, int Q>
static void tune_candidates(const dg_mesh_s* m, std::vector<int2>& vol, std::vector<int2>& lift) {
  if (m->curved)
    tune_candidates_of<DIM, Gen<DIM, P, Q>>(vol, lift);
  else
    tune_candidates_of<DIM, Aff<DIM, P, Q>>(vol, lift);
}

template <int DIM, int P, int Q, bool CV>
static dg_status run_project_g(dg_mesh_s* m, int what, double t, double* out, cudaStream_t s) {
  using C = Cfg<DIM, P, Q>;
  const int nb = (m->E + C::EPB - 1) / C::EPB;
  const size_t lsm = sizeof(double) * C::LIFT_SM;
  DG_CUDA(cudaFuncSetAttribute(project_kernel<DIM, P, Q, CV>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lsm));
  DG_PROF(K_PROJECT, s, project_kernel<DIM, P, Q, CV><<<nb, C::NT, lsm, s>>>(
      m->tab, m->phys, m->geo, gen_geo(m), m->E, what, t, out));
  DG_LAUNCHED(1);
  return DG_OK;
}

template <int DIM, int P, int Q>
static dg_status run_project(dg_mesh_s* m, int what, double t, double* out, cudaStream_t s) {
  if (m->curved) {
    if constexpr (has_curved<DIM, P, Q>()) return run_project_g<DIM, P, Q, true>(m, what, t, out, s);
    return DG_ERR_UNSUPPORTED;
  }
  return run_project_g<DIM, P, Q, false>(m, what, t, out, s);
}

dg_status build_minv_exponents(dg_mesh_s* m, cudaStream_t s) {
#define DG_RUN(D_, P_, Q_) \
  if (m->dim == D_ && m->P == P_ && m->Q == Q_) return launch_minv_exp<D_, P_, Q_>(m, s);
  DG_CURVED_INSTANCES(DG_RUN)
#undef DG_RUN
  return DG_ERR_UNSUPPORTED;
}

bool supported_curved(int dim, int P, int Q) {
#define DG_SUP(D_, P_, Q_) \
  if (dim == D_ && P == P_ && Q == Q_) return true;
  DG_CURVED_INSTANCES(DG_SUP)
#undef DG_SUP
  return false;
}

bool supported(int dim, int P, int Q) {
#define DG_SUP(D_, P_, Q_) \
  if (dim == D_ && P == P_ && Q == Q_) return true;
  DG_INSTANCES(DG_SUP)
#undef DG_SUP
  return false;
}

dg_status launch_residual(dg_mesh_s* m, const EvalArgs& a, cudaStream_t s) {
#define DG_RUN(D_, P_, Q_) \
  if (m->dim == D_ && m->P == P_ && m->Q == Q_) return run_residual<D_, P_, Q_>(m, a, s);
  DG_INSTANCES(DG_RUN)
#undef DG_RUN
  return DG_ERR_UNSUPPORTED;
}

template <int DIM, int P, int Q>
static dg_status run_sensor(dg_mesh_s* m, const double* u, const double* v, const double* eps,
                            double* out, cudaStream_t s) {
  const GenGeo gg = gen_geo(m);
  const int nb = (m->E + SENSOR_WARPS - 1) / SENSOR_WARPS;
  if (m->curved) {
    if constexpr (has_curved<DIM, P, Q>()) {
      DG_PROF(K_SENSOR, s, sensor_kernel<DIM, P, Q, true><<<nb, 32 * SENSOR_WARPS, 0, s>>>(
          m->stab, m->phys, m->geo, gg, m->E, u, v, eps, out));
      DG_LAUNCHED(1);
      return DG_OK;
    }
    return DG_ERR_UNSUPPORTED;
  }
  DG_PROF(K_SENSOR, s, sensor_kernel<DIM, P, Q, false><<<nb, 32 * SENSOR_WARPS, 0, s>>>(
      m->stab, m->phys, m->geo, gg, m->E, u, v, eps, out));
  DG_LAUNCHED(1);
  return DG_OK;
}

dg_status launch_traces(dg_mesh_s* m, const double* u, cudaStream_t s) {
  if (!m->tbuf) {
    const size_t n = sizeof(double) * (size_t)m->E * 2 * m->dim * (1 + m->dim) * m->nv * m->nf;
    DG_CUDA(cudaMalloc((void**)&m->tbuf, n));
    DG_CUDA(cudaMemsetAsync(m->tbuf, 0, n, s));
  }
#define DG_RUN(D_, P_, Q_) \
  if (m->dim == D_ && m->P == P_ && m->Q == Q_) return run_traces<D_, P_, Q_>(m, u, s);
  DG_INSTANCES(DG_RUN)
#undef DG_RUN
  return DG_ERR_UNSUPPORTED;
}

dg_status launch_sensor(dg_mesh_s* m, const double* u, double* out, cudaStream_t s) {
#define DG_RUN(D_, P_, Q_) \
  if (m->dim == D_ && m->P == P_ && m->Q == Q_) return run_sensor<D_, P_, Q_>(m, u, nullptr, nullptr, out, s);
  DG_INSTANCES(DG_RUN)
#undef DG_RUN
  return DG_ERR_UNSUPPORTED;
}

dg_status launch_project(dg_mesh_s* m, int what, double t, double* out, cudaStream_t s) {
#define DG_RUN(D_, P_, Q_) \
  if (m->dim == D_ && m->P == P_ && m->Q == Q_) return run_project<D_, P_, Q_>(m, what, t, out, s);
  DG_INSTANCES(DG_RUN)
#undef DG_RUN
  return DG_ERR_UNSUPPORTED;
}

template <int DIM, int P, int Q>
static dg_status run_autotune(dg_mesh_s* m, int reps, dg_tune_result* res, cudaStream_t s) {
  std::vector<int2> vc, lc;
  tune_candidates<DIM, P, Q>(m, vc, lc);
  // a valid state to time on: the projected analytic field
  DG_TRY(launch_project(m, 0, 0.0, m->w1, s));
  EvalArgs a{};
  a.u = m->w1;
  a.out = m->w2;
  cudaEvent_t e0, e1;
  DG_CUDA(cudaEventCreate(&e0));
  DG_CUDA(cudaEventCreate(&e1));
  const Tune keep = m->tune;
  auto time_it = [&](bool vol) -> double {
    EvalArgs b = a;
    (vol ? b.skip_face : b.skip_vol) = true;
    run_residual<DIM, P, Q>(m, b, s);  // warm-up
    cudaEventRecord(e0, s);
    for (int r = 0; r < reps; ++r) run_residual<DIM, P, Q>(m, b, s);
    cudaEventRecord(e1, s);
    cudaEventSynchronize(e1);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    return ms / reps;
  };
  run_residual<DIM, P, Q>(m, a, s);  // face data for the volume kernel
  // the shape in effect before tuning is timed too when it is not a candidate
  double best = 1e30, dflt = -1.0;
  Tune t = keep;
  for (const int2& c : vc) {
    m->tune.vol_epb = c.x;
    m->tune.vol_threads = c.y;
    const double ms = time_it(true);
    if (c.x == keep.vol_epb && c.y == keep.vol_threads) dflt = ms;
    if (ms < best) {
      best = ms;
      t.vol_epb = c.x;
      t.vol_threads = c.y;
    }
  }
  if (dflt < 0.0) {
    m->tune.vol_epb = keep.vol_epb;
    m->tune.vol_threads = keep.vol_threads;
    dflt = time_it(true);
  }
  res->vol_ms = best;
  res->vol_ms_default = dflt;
  m->tune.vol_epb = t.vol_epb;
  m->tune.vol_threads = t.vol_threads;
  best = 1e30;
  dflt = -1.0;
  for (const int2& c : lc) {
    m->tune.lift_epb = c.x;
    m->tune.lift_threads = c.y;
    const double ms = time_it(false);
    if (c.x == keep.lift_epb && c.y == keep.lift_threads) dflt = ms;
    if (ms < best) {
      best = ms;
      t.lift_epb = c.x;
      t.lift_threads = c.y;
    }
  }
  if (dflt < 0.0) {
    m->tune.lift_epb = keep.lift_epb;
    m->tune.lift_threads = keep.lift_threads;
    dflt = time_it(false);
  }
  res->lift_ms = best;
  res->lift_ms_default = dflt;
  m->tune = t;
  res->vol_epb = t.vol_epb;
  res->vol_threads = t.vol_threads;
  res->lift_epb = t.lift_epb;
  res->lift_threads = t.lift_threads;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  DG_CUDA(cudaGetLastError());
  return DG_OK;
}

void init_tune(dg_mesh_s* m) {
#define DG_RUN(D_, P_, Q_) \
  if (m->dim == D_ && m->P == P_ && m->Q == Q_) default_tune<D_, P_, Q_>(m);
  DG_INSTANCES(DG_RUN)
#undef DG_RUN
}

dg_status autotune(dg_mesh_s* m, int reps, dg_tune_result* res, cudaStream_t s) {
#define DG_RUN(D_, P_, Q_) \
  if (m->dim == D_ && m->P == P_ && m->Q == Q_) return run_autotune<D_, P_, Q_>(m, reps, res, s);
  DG_INSTANCES(DG_RUN)
#undef DG_RUN
  return DG_ERR_UNSUPPORTED;
}

bool tune_valid(dg_mesh_s* m, const dg_tune_result* t) {
  bool ok = false;
#define DG_RUN(D_, P_, Q_)                                                            \
  if (m->dim == D_ && m->P == P_ && m->Q == Q_) {                                     \
    std::vector<int2> vc, lc;                                                         \
    tune_candidates<D_, P_, Q_>(m, vc, lc);                                            \
    bool v = false, l = false;                                                        \
    for (const int2& c : vc) v |= c.x == t->vol_epb && c.y == t->vol_threads;         \
    for (const int2& c : lc) l |= c.x == t->lift_epb && c.y == t->lift_threads;       \
    ok = v && l;                                                                      \
  }
  DG_INSTANCES(DG_RUN)
#undef DG_RUN
  return ok;
}

}  // namespace dg
