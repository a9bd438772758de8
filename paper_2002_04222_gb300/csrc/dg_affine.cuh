// The residual on axis-aligned elements in two kernels:
//   face_fix_kernel  traces of Q and grad Q from the two sides' coefficients,
//                    numerical flux and symmetric flux, the tangential part
//                    of the symmetric flux's lift (D_t^T) on the face;
//   vol_fix_kernel   BwdTrans, Gauss-grid derivatives, volume flux, the lift of
//                    both (D_j^T, J^T), M^-1 B^T, and the residual's or the
//                    Jacobian-free product's epilogue.
// All contractions run in 64-bit fixed point (dg_fix.cuh); FP64 remains for
// the pointwise fluxes, which bound both kernels: 216 volume points of 120 FP64
// instructions and 108 face points of 249 per element at P = 3 (ncu) against
// about 70,000 multiply-adds of contractions, which took 60% of the FP64 pipe's
// time when they ran there.
//
// With H~_r = (2/h_r) H_r, w the 1-D weights and M1 the 1-D mass matrix, the
// metric cancels between M^-1 and the integrals:
//   R = (A x A x A) G,   A = M1^-1 B^T W,
//   G = sum_r Dh_r H~_r + sum_faces lh(q_r) P0 + ld(q_r) P1,
//   Dh[q][k] = w_k l_q'(x_k) / w_q,  lh = l_q(+-1) / w_q,  ld = l_q'(+-1) / w_q,
//   P0 = (2/h_r) (-+ f + T),  T = c beta_s sum_t (2/h_t) Dh_t S_t  (t tangential),
//   P1 = (2/h_r)^2 c beta_s S_r,
// f the numerical flux along +x_r, c = 1/2 inside and 1 on a boundary.
#pragma once
#include "dg_affine.h"
#include "dg_fix.cuh"
#include "dg_physics.cuh"
#include "dg_sumfact.cuh"

namespace dg {

// ------------------------------------------------------------ pointwise fluxes
// H~_r = rh_r (F_r - G_r) at a volume point; dU[r] are reference derivatives
// (the physical ones are rh_r dU[r]).  One reciprocal; rh and mu ride on
// factors that each product needs anyway.
template <int D>
__device__ __forceinline__ void vol_flux_point(const double* U, const double dU[D][D + 2],
                                               const double* rh, const Phys& ph, double fe,
                                               double H[D][D + 2]) {
  const double irho = 1.0 / U[0];
  double vel[D], ke = 0.0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    vel[k] = U[1 + k] * irho;
    ke = fma(U[1 + k], vel[k], ke);
  }
  const double p = ph.gm1 * fma(-0.5, ke, U[D + 1]);
  const double Ep = U[D + 1] + p;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const double vr = vel[i] * rh[i];
    H[i][0] = U[1 + i] * rh[i];
#pragma unroll
    for (int k = 0; k < D; ++k) H[i][1 + k] = U[1 + k] * vr;
    H[i][1 + i] = fma(p, rh[i], H[i][1 + i]);
    H[i][D + 1] = vr * Ep;
  }
  if (!ph.viscous) return;
  const double e = U[D + 1] * irho;
  double mu = ph.mu;
  if (ph.mu_law != 0) mu = viscosity(ph.gMa2 * p * irho, ph);
  if (fe != 0.0) {
    double a = fe * U[0] * (sqrt(ph.gamma * p * irho) + sqrt(ke * irho));
    if (ph.av_mode == 2) {
      double dv[D][D];
#pragma unroll
      for (int j = 0; j < D; ++j)
#pragma unroll
        for (int k = 0; k < D; ++k)
          dv[j][k] = (dU[j][1 + k] - vel[k] * dU[j][0]) * irho * rh[j];
      a *= ducros_ratio<D>(dv);
    }
    mu += a;
  }
  const double mi = mu * irho, ck = ph.gMa2 * ph.gm1 * ph.kappa_fac;
  double dv[D][D], en[D];  // mu d u_k / d x_j; the heat flux
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const double mr = mi * rh[j];
    double s = fma(-e, dU[j][0], dU[j][D + 1]);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const double t = fma(-vel[k], dU[j][0], dU[j][1 + k]);
      s = fma(-t, vel[k], s);
      dv[j][k] = mr * t;
    }
    en[j] = (ck * mr) * s;
  }
  double div = dv[0][0];
#pragma unroll
  for (int k = 1; k < D; ++k) div += dv[k][k];
  const double tt = (2.0 / 3.0) * div;
  double tau[D][D];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    tau[i][i] = fma(2.0, dv[i][i], -tt);
#pragma unroll
    for (int k = i + 1; k < D; ++k) tau[i][k] = tau[k][i] = dv[i][k] + dv[k][i];
  }
#pragma unroll
  for (int i = 0; i < D; ++i) {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      H[i][1 + k] = fma(-rh[i], tau[i][k], H[i][1 + k]);
      en[i] = fma(vel[k], tau[i][k], en[i]);
    }
    H[i][D + 1] = fma(-rh[i], en[i], H[i][D + 1]);
  }
}

// Roe flux along +e_0 between the states on the lower and the upper side
template <int D>
__device__ __forceinline__ void roe_flux_point(const double* UL, const double* UR, const Phys& ph,
                                               double* Fh) {
  // 1/rho and sqrt(rho) of both sides from one reciprocal square root each
  const double rsL = rsqrt(UL[0]), rsR = rsqrt(UR[0]);
  const double iL = rsL * rsL, iR = rsR * rsR;
  const double sL = UL[0] * rsL, sR = UR[0] * rsR;
  double vL[D], vR[D], keL = 0.0, keR = 0.0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    vL[k] = UL[1 + k] * iL;
    vR[k] = UR[1 + k] * iR;
    keL = fma(UL[1 + k], vL[k], keL);
    keR = fma(UR[1 + k], vR[k], keR);
  }
  const double pL = ph.gm1 * fma(-0.5, keL, UL[D + 1]), pR = ph.gm1 * fma(-0.5, keR, UR[D + 1]);
  const double EL = UL[D + 1] + pL, ER = UR[D + 1] + pR;
  const double isum = 1.0 / (sL + sR);
  // Roe averages: the weights sL/(sL+sR), sR/(sL+sR); sL H_L = rs_L (E_L + p_L)
  const double wL = sL * isum, wR = sR * isum;
  double ut[D], du[D], q2 = 0.0, udu = 0.0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    ut[k] = fma(wL, vL[k], wR * vR[k]);
    du[k] = vR[k] - vL[k];
    q2 = fma(ut[k], ut[k], q2);
    if (k != 0) udu = fma(ut[k], du[k], udu);
  }
  const double Ht = fma(rsL, EL, rsR * ER) * isum;
  const double c2 = ph.gm1 * fma(-0.5, q2, Ht);
  const double rc = rsqrt(c2);
  const double c = c2 * rc, ic2 = rc * rc;
  const double dp = pR - pL, rt = sL * sR;
  const double hic2 = 0.5 * ic2, rcd = rt * c * du[0];
  const double a2 = fma(-dp, ic2, UR[0] - UL[0]);
  const double l2 = fabs(ut[0]);
  const double w1 = fabs(ut[0] - c) * ((dp - rcd) * hic2), w5 = fabs(ut[0] + c) * ((dp + rcd) * hic2);
  const double w2 = l2 * a2, ws = l2 * rt, w15 = w1 + w5, wc = (w5 - w1) * c, wt = w15 + w2;
  Fh[0] = 0.5 * (fma(UL[0], vL[0], UR[0] * vR[0]) - wt);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    double f = fma(UL[1 + k], vL[0], UR[1 + k] * vR[0]);
    f = fma(-wt, ut[k], f);
    if (k == 0)
      f += (pL + pR) - wc;
    else
      f = fma(-ws, du[k], f);
    Fh[1 + k] = 0.5 * f;
  }
  double f = fma(EL, vL[0], ER * vR[0]);
  f = fma(-w15, Ht, f);
  f = fma(-wc, ut[0], f);
  f = fma(-0.5 * w2, q2, f);
  Fh[D + 1] = 0.5 * fma(-ws, udu, f);
}

// the other Riemann fluxes along +e_0 (kept out of line: the Roe path's
// registers set the face kernel's occupancy)
template <int D>
__device__ __noinline__ void other_flux_point(const double* UL, const double* UR, const Phys& ph,
                                              double* Fh) {
  double n[D];
#pragma unroll
  for (int k = 0; k < D; ++k) n[k] = k == 0 ? 1.0 : 0.0;
  riemann_flux<D>(UL, UR, n, ph, Fh);
}

// boundary data at a face point in the face's frame (component 0 = normal):
// U the interior state, sgn the outward direction along +e_r; QR the exterior
// Riemann state, QB the viscous state
template <int D>
__device__ __noinline__ bool boundary_point(int bctype, const Phys& ph, const double* x, double t,
                                            int r, double sgn, const double* U, double* QR,
                                            double* QB) {
  constexpr int NV = D + 2;
  const int t0 = r == 0 ? 1 : 0, t1 = r == 2 ? 1 : 2;
  const int ax[3] = {r, t0, t1};
  double Ux[NV], Rx[NV], Bx[NV], n[D];
  for (int k = 0; k < D; ++k) n[k] = k == r ? sgn : 0.0;
  Ux[0] = U[0];
  Ux[NV - 1] = U[NV - 1];
  for (int k = 0; k < D; ++k) Ux[1 + ax[k]] = U[1 + k];
  const bool ad = boundary_states<D>(bctype, ph, x, t, Ux, n, Rx, Bx);
  QR[0] = Rx[0];
  QB[0] = Bx[0];
  QR[NV - 1] = Rx[NV - 1];
  QB[NV - 1] = Bx[NV - 1];
  for (int k = 0; k < D; ++k) {
    QR[1 + k] = Rx[1 + ax[k]];
    QB[1 + k] = Bx[1 + ax[k]];
  }
  return ad;
}

// geometry and connectivity of a face in the face kernel
struct FaceInfo {
  int eA, eB;        // elements below and above the face along x_r (-1: none)
  int r, bc;         // normal direction, boundary type (0: interior)
  double hn, ht[2];  // half of the largest 2/h_n, halves of the tangential 2/h_t
  int rhA[2], rhB[2];  // 2/h_n of each side over the largest, 62-bit halves
  FixScale ct[2];    // c beta_s 2/h_t
  __device__ __forceinline__ void side(int s, int& e, int& lf) const {
    e = s == 0 ? eA : eB;
    lf = 2 * r + 1 - s;  // the side below has the face at its upper end
  }
};

static_assert(sizeof(FaceInfo) <= 128, "face_bytes");

// ------------------------------------------------------------ sides far apart
// Both sides' coefficients enter the face kernel at the larger of their two
// exponents, 59 bits: a side whose variable is more than 2^6 smaller than its
// neighbour's has fewer than a double's 53 left (32 beside one 10^8 times
// larger).  The sums of the derivatives need no more, but a flux can be that
// side's alone, so its values are then evaluated again from its coefficients
// in FP64, over those from the integers.  Out of line: blocks without such a
// face pay for one test (an exponent a side all the way through cost the kernel
// 1.5 to 3%, and the 8x8 P = 2 residual 2 of 27 us).
__device__ __forceinline__ bool far_below(int e, int other) { return other - max(e, FIX_EMIN) > 6; }

// the values of every smaller side, fields 0 and 1 of fld [face][stride]
template <int DIM, int P, int Q, class Info>
__device__ __noinline__ void own_values(const FixTab& ft, const Info* info, const int* sE, int nf,
                                        const double* __restrict__ u, const double* __restrict__ v,
                                        double eps, double* fld, int stride) {
  using A = Aff<DIM, P, Q>;
  constexpr int N = A::N, NV = A::NV, NM = A::NM, NF = A::NF;
  auto B = [&](int q, int k) {  // psi_k(x_q)
    const int2 c = ft.B[q * N + k];
    return ldexp(fma((double)c.x, 4294967296.0, (double)c.y), ft.eB - 62);
  };
  for (int idx = threadIdx.x; idx < nf * 2 * NV * NF; idx += blockDim.x) {
    const int p = idx % NF, fsv = idx / NF, vv = fsv % NV, side = fsv / NV % 2, fb = fsv / (2 * NV);
    const int* e2 = sE + fb * 2 * NV + vv;
    if (info[fb].bc != 0 || !far_below(e2[side * NV], e2[(1 - side) * NV])) continue;
    int e, lf;
    info[fb].side(side, e, lf);
    const int r = lf >> 1, sn = r == 0 ? 1 : (r == 1 ? N : N * N);
    const int s0 = r == 0 ? N : 1, s1 = r == 2 ? N : N * N;
    const long long g = ((long long)e * NV + vv) * NM + ((lf & 1) ? P * sn : 0);
    double s = 0.0;
    for (int b = 0; b < (DIM == 3 ? N : 1); ++b) {
      double row = 0.0;
      for (int a = 0; a < N; ++a) {
        const long long i = g + a * s0 + b * s1;
        row = fma(B(p % Q, a), v ? fma(eps, v[i], u[i]) : u[i], row);
      }
      s = DIM == 3 ? fma(B(p / Q, b), row, s) : row;
    }
    fld[fb * stride + (side * NV + vv) * NF + p] = s;
  }
  __syncthreads();
}

// ------------------------------------------------------------ face kernel
// One thread per (face, variable, line) in the transforms and one per face
// point in the flux.  FPB faces per block.  80 registers: the FP64 pipe waits
// on the other phases unless several blocks share an SM, and the few spilled
// values cost less (16^3 P = 3: 262 us at 128 registers, 245 at 96, 236 at 80;
// FP64 floor 184 us at 16 clocks per warp instruction; the 2-D instances were
// not timed with other limits).
template <int DIM, int P, int Q>
__global__ void __maxnreg__(80) face_fix_kernel(
    const __grid_constant__ FixTab ft, const __grid_constant__ Tables tab,
    const __grid_constant__ Phys ph, const ElemGeo* __restrict__ geo,
    const int32_t* __restrict__ faces, int F, double t, const double* __restrict__ dscal,
    const double* __restrict__ u, const double* __restrict__ v, const double* __restrict__ epsp,
    double* __restrict__ fflux, int32_t* __restrict__ fexp, const int FPB) {
  using A = Aff<DIM, P, Q>;
  constexpr int N = A::N, NV = A::NV, NM = A::NM, NF = A::NF, NT = A::NT, RQ = A::RQ, KK = A::KK;
  constexpr int VALA = 0, VALB = 1, DN = 2, DT = 3;
  extern __shared__ double sm[];
  double* sX = sm;                                   // [FPB][FX]
  double* sY = sX + FPB * A::FX;                     // [FPB][FY]
  FaceInfo* info = (FaceInfo*)(sY + FPB * A::FY);    // [FPB]
  int* sE = (int*)(info + FPB);                      // [FPB][2][NV] coefficients, both sides
  int* sS = sE + FPB * 2 * NV;                       // [FPB][3][NV] outputs f, T, S_n
  int* sT = sS + FPB * 3 * NV;                       // [FPB][NV] scaled tangential S
  const int f0 = blockIdx.x * FPB;
  const int nf = min(FPB, F - f0);
  const int tid = threadIdx.x, nth = blockDim.x;
  if (dscal) t = dscal[0];
  for (int i = tid; i < FPB * 6 * NV; i += nth) sE[i] = 0;
  for (int i = tid; i < nf; i += nth) {
    const int32_t* fp = faces + (long long)(f0 + i) * 6;
    const int eL = fp[0], fL = fp[1], eR = fp[2];
    FaceInfo g;
    g.eA = (fL & 1) ? eL : eR;
    g.eB = (fL & 1) ? eR : eL;
    g.r = fL >> 1;
    g.bc = eR >= 0 ? 0 : ph.bc[fp[5]];
    const int t0 = g.r == 0 ? 1 : 0, t1 = g.r == 2 ? 1 : 2;
    const double rA = geo[g.eA >= 0 ? g.eA : g.eB].rh[g.r], rB = geo[g.eB >= 0 ? g.eB : g.eA].rh[g.r];
    const double rmax = fmax(rA, rB);
    g.hn = 0.5 * rmax;
    const double one = 4611686018427387904.0;  // 2^62
    const double less = fmin(rA, rB) / rmax;  // (one division: the larger's is 1)
    fix_split(__double2ll_rn((rA < rB ? less : 1.0) * one), g.rhA[0], g.rhA[1]);
    fix_split(__double2ll_rn((rA < rB ? 1.0 : less) * one), g.rhB[0], g.rhB[1]);
    const double c = (eR >= 0 ? 0.5 : 1.0) * ph.beta_s;
    g.ht[0] = 0.5 * geo[eL].rh[t0];
    g.ct[0] = fix_scale(c * geo[eL].rh[t0]);
    g.ht[1] = DIM == 3 ? 0.5 * geo[eL].rh[t1] : 0.0;
    g.ct[1] = DIM == 3 ? fix_scale(c * geo[eL].rh[t1]) : g.ct[0];
    info[i] = g;
  }
  __syncthreads();
  // coefficients of both sides, their largest exponent per (face, side, variable)
  {
    const double eps = v ? epsp[0] : 0.0;
    const int lane = tid & 31, nw = nth >> 5;
    for (int j = tid >> 5; j < nf * 2 * NV; j += nw) {
      const int fb = j / (2 * NV), sv = j - fb * 2 * NV, side = sv / NV, vv = sv - side * NV;
      const int e = side == 0 ? info[fb].eA : info[fb].eB;
      if (e < 0) continue;  // warp-uniform
      const long long g = ((long long)e * NV + vv) * NM;
      double* dst = sX + fb * A::FX + sv * NM;
      int m = 0;
      for (int k = lane; k < NM; k += 32) {
        double val = u[g + k];
        if (v) val = fma(eps, v[g + k], val);
        dst[k] = val;
        m = max(m, fix_exp(val));
      }
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) sE[fb * 2 * NV + sv] = m;
    }
  }
  __syncthreads();
  // face coefficients per (face, variable, tangential mode): both sides'
  // values, their sum, and the sum of the normal derivatives scaled by 2/h_n
  // over the larger of the two (a boundary face counts its side twice)
  i64* C0 = (i64*)sY;
  bool far = false;
  for (int idx = tid; idx < nf * NV * NT; idx += nth) {
    const int fb = idx / (NV * NT), rem = idx - fb * NV * NT;
    const int vv = rem / NT, l = rem - vv * NT;
    const FaceInfo& g = info[fb];
    const int r = g.r;
    const int sn = r == 0 ? 1 : (r == 1 ? N : N * N);
    const int s0 = r == 0 ? N : 1, s1 = r == 2 ? N : N * N;
    const int off = (DIM == 3 ? (l % N) * s0 + (l / N) * s1 : l * s0);
    int bad;
    const int eA = sE[(fb * 2) * NV + vv], eB = sE[(fb * 2 + 1) * NV + vv];
    const int em = fix_emax(max(eA, eB), bad);
    far |= g.bc == 0 && far_below(min(eA, eB), max(eA, eB));
    i64 val[2] = {0, 0}, der[2] = {0, 0};
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      if ((side == 0 ? g.eA : g.eB) < 0) continue;
      const double* src = sX + fb * A::FX + (side * NV + vv) * NM + off;
      int xh[N], xl[N];
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const i64 x = to_fix(src[k * sn], em, 59);
        if (k == (side == 0 ? P : 0)) val[side] = x;
        fix_split(x, xh[k], xl[k]);
      }
      // the side below has the face at its upper end
      const i64 d = fix_dot<N>(xh, xl, ft.dp[1 - side]);
      der[side] = side == 0 ? fix_mul(d, g.rhA[0], g.rhA[1]) : fix_mul(d, g.rhB[0], g.rhB[1]);
    }
    if (g.eA < 0) {
      val[0] = val[1];
      der[0] = der[1];
    }
    if (g.eB < 0) {
      val[1] = val[0];
      der[1] = der[0];
    }
    i64* o = C0 + fb * A::FY + vv * NT + l;
    o[VALA * NV * NT] = val[0];
    o[VALB * NV * NT] = val[1];
    o[DN * NV * NT] = der[0] + der[1];
    o[DT * NV * NT] = val[0] + val[1];
  }
  const bool apart = __syncthreads_or(far);
  i64* C1 = (i64*)sX;  // 3-D: first tangential direction on its points, [4][NV][N][RQ]
  if constexpr (DIM == 3) {
    for (int idx = tid; idx < 4 * nf * NV * N; idx += nth) {
      const int kind = idx / (nf * NV * N), rem = idx - kind * nf * NV * N;
      const int fb = rem / (NV * N), vn = rem - fb * NV * N;  // (variable, second mode)
      int xh[N], xl[N];
      fix_line<N>(C0 + fb * A::FY + kind * NV * NT + vn * N, 1, xh, xl);
      i64* o = C1 + fb * A::FX + (kind * NV * N + vn) * RQ;
      if (kind == DT) {
#pragma unroll
        for (int q = 0; q < Q; ++q) o[q] = fix_dot<N>(xh, xl, ft.DB + q * N);
      } else {
#pragma unroll
        for (int q = 0; q < Q; ++q) o[q] = fix_dot<N>(xh, xl, ft.B + q * N);
      }
    }
    __syncthreads();
  }
  // last tangential direction; doubles at the face points, [KK][NV][NF]:
  // both values, d_n and d_t sums (2-D: one d_t)
  for (int idx = tid; idx < KK * nf * NV * (NF / Q); idx += nth) {
    constexpr int NL = NF / Q;
    const int kind = idx / (nf * NV * NL), rem = idx - kind * nf * NV * NL;
    const int fb = rem / (NV * NL), vq = rem - fb * NV * NL;
    const int vv = vq / NL, q0 = vq - vv * NL;
    int bad;
    int se = fix_emax(max(sE[(fb * 2) * NV + vv], sE[(fb * 2 + 1) * NV + vv]), bad) - 1022 - 59;
    int xh[N], xl[N];
    const i64* src;
    bool db;
    if constexpr (DIM == 3) {
      // kinds: A, B, d_n, d_t0 (derivative taken), d_t1 of the sum of A and B
      db = kind == DT + 1;
      se += (kind == DT ? ft.eDB : ft.eB) + (db ? ft.eDB : ft.eB) + (kind == DN ? ft.edp : 0);
      src = C1 + fb * A::FX + ((db ? VALA : kind) * NV + vv) * N * RQ + q0;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        i64 x = src[k * RQ];
        if (db) x += src[k * RQ + (VALB - VALA) * NV * N * RQ];
        fix_split(x, xh[k], xl[k]);
      }
    } else {
      db = kind == DT;
      se += (db ? ft.eDB : ft.eB) + (kind == DN ? ft.edp : 0);
      src = C0 + fb * A::FY + (kind * NV + vv) * NT;
#pragma unroll
      for (int k = 0; k < N; ++k) fix_split(src[k], xh[k], xl[k]);
    }
    double val[Q];
    if (db) {
#pragma unroll
      for (int q = 0; q < Q; ++q) val[q] = fix_to_double(fix_dot<N>(xh, xl, ft.DB + q * N), se, bad);
    } else {
#pragma unroll
      for (int q = 0; q < Q; ++q) val[q] = fix_to_double(fix_dot<N>(xh, xl, ft.B + q * N), se, bad);
    }
    // 2-D writes beside its inputs' region (the next line of the same variable
    // may still read it)
    double* o = (DIM == 3 ? sY + fb * A::FY : sX + fb * A::FX) + (kind * NV + vv) * NF + q0;
#pragma unroll
    for (int q = 0; q < Q; ++q) o[q * NL] = val[q];
  }
  double* sP = DIM == 3 ? sY : sX;
  constexpr int PS = DIM == 3 ? A::FY : A::FX;
  __syncthreads();
  if (apart)
    own_values<DIM, P, Q>(ft, info, sE, nf, u, v, v ? epsp[0] : 0.0, sP, PS);
  // fluxes, one thread per face point
  double* gF = fflux;
  double* gS = fflux + (long long)F * NV * NF;  // [F][2][NV-1][NF]: T, S_n
  for (int idx = tid; idx < nf * NF; idx += nth) {
    const int fb = idx / NF, p = idx - fb * NF;
    const FaceInfo& g = info[fb];
    const int f = f0 + fb, r = g.r;
    // variable order in the face's frame: density, normal, tangential momenta, energy
    int pv[NV];
    pv[0] = 0;
    pv[1] = 1 + r;
    pv[2] = 1 + (r == 0 ? 1 : 0);
    if (DIM == 3) pv[3] = 1 + (r == 2 ? 1 : 2);
    pv[NV - 1] = NV - 1;
    double* pt = sP + fb * PS + p;
    double UA[NV], UB[NV], QS[NV], jump[NV], Fh[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      UA[k] = pt[(VALA * NV + pv[k]) * NF];
      UB[k] = pt[(VALB * NV + pv[k]) * NF];
    }
    bool adiabatic = false;
    double mua = 0.0;
    if (ph.avf) {
      // artificial viscosity: the mean of the two sides' (a boundary: the interior's)
      const double a = g.eA >= 0 ? av_point<DIM>(UA, ph, ph.avf[g.eA]) : 0.0;
      const double b = g.eB >= 0 ? av_point<DIM>(UB, ph, ph.avf[g.eB]) : 0.0;
      mua = g.bc == 0 ? 0.5 * (a + b) : a + b;
      if (ph.av_mode == 2 && mua != 0.0) {
        double Qm[NV], dQ[DIM][NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          Qm[k] = 0.5 * (UA[k] + UB[k]);
          dQ[0][k] = g.hn * pt[(DN * NV + pv[k]) * NF];
#pragma unroll
          for (int j = 1; j < DIM; ++j) dQ[j][k] = g.ht[j - 1] * pt[((DT + j - 1) * NV + pv[k]) * NF];
        }
        mua *= ducros<DIM>(Qm, dQ);
      }
    }
    if (g.bc != 0) {
      const bool below = g.eA >= 0;  // the interior lies below the face
      const double sgn = below ? 1.0 : -1.0;
      const ElemGeo ge = geo[below ? g.eA : g.eB];
      double x[3] = {0, 0, 0}, QR[NV], QB[NV];
      int a = 0;
      for (int k = 0; k < DIM; ++k)
        if (k == r)
          x[k] = ge.x0[k] + (below ? ge.h[k] : 0.0);
        else
          x[k] = ge.x0[k] + 0.5 * (tab.x[a++ == 0 ? p % Q : p / Q] + 1.0) * ge.h[k];
      adiabatic = boundary_point<DIM>(g.bc, ph, x, t, r, sgn, UA, QR, QB);
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        QS[k] = 2.0 * QB[k];
        jump[k] = sgn * (UA[k] - QB[k]);
        if (below)
          UB[k] = QR[k];
        else
          UA[k] = QR[k];
      }
    } else {
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        QS[k] = UA[k] + UB[k];
        jump[k] = UA[k] - UB[k];
      }
    }
    const KeyGroup grp(fb);
    if (ph.riemann == DG_RIEMANN_ROE)
      roe_flux_point<DIM>(UA, UB, ph, Fh);
    else
      other_flux_point<DIM>(UA, UB, ph, Fh);
    if (ph.viscous) {
      const double irs = 1.0 / QS[0];
      double vel[DIM];
#pragma unroll
      for (int k = 0; k < DIM; ++k) vel[k] = QS[1 + k] * irs;
      const double e = QS[NV - 1] * irs;
      double mu = ph.mu;
      if (ph.mu_law != 0) {
        double q2 = 0.0;
#pragma unroll
        for (int k = 0; k < DIM; ++k) q2 = fma(vel[k], vel[k], q2);
        mu = viscosity(ph.gMa2 * ph.gm1 * fma(-0.5, q2, e), ph);
      }
      mu += mua;
      const double mi = 2.0 * mu * irs, ck = ph.gMa2 * ph.gm1 * ph.kappa_fac;
      // symmetric flux S_i = G_i({Q}, e_n (x) jump)
      double a[DIM], Sn[NV], s = fma(-e, jump[0], jump[NV - 1]);
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        const double tk = fma(-vel[k], jump[0], jump[1 + k]);
        s = fma(-tk, vel[k], s);
        a[k] = mi * tk;
      }
      const double tt = (2.0 / 3.0) * a[0];
      Sn[1] = 2.0 * tt;  // 2 a_n - (2/3) a_n
      double en = fma(vel[0], Sn[1], (ck * mi) * s);
#pragma unroll
      for (int k = 1; k < DIM; ++k) {
        Sn[1 + k] = a[k];
        en = fma(vel[k], a[k], en);
      }
      Sn[NV - 1] = adiabatic ? 0.0 : en;
      // row n of G({Q}, {grad Q})
      const double rn = mi * g.hn;
      double dn0 = pt[(DN * NV) * NF], gn[DIM];
      s = fma(-e, dn0, pt[(DN * NV + NV - 1) * NF]);
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        const double tk = fma(-vel[k], dn0, pt[(DN * NV + pv[1 + k]) * NF]);
        s = fma(-tk, vel[k], s);
        gn[k] = rn * tk;
      }
      double ge = (ck * rn) * s, div = gn[0], tau[DIM];
#pragma unroll
      for (int j = 1; j < DIM; ++j) {
        const double* d = pt + (DT + j - 1) * NV * NF;
        const double rt = mi * g.ht[j - 1], d0 = d[0];
        div = fma(rt, fma(-vel[j], d0, d[pv[1 + j] * NF]), div);
        tau[j] = fma(rt, fma(-vel[0], d0, d[pv[1] * NF]), gn[j]);
      }
      tau[0] = fma(2.0, gn[0], (-2.0 / 3.0) * div);
      const double beta = (double)((P + 1) * (P + 1)) * g.hn;
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        ge = fma(vel[k], tau[k], ge);
        Fh[1 + k] += fma(beta, Sn[1 + k], -tau[k]);
      }
      if (!adiabatic) Fh[NV - 1] += fma(beta, en, -ge);
      // outputs: S_n to memory; the tangential S_t (density component zero)
      // into this point's slots, for the lift below
      double* os = gS + ((long long)f * 2 + 1) * (NV - 1) * NF + p;
#pragma unroll
      for (int k = 1; k < NV; ++k) {
        os[(pv[k] - 1) * NF] = Sn[k];
        grp.max(sS + (fb * 3 + 2) * NV + pv[k], fix_exp(Sn[k]));
      }
#pragma unroll
      for (int j = 1; j < DIM; ++j) {
        double* d = pt + (j - 1) * NV * NF;
        double St[NV];
        const int er = g.ct[j - 1].er;
#pragma unroll
        for (int k = 1; k < NV; ++k) St[k] = 0.0;
        St[1] = a[j];
        St[1 + j] = -tt;
        St[NV - 1] = adiabatic ? 0.0 : fma(vel[0], a[j], -tt * vel[j]);
#pragma unroll
        for (int k = 1; k < NV; ++k) {
          d[pv[k] * NF] = St[k];
          grp.max(sT + fb * NV + pv[k], St[k] == 0.0 ? 0 : fix_exp(St[k]) + er);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      gF[((long long)f * NV + pv[k]) * NF + p] = Fh[k];
      grp.max(sS + (fb * 3) * NV + pv[k], fix_exp(Fh[k]));
    }
  }
  __syncthreads();
  // T = sum_t c beta_s (2/h_t) Dh_t S_t on the face's points (momentum and energy)
  if (ph.viscous) {
    if constexpr (DIM == 3) {
      for (int idx = tid; idx < nf * (NV - 1) * Q; idx += nth) {
        const int fb = idx / ((NV - 1) * Q), rem = idx - fb * (NV - 1) * Q;
        const int vv = 1 + rem / Q, q1 = rem % Q;
        int bad, xh[Q], xl[Q];
        const int em = fix_emax(sT[fb * NV + vv], bad);
        double* d = sP + fb * PS + vv * NF + q1 * Q;
        const FixScale sc = info[fb].ct[0];
#pragma unroll
        for (int k = 0; k < Q; ++k) fix_split(to_fix_mul(d[k], sc, em, 60), xh[k], xl[k]);
#pragma unroll
        for (int q = 0; q < Q; ++q) ((i64*)d)[q] = fix_dot<Q>(xh, xl, ft.Dh + q * Q);
      }
      __syncthreads();
    }
    for (int idx = tid; idx < nf * (NV - 1) * (NF / Q); idx += nth) {
      constexpr int NL = NF / Q;
      const int fb = idx / ((NV - 1) * NL), rem = idx - fb * (NV - 1) * NL;
      const int vv = 1 + rem / NL, q0 = rem % NL;
      int bad, xh[Q], xl[Q];
      const int em = fix_emax(sT[fb * NV + vv], bad);
      const double* d = sP + fb * PS + ((DIM - 2) * NV + vv) * NF + q0;
      const i64* d0 = (const i64*)sP + fb * PS + vv * NF + q0;
      const FixScale sc = info[fb].ct[DIM - 2];
#pragma unroll
      for (int k = 0; k < Q; ++k) fix_split(to_fix_mul(d[k * NL], sc, em, 60), xh[k], xl[k]);
      double* o = gS + ((long long)(f0 + fb) * 2 * (NV - 1) + vv - 1) * NF + q0;
      int big = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        i64 x = fix_dot<Q>(xh, xl, ft.Dh + q * Q);
        if (DIM == 3) x += d0[q * NL];
        const double val = fix_to_double(x, em - 1022 - 60 + ft.eDh, bad);
        o[q * NL] = val;
        big = max(big, fix_exp(val));
      }
      KeyGroup(fb * NV + vv).max(sS + (fb * 3 + 1) * NV + vv, big);
    }
    __syncthreads();
  }
  for (int i = tid; i < nf * 3 * NV; i += nth) fexp[(long long)f0 * 3 * NV + i] = sS[i];
}

// ------------------------------------------------------------ volume kernels' shared parts
// Coefficients of the elements e0 .. e0+ne-1 as doubles [ne][NV][NM] in dst,
// their largest exponent per (element, variable) in sE; sZ zeroed.  One warp
// per (element, variable).
template <int DIM, int P, int Q>
__device__ __forceinline__ void load_coefficients(const double* __restrict__ u,
                                                  const double* __restrict__ v, double eps, int e0,
                                                  int ne, double* dst, int* sE, int* sZ) {
  using A = Aff<DIM, P, Q>;
  constexpr int NV = A::NV, NM = A::NM;
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int j = threadIdx.x >> 5; j < ne * NV; j += nw) {
    const long long g = ((long long)e0 * NV + j) * NM;
    int m = 0;
    for (int k = lane; k < NM; k += 32) {
      double val = u[g + k];
      if (v) val = fma(eps, v[g + k], val);
      dst[j * NM + k] = val;
      m = max(m, fix_exp(val));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) {
      sE[j] = m;
      sZ[j] = 0;
    }
  }
}

// BwdTrans: directions 0, 1 (, 2) with B; coefficients in array 1 of s1, the
// other arrays of s1 in between, the values at the Gauss points in s0
template <int DIM, int P, int Q>
__device__ __forceinline__ void bwd_trans(const FixTab& ft, double* s0, double* s1, int ASZ,
                                          const int* sE, int ne) {
  using A = Aff<DIM, P, Q>;
  constexpr int N = A::N, NV = A::NV, N2 = A::N2, RQ = A::RQ, VP = A::VP;
  const int tid = threadIdx.x, nth = blockDim.x;
  i64* t1 = (i64*)(s1 + ASZ);
  for (int idx = tid; idx < ne * NV * N * N2; idx += nth) {
    const int ev = idx / (N * N2);
    int bad, xh[N], xl[N];
    const int em = fix_emax(sE[ev], bad);
    const double* src = s1 + idx * N;
#pragma unroll
    for (int k = 0; k < N; ++k) fix_split(to_fix(src[k], em, 60), xh[k], xl[k]);
    i64* o = t1 + idx * RQ;
#pragma unroll
    for (int q = 0; q < Q; ++q) o[q] = fix_dot<N>(xh, xl, ft.B + q * N);
  }
  __syncthreads();
  // direction 1: [ev][n2][n1][q0] -> [ev][n2][q1][q0]
  i64* t2 = DIM == 3 ? (i64*)(s1 + 2 * ASZ) : (i64*)s0;
  for (int idx = tid; idx < ne * NV * N2 * Q; idx += nth) {
    const int en = idx / Q, q0 = idx - en * Q;
    int xh[N], xl[N];
    fix_line<N>(t1 + en * N * RQ + q0, RQ, xh, xl);
    i64* o = t2 + en * Q * RQ + q0;
#pragma unroll
    for (int q = 0; q < Q; ++q) o[q * RQ] = fix_dot<N>(xh, xl, ft.B + q * N);
  }
  __syncthreads();
  if constexpr (DIM == 3) {
    for (int idx = tid; idx < ne * NV * Q * Q; idx += nth) {
      const int ev = idx / (Q * Q), q10 = idx - ev * Q * Q;
      const int off = (q10 / Q) * RQ + q10 % Q;
      int xh[N], xl[N];
      fix_line<N>(t2 + ev * N * Q * RQ + off, Q * RQ, xh, xl);
      i64* o = (i64*)s0 + ev * VP + off;
#pragma unroll
      for (int q = 0; q < Q; ++q) o[q * Q * RQ] = fix_dot<N>(xh, xl, ft.B + q * N);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------ volume kernel
// EPB elements per block; lines of one direction are one thread's work in the
// contractions, points in the flux.  16^3 P = 3: 270 us with the lift in it
// (680 + 450 us when both ran on the FP64 pipe), FP64 floor 170 us.
template <int DIM, int P, int Q>
__global__ void __launch_bounds__(256, 2) vol_fix_kernel(
    const __grid_constant__ FixTab ft, const __grid_constant__ Phys ph,
    const ElemGeo* __restrict__ geo, int E, const double* __restrict__ u,
    const double* __restrict__ v, const double* __restrict__ epsp,
    const int32_t* __restrict__ eface, const int32_t* __restrict__ faces, int F,
    const double* __restrict__ fflux, const int32_t* __restrict__ fexp,
    const double* __restrict__ force, const double* __restrict__ r_u, double alpha, double beta,
    const double* __restrict__ dscal, double* __restrict__ out, const int EPB) {
  using A = Aff<DIM, P, Q>;
  constexpr int N = A::N, NV = A::NV, NM = A::NM, NQ = A::NQ, NF = A::NF, RQ = A::RQ, VP = A::VP;
  constexpr int N2 = A::N2, LQ = A::LQ;
  extern __shared__ double sm[];
  const int ASZ = EPB * NV * VP;                // one array of the block
  double* s0 = sm;                              // Q; later the partly transformed G
  double* s1 = sm + ASZ;                        // DIM arrays: derivatives, fluxes, G_r
  struct ElFace {
    int f;           // face id
    FixMag c0;       // 2/h_r
    FixScale c1;     // (2/h_r)^2 c beta_s
  };
  static_assert(sizeof(ElFace) <= 32, "vol_bytes");
  ElFace* ef = (ElFace*)(s1 + DIM * ASZ);       // [EPB][2 DIM]
  int* sE = (int*)(ef + EPB * 2 * DIM);         // [EPB][NV] coefficients
  int* sH = sE + EPB * NV;                      // [EPB][NV] fluxes and face data
  int* sZ = sH + EPB * NV;                      // [EPB][NV] bits of the largest |G|
  int* sY = sZ + EPB * NV;                      // [EPB][NV] of A along the last direction
  const int tid = threadIdx.x, nth = blockDim.x;
  const int e0 = blockIdx.x * EPB;
  const int ne = min(EPB, E - e0);
  if (dscal) beta = dscal[1];
  const double eps = v ? epsp[0] : 0.0;
  load_coefficients<DIM, P, Q>(u, v, eps, e0, ne, s1, sE, sZ);
  {
    for (int j = tid; j < ne * 2 * DIM; j += nth) {
      const int eb = j / (2 * DIM), lf = j - eb * 2 * DIM;
      ElFace x;
      x.f = eface[(long long)(e0 + eb) * 2 * DIM + lf];
      const double rh = geo[e0 + eb].rh[lf >> 1];
      x.c0 = fix_mag(rh);
      x.c1 = fix_scale(rh * rh * ph.beta_s * (faces[(long long)x.f * 6 + 2] >= 0 ? 0.5 : 1.0));
      ef[j] = x;
    }
  }
  __syncthreads();
  // the face data's exponents start the maximum of the fluxes'
  for (int j = tid; j < ne * NV; j += nth) {
    const int eb = j / NV, vv = j - eb * NV;
    int m = 0;
#pragma unroll
    for (int lf = 0; lf < 2 * DIM; ++lf) {
      const ElFace& x = ef[eb * 2 * DIM + lf];
      const int32_t* fe = fexp + (long long)x.f * 3 * NV + vv;
      if (fe[0] != 0) m = max(m, min(fe[0] + x.c0.er + ft.elh - ft.eDh, 2047) | (fe[0] == 2047 ? 2047 : 0));
      if (vv > 0 && ph.viscous) {
        if (fe[NV] != 0) m = max(m, min(fe[NV] + x.c0.er + ft.elh - ft.eDh, 2047) | (fe[NV] == 2047 ? 2047 : 0));
        if (fe[2 * NV] != 0)
          m = max(m, min(fe[2 * NV] + x.c1.er + ft.eld - ft.eDh, 2047) | (fe[2 * NV] == 2047 ? 2047 : 0));
      }
    }
    sH[j] = m;
    sY[j] = 0;
  }
  bwd_trans<DIM, P, Q>(ft, s0, s1, ASZ, sE, ne);
  const int seQ = -1022 - 60 + DIM * ft.eB;
  // reference derivatives along every direction, as doubles
  for (int idx = tid; idx < DIM * ne * NV * LQ; idx += nth) {
    const int d = idx / (ne * NV * LQ), rem = idx - d * ne * NV * LQ;
    const int ev = rem / LQ, l = rem - ev * LQ;
    const int a = l % Q, b = l / Q;
    const int off = ev * VP + (d == 0 ? RQ * l : (d == 1 ? a + RQ * Q * b : a + RQ * b));
    const int str = d == 0 ? 1 : (d == 1 ? RQ : RQ * Q);
    int bad, xh[Q], xl[Q];
    const int se = fix_emax(sE[ev], bad) + seQ + ft.eD;
    fix_line<Q>((const i64*)s0 + off, str, xh, xl);
    double* o = s1 + d * ASZ + off;
#pragma unroll
    for (int q = 0; q < Q; ++q) o[q * str] = fix_to_double(fix_dot<Q>(xh, xl, ft.D + q * Q), se, bad);
  }
  __syncthreads();
  // volume flux, in place of the derivatives
  for (int idx = tid; idx < ne * NQ; idx += nth) {
    const int eb = idx / NQ, q = idx - eb * NQ;
    const int off = eb * NV * VP + q + (RQ - Q) * (q / Q);
    double U[NV], dU[DIM][NV], H[DIM][NV], rh[DIM];
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) {
      int bad;
      const int se = fix_emax(sE[eb * NV + vv], bad) + seQ;
      U[vv] = fix_to_double(((const i64*)s0)[off + vv * VP], se, bad);
#pragma unroll
      for (int r = 0; r < DIM; ++r) dU[r][vv] = s1[r * ASZ + off + vv * VP];
    }
#pragma unroll
    for (int r = 0; r < DIM; ++r) rh[r] = geo[e0 + eb].rh[r];
    vol_flux_point<DIM>(U, dU, rh, ph, ph.avf ? ph.avf[e0 + eb] : 0.0, H);
    const KeyGroup grp(eb);
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) {
      int m = 0;
#pragma unroll
      for (int r = 0; r < DIM; ++r) {
        s1[r * ASZ + off + vv * VP] = H[r][vv];
        m = max(m, fix_exp(H[r][vv]));
      }
      grp.max(sH + eb * NV + vv, m);
    }
  }
  __syncthreads();
  // G_r = Dh_r H~_r + lh P0 + ld P1 along every direction; the last direction
  // adds the others and applies A
  const double* gS = fflux + (long long)F * NV * NF;
#pragma unroll
  for (int pass = 0; pass < 2; ++pass) {
    const int nd = pass == 0 ? DIM - 1 : 1;
    for (int idx = tid; idx < nd * ne * NV * LQ; idx += nth) {
      const int dd = idx / (ne * NV * LQ), rem = idx - dd * ne * NV * LQ;
      const int d = pass == 0 ? dd : DIM - 1;
      const int ev = rem / LQ, l = rem - ev * LQ;
      const int eb = ev / NV, vv = ev - eb * NV;
      const int a = l % Q, b = l / Q;
      const int off = ev * VP + (d == 0 ? RQ * l : (d == 1 ? a + RQ * Q * b : a + RQ * b));
      const int str = d == 0 ? 1 : (d == 1 ? RQ : RQ * Q);
      int bad, xh[Q], xl[Q], ph0[2], pl0[2], ph1[2], pl1[2];
      const int em = fix_emax(sH[ev], bad);
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const ElFace& x = ef[eb * 2 * DIM + 2 * d + side];
        // outward flux -f at the lower face, +f at the upper
        const i64 f = to_fix_mul(fflux[((long long)x.f * NV + vv) * NF + l], x.c0,
                                 em - (ft.elh - ft.eDh), 58);
        i64 p0 = side == 0 ? f : -f, p1 = 0;
        if (vv > 0 && ph.viscous) {
          const double* ts = gS + ((long long)x.f * 2 * (NV - 1) + vv - 1) * NF + l;
          p0 += to_fix_mul(ts[0], x.c0, em - (ft.elh - ft.eDh), 58);
          p1 = to_fix_mul(ts[(NV - 1) * NF], x.c1, em - (ft.eld - ft.eDh), 58);
        }
        fix_split(p0, ph0[side], pl0[side]);
        fix_split(p1, ph1[side], pl1[side]);
      }
      double* h = s1 + d * ASZ + off;
#pragma unroll
      for (int k = 0; k < Q; ++k) fix_split(to_fix(h[k * str], em, 58), xh[k], xl[k]);
      u64 used = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        i64 hi = 0, mid = FIX_HALF;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
          const int2 c = ft.Dh[q * Q + k];
          hi += mul_wide(xh[k], c.x);
          mid += mul_wide(xh[k], c.y);
          mid += mul_wide(xl[k], c.x);
        }
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          const int2 c = ft.lh[side][q], e = ft.ld[side][q];
          hi += mul_wide(ph0[side], c.x);
          mid += mul_wide(ph0[side], c.y);
          mid += mul_wide(pl0[side], c.x);
          hi += mul_wide(ph1[side], e.x);
          mid += mul_wide(ph1[side], e.y);
          mid += mul_wide(pl1[side], e.x);
        }
        i64 x = (hi << 2) + (mid >> 30);
        if (pass == 1) {
#pragma unroll
          for (int r = 0; r < DIM - 1; ++r) x += ((const i64*)s1)[r * ASZ + off + q * str];
          used |= (u64)(x ^ (x >> 63));
        }
        ((i64*)h)[q * str] = x;
      }
      if (pass == 1) atomicMax(sZ + ev, 64 - __clzll((i64)used));
    }
    __syncthreads();
  }
  // A = M1^-1 B^T W along the last direction, (the middle one,) and direction 0.
  // G is far below its bound where the volume and the faces cancel, and A's
  // row sums (16 to 32) far above its action, so every stage's input is first
  // shifted up to 60 bits and the last one's result keeps the bits that leaves
  // free; with one scale throughout the result kept 41 bits below the fluxes'
  // largest, and shifting G alone left the weak form's error at 8 times FP64's
  // (4^3 modes on 6^3 points; now at most FP64's).
  for (int j = tid; j < ne * NV; j += nth) sE[j] = 0;
  for (int idx = tid; idx < ne * NV * LQ; idx += nth) {
    const int ev = idx / LQ, l = idx - ev * LQ;
    const int off = DIM == 3 ? l % Q + RQ * (l / Q) : l;
    const int sh = 60 - sZ[ev];
    const i64* g = (const i64*)s1 + (DIM - 1) * ASZ + ev * VP + off;
    constexpr int STR = DIM == 3 ? Q * RQ : RQ;
    int xh[Q], xl[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) fix_split(g[q * STR] << sh, xh[q], xl[q]);
    i64* o = (i64*)s0 + ev * N * STR + off;  // [ev][m_last][...][q0]
    u64 used = 0;
#pragma unroll
    for (int m = 0; m < N; ++m) {
      const i64 x = fix_dot<Q>(xh, xl, ft.A + m * Q);
      used |= (u64)(x ^ (x >> 63));
      o[m * STR] = x;
    }
    atomicMax(sY + ev, 64 - __clzll((i64)used));
  }
  __syncthreads();
  const i64* gl = (const i64*)s0;  // [ev][..][q0] ready for direction 0
  int* sL = sY;                    // its bits
  if constexpr (DIM == 3) {
    i64* t1 = (i64*)s1;            // [ev][n2][n1][q0]
    for (int idx = tid; idx < ne * NV * N * Q; idx += nth) {
      const int en = idx / Q, q0 = idx - en * Q, ev = en / N;
      const int sh = 60 - sY[ev];
      const i64* g = (const i64*)s0 + en * Q * RQ + q0;
      int xh[Q], xl[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) fix_split(g[q * RQ] << sh, xh[q], xl[q]);
      i64* o = t1 + en * N * RQ + q0;
      u64 used = 0;
#pragma unroll
      for (int m = 0; m < N; ++m) {
        const i64 x = fix_dot<Q>(xh, xl, ft.A + m * Q);
        used |= (u64)(x ^ (x >> 63));
        o[m * RQ] = x;
      }
      atomicMax(sE + ev, 64 - __clzll((i64)used));
    }
    __syncthreads();
    gl = t1;
    sL = sE;
  }
  // direction 0 and the epilogue
  const double ie = r_u ? epsp[1] : 0.0;
  for (int idx = tid; idx < ne * NV * N * N2; idx += nth) {
    const int ev = idx / (N * N2);
    int bad, xh[Q], xl[Q];
    const int sh = 60 - sL[ev];
    const int se = fix_emax(sH[ev], bad) - 1022 - 58 + ft.eDh + DIM * ft.eA - (60 - sZ[ev]) - sh - 2 -
                   (DIM == 3 ? 60 - sY[ev] : 0);
#pragma unroll
    for (int q = 0; q < Q; ++q) fix_split(gl[idx * RQ + q] << sh, xh[q], xl[q]);
    const long long gi = (long long)e0 * NV * NM + idx * N;
#pragma unroll
    for (int m = 0; m < N; ++m) {
      double R = fix_to_double(fix_dot<Q, 2>(xh, xl, ft.A + m * Q), se, bad);
      if (force) R += force[gi + m];
      if (r_u) {
        R = (R - r_u[gi + m]) * ie * beta;
        if (alpha != 0.0) R = fma(alpha, v[gi + m], R);
      }
      out[gi + m] = R;
    }
  }
}

// axis-aligned elements; the lift shape of the tuning sets the face kernel's:
// the faces of that many elements (DIM each) per block
template <int DIM, int P, int Q>
dg_status launch_fix(dg_mesh_s* m, const EvalArgs& a, cudaStream_t s) {
  using A = Aff<DIM, P, Q>;
  const int epb = m->tune.vol_epb, fpb = m->tune.lift_epb * DIM;
  const size_t vsm = A::vol_bytes(epb), fsm = A::face_bytes(fpb);
  if (!a.skip_face) {
    DG_CUDA(cudaFuncSetAttribute(face_fix_kernel<DIM, P, Q>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fsm));
    DG_PROF(K_FACE, s, face_fix_kernel<DIM, P, Q>
            <<<(m->F + fpb - 1) / fpb, m->tune.lift_threads, fsm, s>>>(
        m->fix, m->tab, m->phys, m->geo, m->faces, m->F, a.t, a.dscal, a.u, a.v, a.eps, m->fflux,
        m->fexp, fpb));
    DG_LAUNCHED(1);
  }
  if (!a.skip_vol) {
    DG_CUDA(cudaFuncSetAttribute(vol_fix_kernel<DIM, P, Q>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vsm));
    // (the lift family counts the pass too: its work is in this kernel)
    prof_pass(K_LIFT);
    DG_PROF(K_VOL, s, vol_fix_kernel<DIM, P, Q>
            <<<(m->E + epb - 1) / epb, m->tune.vol_threads, vsm, s>>>(
        m->fix, m->phys, m->geo, m->E, a.u, a.v, a.eps, m->eface, m->faces, m->F, m->fflux, m->fexp,
        m->force, a.r_u, a.alpha, a.beta, a.dscal, a.out, epb));
    DG_LAUNCHED(1);
  }
  return DG_OK;
}

}  // namespace dg
