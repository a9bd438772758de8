// The residual on general elements (curved, rotated or sheared) in two
// kernels built like the axis-aligned ones (dg_affine.cuh): contractions and
// here also the products with the metric in 64-bit fixed point, FP64 for the
// pointwise fluxes.  With g[r][j] = d xi_r / d x_j, J = |dx/dxi|, w the Gauss
// weights and J_f the surface Jacobian:
//   R = M_e^-1 (B^T W)^(x)d G,
//   G = sum_r Dh_r (J sum_j g_rj H_j) + sum_faces lh P0 + ld P1,
//   P0 = -+ J_f H^n + sum_t Dh_t T_t,  P1 = T_r  (r normal, t tangential),
//   T_r = c beta_s J_f sum_j g_rj S_j  with each side's own metric,
// the dense M_e^-1 applied in fixed point too (its entries are converted where
// they are used: each serves every variable).  The bubble modes' integrals are
// small and their columns of M_e^-1 large, so mode k enters scaled up by
// 2^a_k, its column scaled down, and each row has an exponent of its own;
// with one exponent for all, 20 of the 60 bits were lost.
#pragma once
#include "dg_affine.cuh"

namespace dg {

struct FaceInfoGen {
  int eA, fA, eB, fB;  // owner and neighbour (-1: none) and their local faces
  int bc;              // boundary type (0: interior)
  FixScale cb;         // c beta_s
  __device__ __forceinline__ void side(int s, int& e, int& lf) const {
    e = s == 0 ? eA : eB;
    lf = s == 0 ? fA : fB;
  }
};
static_assert(sizeof(FaceInfoGen) <= 64, "face_bytes");

// Roe flux along the unit normal n
template <int D>
__device__ __forceinline__ void roe_flux_normal(const double* UL, const double* UR, const double* n,
                                                const Phys& ph, double* Fh) {
  const double rsL = rsqrt(UL[0]), rsR = rsqrt(UR[0]);
  const double iL = rsL * rsL, iR = rsR * rsR;
  const double sL = UL[0] * rsL, sR = UR[0] * rsR;
  double vL[D], vR[D], keL = 0.0, keR = 0.0, unL = 0.0, unR = 0.0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    vL[k] = UL[1 + k] * iL;
    vR[k] = UR[1 + k] * iR;
    keL = fma(UL[1 + k], vL[k], keL);
    keR = fma(UR[1 + k], vR[k], keR);
    unL = fma(vL[k], n[k], unL);
    unR = fma(vR[k], n[k], unR);
  }
  const double pL = ph.gm1 * fma(-0.5, keL, UL[D + 1]), pR = ph.gm1 * fma(-0.5, keR, UR[D + 1]);
  const double EL = UL[D + 1] + pL, ER = UR[D + 1] + pR;
  const double isum = 1.0 / (sL + sR), wL = sL * isum, wR = sR * isum;
  double ut[D], du[D], q2 = 0.0, udu = 0.0, unt = 0.0, dun = 0.0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    ut[k] = fma(wL, vL[k], wR * vR[k]);
    du[k] = vR[k] - vL[k];
    q2 = fma(ut[k], ut[k], q2);
    udu = fma(ut[k], du[k], udu);
    unt = fma(ut[k], n[k], unt);
    dun = fma(du[k], n[k], dun);
  }
  const double Ht = fma(rsL, EL, rsR * ER) * isum;
  const double c2 = ph.gm1 * fma(-0.5, q2, Ht);
  const double rc = rsqrt(c2), c = c2 * rc, ic2 = rc * rc;
  const double dp = pR - pL, rt = sL * sR, hic2 = 0.5 * ic2, rcd = rt * c * dun;
  const double a2 = fma(-dp, ic2, UR[0] - UL[0]), l2 = fabs(unt);
  const double w1 = fabs(unt - c) * ((dp - rcd) * hic2), w5 = fabs(unt + c) * ((dp + rcd) * hic2);
  const double w2 = l2 * a2, ws = l2 * rt, w15 = w1 + w5, wc = (w5 - w1) * c, wt = w15 + w2;
  Fh[0] = 0.5 * (fma(UL[0], unL, UR[0] * unR) - wt);
  const double pn = (pL + pR) - wc + ws * dun;  // along n: pressure and acoustic parts
#pragma unroll
  for (int k = 0; k < D; ++k) {
    double f = fma(UL[1 + k], unL, UR[1 + k] * unR);
    f = fma(-wt, ut[k], f);
    f = fma(-ws, du[k], f);
    Fh[1 + k] = 0.5 * fma(pn, n[k], f);
  }
  double f = fma(EL, unL, ER * unR);
  f = fma(-w15, Ht, f);
  f = fma(-wc, unt, f);
  f = fma(-0.5 * w2, q2, f);
  Fh[D + 1] = 0.5 * fma(-ws, fma(-unt, dun, udu), f);
}

template <int D>
__device__ __noinline__ void other_flux_normal(const double* UL, const double* UR, const double* n,
                                               const Phys& ph, double* Fh) {
  riemann_flux<D>(UL, UR, n, ph, Fh);
}
template <int D>
__device__ __noinline__ bool boundary_normal(int bctype, const Phys& ph, const double* x, double t,
                                             const double* U, const double* n, double* QR,
                                             double* QB) {
  return boundary_states<D>(bctype, ph, x, t, U, n, QR, QB);
}

// ------------------------------------------------------------ face kernel
template <int DIM, int P, int Q>
__global__ void __launch_bounds__(256, 2) face_gen_kernel(
    const __grid_constant__ FixTab ft, const __grid_constant__ Phys ph,
    const __grid_constant__ GenGeo gg, const int32_t* __restrict__ faces, int F, double t,
    const double* __restrict__ dscal, const double* __restrict__ u, const double* __restrict__ v,
    const double* __restrict__ epsp, double* __restrict__ fflux, int32_t* __restrict__ fexp,
    const int FPB) {
  using A = Gen<DIM, P, Q>;
  constexpr int N = A::N, NV = A::NV, NM = A::NM, NF = A::NF, NT = A::NT, RQ = A::RQ;
  constexpr int NL = NF / Q;
  extern __shared__ double sm[];
  double* sX = sm;                                  // [FPB][GX]
  double* sY = sX + FPB * A::GX;                    // [FPB][GY]
  FaceInfoGen* info = (FaceInfoGen*)(sY + FPB * A::GY);
  int* sE = (int*)(info + FPB);                     // [FPB][2][NV] coefficients
  int* sF = sE + FPB * 2 * NV;                      // [FPB][NV] H^n
  int* sS = sF + FPB * NV;                          // [FPB][NV] S_i
  int* sT = sS + FPB * NV;                          // [FPB][2][2][NV] lifted parts of both sides
  int* sM = sT + FPB * 4 * NV;                      // [FPB][2] metrics times c beta_s J_f
  const int f0 = blockIdx.x * FPB;
  const int nf = min(FPB, F - f0);
  const int tid = threadIdx.x, nth = blockDim.x;
  if (dscal) t = dscal[0];
  for (int i = tid; i < FPB * (8 * NV + 2); i += nth) sE[i] = 0;
  for (int i = tid; i < nf; i += nth) {
    const int32_t* fp = faces + (long long)(f0 + i) * 6;
    FaceInfoGen g;
    g.eA = fp[0];
    g.fA = fp[1];
    g.eB = fp[2];
    g.fB = fp[3];
    g.bc = g.eB >= 0 ? 0 : ph.bc[fp[5]];
    g.cb = fix_scale((g.eB >= 0 ? 0.5 : 1.0) * ph.beta_s);
    info[i] = g;
  }
  __syncthreads();
  {
    const double eps = v ? epsp[0] : 0.0;
    const int lane = tid & 31, nw = nth >> 5;
    for (int j = tid >> 5; j < nf * 2 * NV; j += nw) {
      const int fb = j / (2 * NV), sv = j - fb * 2 * NV, side = sv / NV, vv = sv - side * NV;
      const int e = side == 0 ? info[fb].eA : info[fb].eB;
      if (e < 0) continue;  // warp-uniform
      const long long g = ((long long)e * NV + vv) * NM;
      double* dst = sX + fb * A::GX + sv * NM;
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
  // per side: the face's coefficients and those of the normal derivative
  i64* C0 = (i64*)sY;  // [2 side][2][NV][NT]
  bool far = false;
  for (int idx = tid; idx < nf * 2 * NV * NT; idx += nth) {
    const int fb = idx / (2 * NV * NT), rem = idx - fb * 2 * NV * NT;
    const int sv = rem / NT, l = rem - sv * NT, side = sv / NV, vv = sv - side * NV;
    const FaceInfoGen& g = info[fb];
    if (side == 1 && g.eB < 0) continue;
    const int lf = side == 0 ? g.fA : g.fB, r = lf >> 1;
    const int sn = r == 0 ? 1 : (r == 1 ? N : N * N);
    const int s0 = r == 0 ? N : 1, s1 = r == 2 ? N : N * N;
    const double* src = sX + fb * A::GX + sv * NM +
                        (DIM == 3 ? (l % N) * s0 + (l / N) * s1 : l * s0);
    int bad, xh[N], xl[N];
    const int eA = sE[(fb * 2) * NV + vv], eB = sE[(fb * 2 + 1) * NV + vv];
    const int em = fix_emax(max(eA, eB), bad);
    far |= g.bc == 0 && far_below(min(eA, eB), max(eA, eB));
    i64 first = 0, last = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const i64 x = to_fix(src[k * sn], em, 59);
      if (k == 0) first = x;
      if (k == P) last = x;
      fix_split(x, xh[k], xl[k]);
    }
    i64* o = C0 + fb * A::GY + (side * 2 * NV + vv) * NT + l;
    o[0] = (lf & 1) ? last : first;
    o[NV * NT] = (lf & 1) ? fix_dot<N>(xh, xl, ft.dp[1]) : fix_dot<N>(xh, xl, ft.dp[0]);
  }
  const bool apart = __syncthreads_or(far);
  // 3-D, first tangential direction: per side B and DB on the values, B on the
  // normal derivative
  i64* C1 = (i64*)sX;  // [2 side][3][NV][N][RQ]
  if constexpr (DIM == 3) {
    for (int idx = tid; idx < 6 * nf * NV * N; idx += nth) {
      const int kind = idx / (nf * NV * N), rem = idx - kind * nf * NV * N;
      const int fb = rem / (NV * N), vn = rem - fb * NV * N;
      const int side = kind / 3, kk = kind - 3 * side;
      if (side == 1 && info[fb].eB < 0) continue;
      int xh[N], xl[N];
      fix_line<N>(C0 + fb * A::GY + (side * 2 + (kk == 2)) * NV * NT + vn * N, 1, xh, xl);
      i64* o = C1 + fb * A::GX + (kind * NV * N + vn) * RQ;
      if (kk == 1) {
#pragma unroll
        for (int q = 0; q < Q; ++q) o[q] = fix_dot<N>(xh, xl, ft.DB + q * N);
      } else {
#pragma unroll
        for (int q = 0; q < Q; ++q) o[q] = fix_dot<N>(xh, xl, ft.B + q * N);
      }
    }
    __syncthreads();
  }
  // last tangential direction: fields [NFLD][NV][NF], the values as doubles,
  // the derivatives as integers of one scale: 0, 1 values; 2 + DIM side + (0
  // normal, 1.. tangential)
  const int eT = max(ft.edp + ft.eB, ft.eDB) + (DIM == 3 ? ft.eB : 0);
  for (int idx = tid; idx < A::NFLD * nf * NV * NL; idx += nth) {
    const int kind = idx / (nf * NV * NL), rem = idx - kind * nf * NV * NL;
    const int fb = rem / (NV * NL), vq = rem - fb * NV * NL;
    const int vv = vq / NL, q0 = vq - vv * NL;
    const int side = kind < 2 ? kind : (kind - 2) / DIM, d = kind < 2 ? -1 : (kind - 2) % DIM;
    if (side == 1 && info[fb].eB < 0) continue;
    int xh[N], xl[N];
    const bool db = d == DIM - 1;  // the derivative along this direction
    int sh;
    if constexpr (DIM == 3) {
      const int kk = d == 0 ? 2 : (d == 1 ? 1 : 0);
      fix_line<N>(C1 + fb * A::GX + ((side * 3 + kk) * NV + vv) * N * RQ + q0, RQ, xh, xl);
      sh = eT - (d == 0 ? ft.edp + 2 * ft.eB : ft.eDB + ft.eB);
    } else {
      fix_line<N>(C0 + fb * A::GY + ((side * 2 + (d == 0)) * NV + vv) * NT, 1, xh, xl);
      sh = eT - (d == 0 ? ft.edp + ft.eB : ft.eDB);
    }
    i64 y[Q];
    if (db) {
#pragma unroll
      for (int q = 0; q < Q; ++q) y[q] = fix_dot<N>(xh, xl, ft.DB + q * N);
    } else {
#pragma unroll
      for (int q = 0; q < Q; ++q) y[q] = fix_dot<N>(xh, xl, ft.B + q * N);
    }
    double* o = (DIM == 3 ? sY + fb * A::GY : sX + fb * A::GX) + (kind * NV + vv) * NF + q0;
    if (kind < 2) {
      int bad;
      const int se = fix_emax(max(sE[(fb * 2) * NV + vv], sE[(fb * 2 + 1) * NV + vv]), bad) - 1022 -
                     59 + (DIM - 1) * ft.eB;
#pragma unroll
      for (int q = 0; q < Q; ++q) o[q * NL] = fix_to_double(y[q], se, bad);
    } else {
#pragma unroll
      for (int q = 0; q < Q; ++q) ((i64*)o)[q * NL] = fix_shift(y[q], sh);
    }
  }
  double* sP = DIM == 3 ? sY : sX;
  constexpr int PS = DIM == 3 ? A::GY : A::GX;
  __syncthreads();
  if (apart)
    own_values<DIM, P, Q>(ft, info, sE, nf, u, v, v ? epsp[0] : 0.0, sP, PS);
  double* gS = fflux + (long long)F * NV * NF;  // [E][2 DIM][2][NV-1][NF]
  for (int idx = tid; idx < nf * NF; idx += nth) {
    const int fb = idx / NF, p = idx - fb * NF;
    const FaceInfoGen& g = info[fb];
    const int f = f0 + fb;
    const bool interior = g.eB >= 0;
    const KeyGroup grp(fb);
    double* pt = sP + fb * PS + p;
    const double* fd = gg.fdat + (long long)f * (2 * DIM + 1) * NF + p;
    // face-average gradient: metrics as integers of the point's largest
    // exponent, both sides' products in one sum
    double dQ[DIM][NV];
    const double Jf = fd[DIM * NF] * ft.iw[p % Q] * (DIM == 3 ? ft.iw[p / Q] : 1.0);
    const FixMag sJ = fix_mag(Jf);
    {
      const double* gA = gg.fgeo + ((long long)g.eA * 2 * DIM + g.fA) * DIM * DIM * NF + p;
      const double* gB = interior ? gg.fgeo + ((long long)g.eB * 2 * DIM + g.fB) * DIM * DIM * NF + p : gA;
      int eg = 0, egB = 0;
#pragma unroll
      for (int i = 0; i < DIM * DIM; ++i) eg = max(eg, fix_exp(gA[i * NF]));
      if (ph.viscous) grp.max(sM + fb * 2, eg + sJ.er + g.cb.er);
      if (interior) {
#pragma unroll
        for (int i = 0; i < DIM * DIM; ++i) egB = max(egB, fix_exp(gB[i * NF]));
        if (ph.viscous) grp.max(sM + fb * 2 + 1, egB + sJ.er + g.cb.er);
      }
      int gbad;
      eg = fix_emax(max(eg, egB), gbad);
      i64 acc[DIM][NV];
#pragma unroll
      for (int j = 0; j < DIM; ++j)
#pragma unroll
        for (int vv = 0; vv < NV; ++vv) acc[j][vv] = 0;
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        if (side == 1 && !interior) break;
        const int r = (side == 0 ? g.fA : g.fB) >> 1;
        const int ax[3] = {r, r == 0 ? 1 : 0, r == 2 ? 1 : 2};  // normal, tangential
        const double* gp = side == 0 ? gA : gB;
        int ch[DIM][DIM], cl[DIM][DIM];
#pragma unroll
        for (int a = 0; a < DIM; ++a)
#pragma unroll
          for (int j = 0; j < DIM; ++j)
            fix_split(to_fix(gp[(ax[a] * DIM + j) * NF], eg, 59), ch[a][j], cl[a][j]);
#pragma unroll
        for (int vv = 0; vv < NV; ++vv) {
          int xh[DIM], xl[DIM];
#pragma unroll
          for (int a = 0; a < DIM; ++a)
            fix_split(((const i64*)pt)[((2 + DIM * side + a) * NV + vv) * NF], xh[a], xl[a]);
#pragma unroll
          for (int j = 0; j < DIM; ++j) {
            i64 hi = 0, mid = FIX_HALF;
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
              hi += mul_wide(xh[a], ch[a][j]);
              mid += mul_wide(xh[a], cl[a][j]);
              mid += mul_wide(xl[a], ch[a][j]);
            }
            acc[j][vv] += (hi << 2) + (mid >> 30);
          }
        }
      }
#pragma unroll
      for (int vv = 0; vv < NV; ++vv) {
        int bad;
        const int em = fix_emax(max(sE[(fb * 2) * NV + vv], sE[(fb * 2 + 1) * NV + vv]), bad);
        const int se = em - 1022 - 59 + eT + 62 + eg - 1022 - 59 - (interior ? 1 : 0);
#pragma unroll
        for (int j = 0; j < DIM; ++j) dQ[j][vv] = fix_to_double(acc[j][vv], se, bad | gbad);
      }
    }
    double n[DIM], UA[NV], UB[NV], Qa[NV], jump[NV], Fh[NV];
#pragma unroll
    for (int j = 0; j < DIM; ++j) n[j] = fd[j * NF];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      UA[k] = pt[k * NF];
      UB[k] = interior ? pt[(NV + k) * NF] : UA[k];
    }
    double mua = 0.0;
    if (ph.avf) mua = av_face<DIM>(ph, g.eA, g.eB, UA, UB, dQ);
    bool adiabatic = false;
    if (!interior) {
      double x[3] = {0, 0, 0};
#pragma unroll
      for (int j = 0; j < DIM; ++j) x[j] = fd[(DIM + 1 + j) * NF];
      adiabatic = boundary_normal<DIM>(g.bc, ph, x, t, UA, n, UB, Qa);
#pragma unroll
      for (int k = 0; k < NV; ++k) jump[k] = UA[k] - Qa[k];
    } else {
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        Qa[k] = 0.5 * (UA[k] + UB[k]);
        jump[k] = UA[k] - UB[k];
      }
    }
    if (ph.riemann == DG_RIEMANN_ROE)
      roe_flux_normal<DIM>(UA, UB, n, ph, Fh);
    else
      other_flux_normal<DIM>(UA, UB, n, ph, Fh);
    if (ph.viscous) {
      const double irho = 1.0 / Qa[0];
      double vel[DIM];
#pragma unroll
      for (int k = 0; k < DIM; ++k) vel[k] = Qa[1 + k] * irho;
      const double e = Qa[NV - 1] * irho;
      double mu = ph.mu;
      if (ph.mu_law != 0) {
        double q2 = 0.0;
#pragma unroll
        for (int k = 0; k < DIM; ++k) q2 = fma(vel[k], vel[k], q2);
        mu = viscosity(ph.gMa2 * ph.gm1 * fma(-0.5, q2, e), ph);
      }
      mu += mua;
      const double mi = mu * irho, ck = ph.gMa2 * ph.gm1 * ph.kappa_fac;
      // S_i = G_i({Q}, n (x) jump): stresses a_i n_k + n_i a_k - 2/3 delta_ik a.n
      double a[DIM], an = 0.0, va = 0.0, vn = 0.0, s = fma(-e, jump[0], jump[NV - 1]);
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        const double tk = fma(-vel[k], jump[0], jump[1 + k]);
        s = fma(-tk, vel[k], s);
        a[k] = mi * tk;
        an = fma(a[k], n[k], an);
        va = fma(a[k], vel[k], va);
        vn = fma(n[k], vel[k], vn);
      }
      const double hq = fma(ck * mi, s, va), tt = (2.0 / 3.0) * an;
      // row n of G({Q}, {grad Q})
      double gdn[DIM], gnd[DIM], div = 0.0, dn0 = 0.0, dnE = 0.0;
#pragma unroll
      for (int k = 0; k < DIM; ++k) gdn[k] = gnd[k] = 0.0;
#pragma unroll
      for (int j = 0; j < DIM; ++j) {
        dn0 = fma(n[j], dQ[j][0], dn0);
        dnE = fma(n[j], dQ[j][NV - 1], dnE);
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
          const double tk = fma(-vel[k], dQ[j][0], dQ[j][1 + k]);  // rho d u_k / d x_j
          gdn[k] = fma(n[j], tk, gdn[k]);
          gnd[j] = fma(n[k], tk, gnd[j]);
          if (j == k) div += tk;
        }
      }
      const double beta = gg.fbeta[f], t23 = (2.0 / 3.0) * div;
      double sg = fma(-e, dn0, dnE), eg = 0.0;
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        sg = fma(-gdn[k], vel[k], sg);
        const double tau = mi * fma(-t23, n[k], gdn[k] + gnd[k]);
        eg = fma(vel[k], tau, eg);
        // n.S along x_k: a_k + (a.n) n_k / 3
        Fh[1 + k] += fma(beta, fma((1.0 / 3.0) * an, n[k], a[k]), -tau);
      }
      eg = fma(ck * mi, sg, eg);
      if (!adiabatic) Fh[NV - 1] += fma(beta, fma((1.0 / 3.0) * an, vn, hq), -eg);
      // S_i into fields 0 .. DIM-1 of this point (density component zero)
      int big[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) big[k] = 0;
#pragma unroll
      for (int i = 0; i < DIM; ++i) {
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
          double x = fma(a[i], n[k], n[i] * a[k]);
          if (i == k) x -= tt;
          pt[(i * NV + 1 + k) * NF] = x;
          big[1 + k] = max(big[1 + k], fix_exp(x));
        }
        const double x = adiabatic ? 0.0 : fma(n[i], hq, fma(a[i], vn, -tt * vel[i]));
        pt[(i * NV + NV - 1) * NF] = x;
        big[NV - 1] = max(big[NV - 1], fix_exp(x));
      }
#pragma unroll
      for (int k = 1; k < NV; ++k) grp.max(sS + fb * NV + k, big[k]);
    }
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const double x = Fh[k] * Jf;
      fflux[((long long)f * NV + k) * NF + p] = x;
      grp.max(sF + fb * NV + k, fix_exp(x));
    }
  }
  __syncthreads();
  if (ph.viscous) {
    // T_r of both sides: P1 (r normal) to memory, the tangential ones as
    // integers into fields DIM + side (DIM - 1) + t
    constexpr int NTT = DIM - 1;
    for (int idx = tid; idx < nf * NF; idx += nth) {
      const int fb = idx / NF, p = idx - fb * NF;
      const FaceInfoGen& g = info[fb];
      double* pt = sP + fb * PS + p;
      const double Jf = gg.fdat[((long long)(f0 + fb) * (2 * DIM + 1) + DIM) * NF + p] *
                        ft.iw[p % Q] * (DIM == 3 ? ft.iw[p / Q] : 1.0);
      FixScale sJ = fix_scale(Jf);
      {  // times c beta_s: the mantissas' product is in (2^60, 2^62)
        i64 m = fix_mul((i64)(((u64)(unsigned)sJ.h << 32) + (i64)sJ.l), g.cb.h, g.cb.l);
        fix_split(m, sJ.h, sJ.l);
        sJ.er += g.cb.er;
        sJ.sg ^= g.cb.sg;
      }
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const int e = side == 0 ? g.eA : g.eB, lf = side == 0 ? g.fA : g.fB;
        if (e < 0) continue;
        const int r = lf >> 1;
        const int ax[3] = {r, r == 0 ? 1 : 0, r == 2 ? 1 : 2};
        const double* gp = gg.fgeo + ((long long)e * 2 * DIM + lf) * DIM * DIM * NF + p;
        int gbad;
        const int em = fix_emax(sM[fb * 2 + side], gbad);
        int ch[DIM][DIM], cl[DIM][DIM];
#pragma unroll
        for (int a = 0; a < DIM; ++a)
#pragma unroll
          for (int j = 0; j < DIM; ++j)
            fix_split(to_fix_mul(gp[(ax[a] * DIM + j) * NF], sJ, em, 60), ch[a][j], cl[a][j]);
#pragma unroll
        for (int vv = 1; vv < NV; ++vv) {
          int bad, xh[DIM], xl[DIM];
          const int es = fix_emax(sS[fb * NV + vv], bad);
#pragma unroll
          for (int j = 0; j < DIM; ++j) fix_split(to_fix(pt[(j * NV + vv) * NF], es, 60), xh[j], xl[j]);
#pragma unroll
          for (int a = 0; a < DIM; ++a) {
            i64 hi = 0, mid = FIX_HALF;
#pragma unroll
            for (int j = 0; j < DIM; ++j) {
              hi += mul_wide(xh[j], ch[a][j]);
              mid += mul_wide(xh[j], cl[a][j]);
              mid += mul_wide(xl[j], ch[a][j]);
            }
            const i64 y = (hi << 2) + (mid >> 30);
            if (a == 0) {
              const double x = fix_to_double(y, em + es - 2044 - 58, bad | gbad);
              gS[((((long long)e * 2 * DIM + lf) * 2 + 1) * (NV - 1) + vv - 1) * NF + p] = x;
              KeyGroup(fb).max(sT + ((fb * 2 + side) * 2 + 1) * NV + vv, fix_exp(x));
            } else {
              ((i64*)pt)[((DIM + side * NTT + a - 1) * NV + vv) * NF] = y;
            }
          }
        }
      }
    }
    __syncthreads();
    if constexpr (DIM == 3) {
      for (int idx = tid; idx < nf * 2 * (NV - 1) * Q; idx += nth) {
        const int fb = idx / (2 * (NV - 1) * Q), rem = idx - fb * 2 * (NV - 1) * Q;
        const int side = rem / ((NV - 1) * Q), rv = rem - side * (NV - 1) * Q;
        const int vv = 1 + rv / Q, q1 = rv % Q;
        if (side == 1 && info[fb].eB < 0) continue;
        int xh[Q], xl[Q];
        i64* d = (i64*)sP + fb * PS + ((DIM + side * NTT) * NV + vv) * NF + q1 * Q;
        fix_line<Q>(d, 1, xh, xl);
#pragma unroll
        for (int q = 0; q < Q; ++q) d[q] = fix_dot<Q>(xh, xl, ft.Dh + q * Q);
      }
      __syncthreads();
    }
    for (int idx = tid; idx < nf * 2 * (NV - 1) * NL; idx += nth) {
      const int fb = idx / (2 * (NV - 1) * NL), rem = idx - fb * 2 * (NV - 1) * NL;
      const int side = rem / ((NV - 1) * NL), rv = rem - side * (NV - 1) * NL;
      const int vv = 1 + rv / NL, q0 = rv % NL;
      const FaceInfoGen& g = info[fb];
      const int e = side == 0 ? g.eA : g.eB, lf = side == 0 ? g.fA : g.fB;
      if (e < 0) continue;
      int bad, gbad, xh[Q], xl[Q];
      const int se = fix_emax(sM[fb * 2 + side], gbad) + fix_emax(sS[fb * NV + vv], bad) - 2044 - 58 +
                     ft.eDh;
      const i64* d = (const i64*)sP + fb * PS + ((DIM + side * NTT + NTT - 1) * NV + vv) * NF + q0;
      const i64* d0 = (const i64*)sP + fb * PS + ((DIM + side * NTT) * NV + vv) * NF + q0;
      fix_line<Q>(d, NL, xh, xl);
      double* o = gS + (((long long)e * 2 * DIM + lf) * 2 * (NV - 1) + vv - 1) * NF + q0;
      int big = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        i64 x = fix_dot<Q>(xh, xl, ft.Dh + q * Q);
        if (DIM == 3) x += d0[q * NL];
        const double val = fix_to_double(x, se, bad | gbad);
        o[q * NL] = val;
        big = max(big, fix_exp(val));
      }
      KeyGroup((fb * 2 + side) * NV + vv).max(sT + (fb * 2 + side) * 2 * NV + vv, big);
    }
    __syncthreads();
  }
  for (int i = tid; i < nf * NV; i += nth) fexp[(long long)f0 * NV + i] = sF[i];
  for (int i = tid; i < nf * 4 * NV; i += nth) {
    const int fb = i / (4 * NV), rem = i - fb * 4 * NV, side = rem / (2 * NV);
    const int e = side == 0 ? info[fb].eA : info[fb].eB, lf = side == 0 ? info[fb].fA : info[fb].fB;
    if (e >= 0) fexp[(long long)F * NV + ((long long)e * 2 * DIM + lf) * 2 * NV + rem - side * 2 * NV] = sT[i];
  }
}

// a_k of mode k: the sum of its directions' scales
template <int DIM, int N>
__device__ __forceinline__ int mode_scale(const FixTab& ft, int k) {
  return ft.aw[k % N] + ft.aw[(k / N) % N] + (DIM == 3 ? ft.aw[k / (N * N)] : 0);
}

// ------------------------------------------------------------ volume kernel
template <int DIM, int P, int Q>
__global__ void __launch_bounds__(256, 2) vol_gen_kernel(
    const __grid_constant__ FixTab ft, const __grid_constant__ Phys ph,
    const __grid_constant__ GenGeo gg, const int32_t* __restrict__ eminv, int E,
    const double* __restrict__ u, const double* __restrict__ v, const double* __restrict__ epsp,
    const int32_t* __restrict__ eface, const int32_t* __restrict__ faces, int F,
    const double* __restrict__ fflux, const int32_t* __restrict__ fexp,
    const double* __restrict__ force, const double* __restrict__ r_u, double alpha, double beta,
    const double* __restrict__ dscal, double* __restrict__ out, const int EPB) {
  using A = Gen<DIM, P, Q>;
  constexpr int N = A::N, NV = A::NV, NM = A::NM, NQ = A::NQ, NF = A::NF, RQ = A::RQ, VP = A::VP;
  constexpr int N2 = A::N2, LQ = A::LQ;
  extern __shared__ double sm[];
  const int ASZ = EPB * NV * VP;
  double* s0 = sm;
  double* s1 = sm + ASZ;
  int* ef = (int*)(s1 + DIM * ASZ);   // [EPB][2 DIM] face id; -1 - id where not the owner
  int* sE = ef + EPB * 2 * DIM;       // [EPB][NV] coefficients
  int* sF = sE + EPB * NV;            // [EPB][NV] face data, as exponents of G's terms
  int* sH = sF + EPB * NV;            // [EPB][NV] fluxes
  int* sZ = sH + EPB * NV;            // [EPB][NV] bits of the largest |G|
  int* sG = sZ + EPB * NV;            // [EPB] metrics times J
  int* sA = sG + EPB;                 // [NM] a_k
  const int tid = threadIdx.x, nth = blockDim.x;
  const int e0 = blockIdx.x * EPB;
  const int ne = min(EPB, E - e0);
  if (dscal) beta = dscal[1];
  load_coefficients<DIM, P, Q>(u, v, v ? epsp[0] : 0.0, e0, ne, s1, sE, sZ);
  for (int j = tid; j < ne * 2 * DIM; j += nth) {
    const int f = eface[(long long)e0 * 2 * DIM + j];
    const int32_t* fp = faces + (long long)f * 6;
    ef[j] = fp[0] == e0 + j / (2 * DIM) && fp[1] == j % (2 * DIM) ? f : -1 - f;
  }
  for (int j = tid; j < ne * NV; j += nth) sH[j] = 0;
  for (int j = tid; j < ne; j += nth) sG[j] = 0;
  for (int j = tid; j < NM; j += nth) sA[j] = mode_scale<DIM, N>(ft, j);
  __syncthreads();
  const int32_t* fxs = fexp + (long long)F * NV;  // [E][2 DIM][2][NV]
  for (int j = tid; j < ne * NV; j += nth) {
    const int eb = j / NV, vv = j - eb * NV;
    int m = 0;
#pragma unroll
    for (int lf = 0; lf < 2 * DIM; ++lf) {
      const int i = ef[eb * 2 * DIM + lf], f = i >= 0 ? i : -1 - i;
      auto add = [&](int e, int by) {
        if (e != 0) m = max(m, e == 2047 ? 4095 : e + by);
      };
      add(fexp[(long long)f * NV + vv], ft.elh - ft.eDh);
      if (vv > 0 && ph.viscous) {
        const int32_t* x = fxs + ((long long)(e0 + eb) * 2 * DIM + lf) * 2 * NV + vv;
        add(x[0], ft.elh - ft.eDh);
        add(x[NV], ft.eld - ft.eDh);
      }
    }
    sF[j] = m;
  }
  bwd_trans<DIM, P, Q>(ft, s0, s1, ASZ, sE, ne);
  const int seQ = -1022 - 60 + DIM * ft.eB;
  // reference derivatives along every direction, as integers
  for (int idx = tid; idx < DIM * ne * NV * LQ; idx += nth) {
    const int d = idx / (ne * NV * LQ), rem = idx - d * ne * NV * LQ;
    const int ev = rem / LQ, l = rem - ev * LQ;
    const int a = l % Q, b = l / Q;
    const int off = ev * VP + (d == 0 ? RQ * l : (d == 1 ? a + RQ * Q * b : a + RQ * b));
    const int str = d == 0 ? 1 : (d == 1 ? RQ : RQ * Q);
    int xh[Q], xl[Q];
    fix_line<Q>((const i64*)s0 + off, str, xh, xl);
    i64* o = (i64*)s1 + d * ASZ + off;
#pragma unroll
    for (int q = 0; q < Q; ++q) o[q * str] = fix_dot<Q>(xh, xl, ft.D + q * Q);
  }
  __syncthreads();
  // physical gradients (metrics as integers of the point's largest exponent)
  // and volume flux, in place of the derivatives
  for (int idx = tid; idx < ne * NQ; idx += nth) {
    const int eb = idx / NQ, q = idx - eb * NQ;
    const int off = eb * NV * VP + q + (RQ - Q) * (q / Q);
    const double* gp = gg.vgeo + (long long)(e0 + eb) * (DIM * DIM + 1) * NQ + q;
    double U[NV], dU[DIM][NV], H[DIM][NV];
    const KeyGroup grp(eb);
    {
      int eg = 0, gbad, ch[DIM][DIM], cl[DIM][DIM];
      double g[DIM][DIM];
#pragma unroll
      for (int r = 0; r < DIM; ++r)
#pragma unroll
        for (int j = 0; j < DIM; ++j) {
          g[r][j] = gp[(r * DIM + j) * NQ];
          eg = max(eg, fix_exp(g[r][j]));
        }
      // J up to its weights: the exponent bound of J g
      const int qx = q % Q, qy = (q / Q) % Q, qz = q / (Q * Q);
      const double J = gp[DIM * DIM * NQ] * ft.iw[qx] * ft.iw[qy] * (DIM == 3 ? ft.iw[qz] : 1.0);
      grp.max(sG + eb, eg + fix_exp(J) - 1022);
      eg = fix_emax(eg, gbad);
#pragma unroll
      for (int r = 0; r < DIM; ++r)
#pragma unroll
        for (int j = 0; j < DIM; ++j) fix_split(to_fix(g[r][j], eg, 60), ch[r][j], cl[r][j]);
#pragma unroll
      for (int vv = 0; vv < NV; ++vv) {
        int bad, xh[DIM], xl[DIM];
        const int se = fix_emax(sE[eb * NV + vv], bad) + seQ;
        U[vv] = fix_to_double(((const i64*)s0)[off + vv * VP], se, bad);
#pragma unroll
        for (int r = 0; r < DIM; ++r)
          fix_split(((const i64*)s1)[r * ASZ + off + vv * VP], xh[r], xl[r]);
#pragma unroll
        for (int j = 0; j < DIM; ++j) {
          i64 hi = 0, mid = FIX_HALF;
#pragma unroll
          for (int r = 0; r < DIM; ++r) {
            hi += mul_wide(xh[r], ch[r][j]);
            mid += mul_wide(xh[r], cl[r][j]);
            mid += mul_wide(xl[r], ch[r][j]);
          }
          dU[j][vv] = fix_to_double((hi << 2) + (mid >> 30), se + ft.eD + 62 + eg - 1022 - 60, bad | gbad);
        }
      }
    }
    double one[DIM];
#pragma unroll
    for (int r = 0; r < DIM; ++r) one[r] = 1.0;
    vol_flux_point<DIM>(U, dU, one, ph, ph.avf ? ph.avf[e0 + eb] : 0.0, H);
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
  // contravariant fluxes J sum_j g_rj H_j as integers of G's scale: the larger
  // of theirs and the face data's exponents
  auto g_exp = [&](int ev, int& bad) {
    int b0, b1, b2;
    const int em = fix_emax(sH[ev], b0) + fix_emax(sG[ev / NV], b1) - 1020;
    const int m = fix_emax(max(em, sF[ev]), b2);
    bad = b0 | b1 | b2;
    return m;
  };
  for (int idx = tid; idx < ne * NQ; idx += nth) {
    const int eb = idx / NQ, q = idx - eb * NQ;
    const int off = eb * NV * VP + q + (RQ - Q) * (q / Q);
    const double* gp = gg.vgeo + (long long)(e0 + eb) * (DIM * DIM + 1) * NQ + q;
    const int qx = q % Q, qy = (q / Q) % Q, qz = q / (Q * Q);
    const FixMag sJ =
        fix_mag(gp[DIM * DIM * NQ] * ft.iw[qx] * ft.iw[qy] * (DIM == 3 ? ft.iw[qz] : 1.0));
    int gbad, ch[DIM][DIM], cl[DIM][DIM];
    const int eg = fix_emax(sG[eb], gbad);
#pragma unroll
    for (int r = 0; r < DIM; ++r)
#pragma unroll
      for (int j = 0; j < DIM; ++j)
        fix_split(to_fix_mul(gp[(r * DIM + j) * NQ], sJ, eg, 60), ch[r][j], cl[r][j]);
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) {
      int b0, bad, xh[DIM], xl[DIM];
      const int eh = fix_emax(sH[eb * NV + vv], b0);
      const int sh = g_exp(eb * NV + vv, bad) - (eh + eg - 1020);
#pragma unroll
      for (int j = 0; j < DIM; ++j) fix_split(to_fix(s1[j * ASZ + off + vv * VP], eh, 58), xh[j], xl[j]);
#pragma unroll
      for (int r = 0; r < DIM; ++r) {
        i64 hi = 0, mid = FIX_HALF;
#pragma unroll
        for (int j = 0; j < DIM; ++j) {
          hi += mul_wide(xh[j], ch[r][j]);
          mid += mul_wide(xh[j], cl[r][j]);
          mid += mul_wide(xl[j], ch[r][j]);
        }
        ((i64*)s1)[r * ASZ + off + vv * VP] =
            fix_shift((hi << 2) + (mid >> 30), sh);
      }
    }
  }
  __syncthreads();
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
      const int em = g_exp(ev, bad);
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const int lf = 2 * d + side, i = ef[eb * 2 * DIM + lf], f = i >= 0 ? i : -1 - i;
        // the owner's outward flux is H^n, the neighbour's -H^n
        const i64 fx = to_fix(fflux[((long long)f * NV + vv) * NF + l], em - (ft.elh - ft.eDh), 58);
        i64 p0 = i >= 0 ? -fx : fx, p1 = 0;
        if (vv > 0 && ph.viscous) {
          const double* ts = gS + (((long long)(e0 + eb) * 2 * DIM + lf) * 2 * (NV - 1) + vv - 1) * NF + l;
          p0 += to_fix(ts[0], em - (ft.elh - ft.eDh), 58);
          p1 = to_fix(ts[(NV - 1) * NF], em - (ft.eld - ft.eDh), 58);
        }
        fix_split(p0, ph0[side], pl0[side]);
        fix_split(p1, ph1[side], pl1[side]);
      }
      i64* h = (i64*)s1 + d * ASZ + off;
      fix_line<Q>(h, str, xh, xl);
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
        h[q * str] = x;
      }
      if (pass == 1) atomicMax(sZ + ev, 64 - __clzll((i64)used));
    }
    __syncthreads();
  }
  // B^T W along the last direction, (the middle one,) and direction 0, whose
  // results' bits go to sE
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
    i64* o = (i64*)s0 + ev * N * STR + off;
#pragma unroll
    for (int m = 0; m < N; ++m) o[m * STR] = fix_dot<Q>(xh, xl, ft.BW + m * Q);
  }
  __syncthreads();
  const i64* gl = (const i64*)s0;
  if constexpr (DIM == 3) {
    i64* t1 = (i64*)s1;
    for (int idx = tid; idx < ne * NV * N * Q; idx += nth) {
      const int en = idx / Q, q0 = idx - en * Q;
      int xh[Q], xl[Q];
      fix_line<Q>((const i64*)s0 + en * Q * RQ + q0, RQ, xh, xl);
      i64* o = t1 + en * N * RQ + q0;
#pragma unroll
      for (int m = 0; m < N; ++m) o[m * RQ] = fix_dot<Q>(xh, xl, ft.BW + m * Q);
    }
    __syncthreads();
    gl = t1;
  }
  int2* sL = (int2*)(s1 + (DIM - 1) * ASZ);  // [ev][NM] halves of L
  for (int idx = tid; idx < ne * NV * N * N2; idx += nth) {
    int xh[Q], xl[Q];
    fix_line<Q>(gl + idx * RQ, 1, xh, xl);
    u64 used = 0;
#pragma unroll
    for (int m = 0; m < N; ++m) {
      int2 h;
      const i64 x = fix_dot<Q>(xh, xl, ft.BW + m * Q);
      used |= (u64)(x ^ (x >> 63));
      fix_split(x, h.x, h.y);
      sL[idx * N + m] = h;
    }
    atomicMax(sE + idx / (N * N2), 64 - __clzll((i64)used));
  }
  __syncthreads();
  // M_e^-1: a thread per (element, mode, part of the sum), every variable; the
  // parts meet in s0
  {
    constexpr int PARTS = NM >= 64 || DIM == 2 && NM >= 16 ? 2 : 4;
    constexpr int KP = (NM + PARTS - 1) / PARTS;
    static_assert(PARTS * NM <= A::VP * DIM, "the parts end before sL");
    i64* y0 = (i64*)s0;  // [ne][PARTS][NV][NM], over s0 and the arrays before sL
    for (int idx = tid; idx < ne * NM * PARTS; idx += nth) {
      const int eb = idx / (NM * PARTS), rem = idx - eb * NM * PARTS;
      const int part = rem / NM, m = rem - part * NM;
      const double* Mi = gg.minv + (long long)(e0 + eb) * NM * NM + m;
      const int em = eminv[(long long)(e0 + eb) * NM + m] + 1022;
      // rows cancel by 2^12 and more, so the sums keep every bit (the low
      // halves' product too, and the middle accumulator's remainder from one
      // group of four terms to the next) and the result as many below its
      // unit as |L| leaves free
      i64 y[NV], mid[NV];
      int sh[NV];
#pragma unroll
      for (int vv = 0; vv < NV; ++vv) {
        sh[vv] = min(62 - sE[eb * NV + vv], 28);
        y[vv] = 0;
        mid[vv] = FIX_HALF >> sh[vv];
      }
      const int k1 = min(NM, (part + 1) * KP);
      for (int k0 = part * KP; k0 < k1; k0 += 4) {
        i64 hi[NV];
#pragma unroll
        for (int vv = 0; vv < NV; ++vv) hi[vv] = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int k = k0 + i;
          if (k < k1) {
            int ch, cl;
            fix_split(to_fix(Mi[(long long)k * NM], em + sA[k], 62), ch, cl);  // M^-1 is symmetric
#pragma unroll
            for (int vv = 0; vv < NV; ++vv) {
              const int2 x = sL[(eb * NV + vv) * NM + k];
              hi[vv] += mul_wide(x.x, ch);
              mid[vv] += mul_wide(x.x, cl);
              mid[vv] += mul_wide(x.y, ch);
              mid[vv] += (i64)__mulhi(x.y, cl);
            }
          }
        }
#pragma unroll
        for (int vv = 0; vv < NV; ++vv) {
          y[vv] += (hi[vv] << (2 + sh[vv])) + (mid[vv] >> (30 - sh[vv]));
          mid[vv] &= (1ll << (30 - sh[vv])) - 1;
        }
      }
#pragma unroll
      for (int vv = 0; vv < NV; ++vv) y0[((eb * PARTS + part) * NV + vv) * NM + m] = y[vv];
    }
    __syncthreads();
    const double ie = r_u ? epsp[1] : 0.0;
    for (int idx = tid; idx < ne * NV * NM; idx += nth) {
      const int ev = idx / NM, eb = ev / NV, vm = idx - eb * NV * NM;
      int bad;
      const int se = g_exp(ev, bad) - 1022 - 58 + ft.eDh - (60 - sZ[ev]) - min(62 - sE[ev], 28) +
                     eminv[(long long)(e0 + eb) * NM + idx % NM];
      i64 y = 0;
#pragma unroll
      for (int part = 0; part < PARTS; ++part) y += y0[(eb * PARTS + part) * NV * NM + vm];
      double R = fix_to_double(y, se, bad);
      const long long gi = (long long)e0 * NV * NM + idx;
      if (force) R += force[gi];
      if (r_u) {
        R = (R - r_u[gi]) * ie * beta;
        if (alpha != 0.0) R = fma(alpha, v[gi], R);
      }
      out[gi] = R;
    }
  }
}

// exponents of the row sums of each element's M^-1 (symmetric), column k scaled
// by 2^-a_k
template <int DIM, int N>
__global__ void __launch_bounds__(128) minv_exp_kernel(const __grid_constant__ FixTab ft,
                                                       const double* __restrict__ minv,
                                                       int32_t* __restrict__ eminv) {
  constexpr int NM = DIM == 3 ? N * N * N : N * N;
  const long long e = blockIdx.x;
  for (int m = threadIdx.x; m < NM; m += 128) {
    double s = 0.0;
    for (int k = 0; k < NM; ++k)
      s += ldexp(fabs(minv[(e * NM + k) * NM + m]), -mode_scale<DIM, N>(ft, k));
    eminv[e * NM + m] = ilogb(s) + 1;
  }
}

// the exponents of M^-1, when the mesh is created
template <int DIM, int P, int Q>
dg_status launch_minv_exp(dg_mesh_s* m, cudaStream_t s) {
  minv_exp_kernel<DIM, P + 1><<<m->E, 128, 0, s>>>(m->fix, m->minv, m->eminv);
  DG_LAUNCHED(1);
  return DG_OK;
}

template <int DIM, int P, int Q>
dg_status launch_gen(dg_mesh_s* m, const EvalArgs& a, cudaStream_t s) {
  using A = Gen<DIM, P, Q>;
  const int epb = m->tune.vol_epb, fpb = m->tune.lift_epb * DIM;
  const size_t vsm = A::vol_bytes(epb), fsm = A::face_bytes(fpb);
  const GenGeo gg = gen_geo(m);
  if (!a.skip_face) {
    DG_CUDA(cudaFuncSetAttribute(face_gen_kernel<DIM, P, Q>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fsm));
    DG_PROF(K_FACE, s, face_gen_kernel<DIM, P, Q>
            <<<(m->F + fpb - 1) / fpb, m->tune.lift_threads, fsm, s>>>(
        m->fix, m->phys, gg, m->faces, m->F, a.t, a.dscal, a.u, a.v, a.eps, m->fflux, m->fexp, fpb));
    DG_LAUNCHED(1);
  }
  if (!a.skip_vol) {
    DG_CUDA(cudaFuncSetAttribute(vol_gen_kernel<DIM, P, Q>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vsm));
    prof_pass(K_LIFT);  // (as on axis-aligned elements)
    DG_PROF(K_VOL, s, vol_gen_kernel<DIM, P, Q>
            <<<(m->E + epb - 1) / epb, m->tune.vol_threads, vsm, s>>>(
        m->fix, m->phys, gg, m->eminv, m->E, a.u, a.v, a.eps, m->eface, m->faces, m->F, m->fflux,
        m->fexp, m->force, a.r_u, a.alpha, a.beta, a.dscal, a.out, epb));
    DG_LAUNCHED(1);
  }
  return DG_OK;
}

}  // namespace dg
