// Dense FP64 vector kernels of the Krylov/Newton layer.  Reductions use a
// fixed grid (RED_BLOCKS blocks, fixed per-block chunks, fixed-shape trees)
// so that every norm and dot product repeats bitwise from run to run.
#include <cooperative_groups.h>
#include "dg_internal.h"

namespace dg {

constexpr int RT = 256;

__device__ __forceinline__ double block_sum(double v, double* sh) {
  sh[threadIdx.x] = v;
  __syncthreads();
#pragma unroll
  for (int s = RT / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  double r = sh[0];
  __syncthreads();
  return r;
}

// ---------------------------------------------------------------- short vectors
// Up to SMALL_N entries one cluster of 8 blocks does a whole reduction or the
// whole Gram-Schmidt tail of an Arnoldi step in one launch: the entries stay in
// registers, warps reduce eight sums at once (9 FP64 additions instead of 40:
// the pipe retires one warp addition per 16 clocks), the blocks' sums meet in
// distributed shared memory in rank order.  On the 8x8 P = 2 vortex (2304
// unknowns) the 9 launches of the tail took about 40 us.  Every k up to the
// largest restart gains up to this n (us per tail in a graph, one cluster / the
// grid-wide kernels: n = 2304 k = 8 16 / 39, k = 30 38 / 100; n = 16,384 k = 8
// 31 / 40, k = 30 94 / 101, k = 64 178 / 182; a dot product 4.1 / 6.0); beyond it
// the cluster's 8 SMs of FP64 fall behind and the entries leave the registers.
namespace cg = cooperative_groups;
constexpr int CL = 8, CT = 256, CR = 8;
constexpr long long SMALL_N = (long long)CL * CT * CR;

// the warp's sums of a[0..7]; lane l with l % 4 == 0 returns that of entry
// sum8_index(l)
__device__ __forceinline__ int sum8_index(int lane) {
  return ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
}
__device__ __forceinline__ double warp_sum8(double* a, int lane) {
#pragma unroll
  for (int o = 16, c = 4; o >= 4; o >>= 1, c >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int j = 0; j < c; ++j) {
      const double give = up ? a[j] : a[j + c];
      a[j] = (up ? a[j + c] : a[j]) + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  double r = a[0];
  r += __shfl_xor_sync(0xffffffffu, r, 2);
  r += __shfl_xor_sync(0xffffffffu, r, 1);
  return r;
}
// the block's sums of a[0..7] into out[0..7] (shared memory; sw: [8 warps][8])
__device__ __forceinline__ void block_sum8(double* a, double (*sw)[8], double* out) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const double r = warp_sum8(a, lane);
  if ((lane & 3) == 0) sw[wp][sum8_index(lane)] = r;
  __syncthreads();
  if (threadIdx.x < 8) {
    double t = 0.0;
#pragma unroll
    for (int k = 0; k < CT / 32; ++k) t += sw[k][threadIdx.x];
    out[threadIdx.x] = t;
  }
  __syncthreads();
}

// two classical Gram-Schmidt passes of w against V_0 .. V_{k-1}, the norm and
// the normalisation: hd[i], hd[ld + i] the passes' coefficients, hd[2 ld] =
// |w|^2 after them; w /= |w| unless that is 0 or not finite
__global__ void __cluster_dims__(CL) __launch_bounds__(CT) orth_cluster_kernel(
    const double* __restrict__ V, int k, double* __restrict__ w, int n, double* __restrict__ hd,
    int ld) {
  __shared__ double sw[CT / 32][8], part[3][MAX_RESTART + 8], h[MAX_RESTART + 8];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), t0 = rank * CT + threadIdx.x;
  double x[CR];
#pragma unroll
  for (int r = 0; r < CR; ++r) {
    const int i = t0 + r * CL * CT;
    x[r] = i < n ? w[i] : 0.0;
  }
  for (int pass = 0; pass < 3; ++pass) {
    const int nv = pass == 2 ? 1 : k;
    for (int i0 = 0; i0 < nv; i0 += 8) {
      double a[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) a[j] = 0.0;
#pragma unroll
      for (int r = 0; r < CR; ++r) {
        const int i = t0 + r * CL * CT;
        if (i < n) {
          if (pass == 2) {
            a[0] = fma(x[r], x[r], a[0]);
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (i0 + j < nv) a[j] = fma(V[(long long)(i0 + j) * n + i], x[r], a[j]);
          }
        }
      }
      block_sum8(a, sw, part[pass] + i0);
    }
    cl.sync();
    for (int i = threadIdx.x; i < nv; i += CT) {
      double s = 0.0;
#pragma unroll
      for (int b = 0; b < CL; ++b) s += cl.map_shared_rank(part[pass], b)[i];
      h[i] = s;
      if (rank == 0) hd[pass * ld + i] = s;
    }
    __syncthreads();
    if (pass == 2) break;
#pragma unroll
    for (int r = 0; r < CR; ++r) {
      const int i = t0 + r * CL * CT;
      if (i < n)
        for (int j = 0; j < k; ++j) x[r] = fma(-h[j], V[(long long)j * n + i], x[r]);
    }
    __syncthreads();  // h is overwritten by the next pass
  }
  if (threadIdx.x == 0) {
    const double nw = sqrt(h[0]);
    h[1] = nw > 0.0 && isfinite(nw) ? 1.0 / nw : 0.0;
  }
  __syncthreads();
  const double sc = h[1];
#pragma unroll
  for (int r = 0; r < CR; ++r) {
    const int i = t0 + r * CL * CT;
    if (i < n) w[i] = sc == 0.0 ? x[r] : fma(sc, x[r], 0.0 * x[r]);
  }
  cl.sync();  // no block leaves while another reads its sums
}

// out[0] = a.b, or with eps the JFNK step from |a|, |b| (eps_finish_kernel)
__global__ void __cluster_dims__(CL) __launch_bounds__(CT) dot_cluster_kernel(
    const double* __restrict__ a, const double* __restrict__ b, int n, int eps,
    double* __restrict__ out) {
  __shared__ double sw[CT / 32][8], part[8];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), t0 = rank * CT + threadIdx.x;
  double s[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) s[j] = 0.0;
#pragma unroll
  for (int r = 0; r < CR; ++r) {
    const int i = t0 + r * CL * CT;
    if (i < n) {
      const double x = a[i], y = b[i];
      if (eps) {
        s[0] = fma(x, x, s[0]);
        s[1] = fma(y, y, s[1]);
      } else {
        s[0] = fma(x, y, s[0]);
      }
    }
  }
  block_sum8(s, sw, part);
  cl.sync();
  if (rank == 0 && threadIdx.x == 0) {
    double p = 0.0, q = 0.0;
#pragma unroll
    for (int r = 0; r < CL; ++r) {
      p += cl.map_shared_rank(part, r)[0];
      q += cl.map_shared_rank(part, r)[1];
    }
    if (!eps) {
      out[0] = p;
    } else {
      const double nu = sqrt(p), nv = sqrt(q);
      const double e = nv > 0.0 ? 1.4901161193847656e-08 * (nu > 0.0 ? nu : 1.0) / nv : 0.0;
      out[0] = e;
      out[1] = e > 0.0 ? 1.0 / e : 0.0;
      out[2] = nu;
      out[3] = nv;
    }
  }
  cl.sync();
}

// partial[b] = sum over chunk b of a*b  (nvec independent pairs at stride)
__global__ void __launch_bounds__(RT) dot_partial_kernel(const double* __restrict__ a,
                                                         const double* __restrict__ b,
                                                         long long n, double* __restrict__ partial) {
  __shared__ double sh[RT];
  const long long chunk = (n + gridDim.x - 1) / gridDim.x;
  const long long lo = blockIdx.x * chunk;
  const long long hi = lo + chunk < n ? lo + chunk : n;
  double s = 0.0;
  for (long long i = lo + threadIdx.x; i < hi; i += RT) s = fma(a[i], b[i], s);
  s = block_sum(s, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void __launch_bounds__(RT) finish_kernel(const double* __restrict__ partial, int np,
                                                    int nsum, double* __restrict__ out) {
  // out[j] = sum_b partial[j*np + b] for j < nsum (one block per j)
  __shared__ double sh[RT];
  const int j = blockIdx.x;
  double s = 0.0;
  for (int i = threadIdx.x; i < np; i += RT) s += partial[(long long)j * np + i];
  s = block_sum(s, sh);
  if (threadIdx.x == 0 && j < nsum) out[j] = s;
}

dg_status dot(const double* a, const double* b, long long n, double* partial, double* out,
              cudaStream_t s) {
  if (n <= SMALL_N) {
    DG_PROF(K_DOT, s, dot_cluster_kernel<<<CL, CT, 0, s>>>(a, b, (int)n, 0, out));
    DG_LAUNCHED(1);
    return DG_OK;
  }
  DG_PROF(K_DOT, s, dot_partial_kernel<<<RED_BLOCKS, RT, 0, s>>>(a, b, n, partial));
  DG_PROF(K_DOT, s, finish_kernel<<<1, RT, 0, s>>>(partial, RED_BLOCKS, 1, out));
  DG_LAUNCHED(2);
  return DG_OK;
}

dg_status finish_sum(const double* partial, int np, double* out, cudaStream_t s) {
  finish_kernel<<<1, RT, 0, s>>>(partial, np, 1, out);
  DG_LAUNCHED(1);
  return DG_OK;
}

// partial[i*RED_BLOCKS + b] = chunk-b part of V_i . w for i in [8*blockIdx.y, +8)
__global__ void __launch_bounds__(RT) multi_dot_kernel(const double* __restrict__ V, int k,
                                                       const double* __restrict__ w, long long n,
                                                       double* __restrict__ partial) {
  __shared__ double sh[RT];
  const long long chunk = (n + gridDim.x - 1) / gridDim.x;
  const long long lo = blockIdx.x * chunk;
  const long long hi = lo + chunk < n ? lo + chunk : n;
  const int i0 = blockIdx.y * 8;
  double acc[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] = 0.0;
  for (long long x = lo + threadIdx.x; x < hi; x += RT) {
    const double wx = w[x];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (i0 + j < k) acc[j] = fma(V[(long long)(i0 + j) * n + x], wx, acc[j]);
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const double s = block_sum(acc[j], sh);
    if (threadIdx.x == 0 && i0 + j < k) partial[(long long)(i0 + j) * gridDim.x + blockIdx.x] = s;
  }
}

dg_status multi_dot(const double* V, int k, const double* w, long long n, double* partial,
                    double* out, cudaStream_t s) {
  dim3 grid(RED_BLOCKS, (k + 7) / 8);
  DG_PROF(K_MULTIDOT, s, multi_dot_kernel<<<grid, RT, 0, s>>>(V, k, w, n, partial));
  DG_PROF(K_MULTIDOT, s, finish_kernel<<<k, RT, 0, s>>>(partial, RED_BLOCKS, k, out));
  DG_LAUNCHED(2);
  return DG_OK;
}

// w -= sum_i h_i V_i
__global__ void multi_axpy_kernel(double* __restrict__ w, const double* __restrict__ V, int k,
                                  const double* __restrict__ h, long long n) {
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n;
       x += (long long)gridDim.x * blockDim.x) {
    double acc = w[x];
    for (int i = 0; i < k; ++i) acc = fma(-h[i], V[(long long)i * n + x], acc);
    w[x] = acc;
  }
}

static int grid_for(long long n) {
  long long g = (n + 255) / 256;
  return (int)(g < 152 * 16 ? g : 152 * 16);
}

dg_status multi_axpy(double* w, const double* V, int k, const double* h, long long n,
                     cudaStream_t s) {
  DG_PROF(K_MULTIAXPY, s, multi_axpy_kernel<<<grid_for(n), 256, 0, s>>>(w, V, k, h, n));
  DG_LAUNCHED(1);
  return DG_OK;
}

// y = a x + b y; with b = 0, y is output only and is not read (a fresh
// buffer may hold anything, and 0 * NaN is NaN).  x may be y (scaling in
// place), hence no __restrict__.
__global__ void axpby_kernel(double* y, double a, const double* x, double b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    y[i] = b == 0.0 ? a * x[i] : fma(a, x[i], b * y[i]);
}
dg_status axpby(double* y, double a, const double* x, double b, long long n, cudaStream_t s) {
  DG_PROF(K_VEC, s, axpby_kernel<<<grid_for(n), 256, 0, s>>>(y, a, x, b, n));
  DG_LAUNCHED(1);
  return DG_OK;
}

__global__ void lincomb_kernel(double* __restrict__ y, const double* __restrict__ x, double a,
                               const double* __restrict__ z, double b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    y[i] = fma(a, x[i], b * z[i]);
}
dg_status lincomb(double* y, const double* x, double a, const double* z, double b, long long n,
                  cudaStream_t s) {
  DG_PROF(K_VEC, s, lincomb_kernel<<<grid_for(n), 256, 0, s>>>(y, x, a, z, b, n));
  DG_LAUNCHED(1);
  return DG_OK;
}

// y = x * s or x / s with s a device scalar (the reciprocal formed once per
// block: an FP64 division per thread would cost more than the stream)
__global__ void scale_dev_kernel(double* __restrict__ y, const double* __restrict__ x,
                                 const double* __restrict__ sdev, int inv, long long n) {
  __shared__ double ss;
  if (threadIdx.x == 0) ss = inv ? 1.0 / sdev[0] : sdev[0];
  __syncthreads();
  const double s = ss;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    y[i] = x[i] * s;
}
dg_status scale_dev(double* y, const double* x, const double* sdev, int inv, long long n,
                    cudaStream_t s) {
  scale_dev_kernel<<<grid_for(n), 256, 0, s>>>(y, x, sdev, inv, n);
  DG_LAUNCHED(1);
  return DG_OK;
}

// eps = sqrt(2^-52) ||u|| / ||v|| (sqrt(2^-52)/||v|| when u = 0); eps = 0 when v = 0
__global__ void eps_finish_kernel(const double* __restrict__ partial, double* __restrict__ eps) {
  __shared__ double sh[RT];
  double su = 0.0, sv = 0.0;
  for (int i = threadIdx.x; i < RED_BLOCKS; i += RT) {
    su += partial[i];
    sv += partial[RED_BLOCKS + i];
  }
  su = block_sum(su, sh);
  sv = block_sum(sv, sh);
  if (threadIdx.x == 0) {
    const double nu = sqrt(su), nv = sqrt(sv);
    const double e = nv > 0.0 ? 1.4901161193847656e-08 * (nu > 0.0 ? nu : 1.0) / nv : 0.0;
    eps[0] = e;
    eps[1] = e > 0.0 ? 1.0 / e : 0.0;
    eps[2] = nu;
    eps[3] = nv;
  }
}

dg_status jvp_eps(const double* u, const double* v, long long n, double* partial, double* eps,
                  cudaStream_t s) {
  if (n <= SMALL_N) {
    DG_PROF(K_DOT, s, dot_cluster_kernel<<<CL, CT, 0, s>>>(u, v, (int)n, 1, eps));
    DG_LAUNCHED(1);
    return DG_OK;
  }
  DG_PROF(K_DOT, s, dot_partial_kernel<<<RED_BLOCKS, RT, 0, s>>>(u, u, n, partial));
  DG_PROF(K_DOT, s, dot_partial_kernel<<<RED_BLOCKS, RT, 0, s>>>(v, v, n, partial + RED_BLOCKS));
  DG_PROF(K_DOT, s, eps_finish_kernel<<<1, RT, 0, s>>>(partial, eps));
  DG_LAUNCHED(3);
  return DG_OK;
}

// Nneg = S + dta R - u  (= -N(u) of Eq. nonlinear-equation-system)
__global__ void newton_resid_kernel(double* __restrict__ Nn, const double* __restrict__ u,
                                    const double* __restrict__ S, const double* __restrict__ R,
                                    double dta, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    Nn[i] = fma(dta, R[i], S[i]) - u[i];
}
dg_status newton_resid(double* N, const double* u, const double* S, const double* R, double dta,
                       long long n, cudaStream_t s) {
  DG_PROF(K_VEC, s, newton_resid_kernel<<<grid_for(n), 256, 0, s>>>(N, u, S, R, dta, n));
  DG_LAUNCHED(1);
  return DG_OK;
}

__global__ void set_scalars_kernel(double* __restrict__ d, double a, double b) {
  d[0] = a;
  d[1] = b;
}
dg_status set_scalars(double* d, double a, double b, cudaStream_t s) {
  DG_PROF(K_VEC, s, set_scalars_kernel<<<1, 1, 0, s>>>(d, a, b));
  DG_LAUNCHED(1);
  return DG_OK;
}

// the Arnoldi normalisation with the norm read on the device: h = sqrt(*hsq),
// w = (1/h) w + 0 w as axpby_kernel forms it, skipped when h is 0 or not finite
__global__ void normalize_dev_kernel(double* __restrict__ w, const double* __restrict__ hsq,
                                     long long n) {
  __shared__ double sa;  // 1/h once per block (FP64 sqrt and division are long sequences)
  if (threadIdx.x == 0) {
    const double h = sqrt(hsq[0]);
    sa = (h > 0.0 && isfinite(h)) ? 1.0 / h : 0.0;
  }
  __syncthreads();
  const double a = sa;
  if (a == 0.0) return;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    w[i] = fma(a, w[i], 0.0 * w[i]);
}
dg_status normalize_dev(double* w, const double* hsq, long long n, cudaStream_t s) {
  DG_PROF(K_VEC, s, normalize_dev_kernel<<<grid_for(n), 256, 0, s>>>(w, hsq, n));
  DG_LAUNCHED(1);
  return DG_OK;
}

// The Gram-Schmidt tail of an Arnoldi step: w against V_0 .. V_{k-1} twice, the
// coefficients in hd[0..k) and hd[ld..ld+k), |w|^2 in hd[2 ld], w normalised.
// Every solver takes it, so that they agree bit for bit.
dg_status orthonormalise(double* w, const double* V, int k, long long n, double* partial,
                         double* hd, int ld, cudaStream_t s) {
  if (n <= SMALL_N) {
    DG_PROF(K_MULTIDOT, s, orth_cluster_kernel<<<CL, CT, 0, s>>>(V, k, w, (int)n, hd, ld));
    DG_LAUNCHED(1);
    return DG_OK;
  }
  DG_TRY(multi_dot(V, k, w, n, partial, hd, s));
  DG_TRY(multi_axpy(w, V, k, hd, n, s));
  DG_TRY(multi_dot(V, k, w, n, partial, hd + ld, s));
  DG_TRY(multi_axpy(w, V, k, hd + ld, n, s));
  DG_TRY(dot(w, w, n, partial, hd + 2 * ld, s));
  return normalize_dev(w, hd + 2 * ld, n, s);
}

}  // namespace dg
