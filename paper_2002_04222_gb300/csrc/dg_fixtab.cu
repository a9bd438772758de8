// Host construction of the fixed-point 1-D tables (FixTab), in long double so
// that each entry is right to its 62 bits: Gauss-Legendre points by Newton's
// method on P_Q, the modified basis by polynomial coefficients, the
// collocation derivative and the end values in barycentric form, the mass
// matrix by elimination.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>
#include "dg_internal.h"

namespace dg {
namespace {

typedef long double ld;
constexpr ld LD_PI = 3.141592653589793238462643383279502884L;

ld poly_at(const std::vector<ld>& c, ld x) {
  ld s = 0;
  for (size_t i = c.size(); i-- > 0;) s = s * x + c[i];
  return s;
}
std::vector<ld> poly_diff(const std::vector<ld>& c) {
  std::vector<ld> d;
  for (size_t i = 1; i < c.size(); ++i) d.push_back((ld)i * c[i]);
  if (d.empty()) d.push_back(0);
  return d;
}
std::vector<ld> poly_mul(const std::vector<ld>& a, const std::vector<ld>& b) {
  std::vector<ld> r(a.size() + b.size() - 1, 0);
  for (size_t i = 0; i < a.size(); ++i)
    for (size_t j = 0; j < b.size(); ++j) r[i + j] += a[i] * b[j];
  return r;
}

// the modified basis psi_0..psi_P as polynomials (Jacobi P^(1,1) by recurrence)
std::vector<std::vector<ld>> modified_polys(int P) {
  std::vector<std::vector<ld>> jac = {{1}, {0, 2}};
  for (int k = 1; k < P; ++k) {
    const ld a1 = 2.0L * (k + 1) * (k + 3) * (2 * k + 2), a3 = (2.0L * k + 2) * (2 * k + 3) * (2 * k + 4),
             a4 = 2.0L * (k + 1) * (k + 1) * (2 * k + 4);
    std::vector<ld> p = poly_mul({0, a3}, jac[k]);
    for (size_t i = 0; i < jac[k - 1].size(); ++i) p[i] -= a4 * jac[k - 1][i];
    for (ld& c : p) c /= a1;
    jac.push_back(p);
  }
  std::vector<std::vector<ld>> b = {{0.5L, -0.5L}};
  for (int p = 1; p < P; ++p) b.push_back(poly_mul({0.25L, 0, -0.25L}, jac[p - 1]));
  b.push_back({0.5L, 0.5L});
  return b;
}

// entries of `rows` x `cols` values as halves of c 2^(62 - e)
void store(const ld* c, int rows, int cols, int e, int2* out) {
  for (int i = 0; i < rows * cols; ++i) {
    const long long C = (long long)std::llround(std::ldexp(c[i], 62 - e));
    const int lo = (int)(unsigned)(unsigned long long)C;
    out[i] = make_int2((int)((C - lo) >> 32), lo);
  }
}
// smallest e with every row's sum of magnitudes <= 2^e
int row_exponent(const ld* c, int rows, int cols) {
  ld big = 0;
  for (int r = 0; r < rows; ++r) {
    ld s = 0;
    for (int k = 0; k < cols; ++k) s += std::fabs(c[r * cols + k]);
    big = std::max(big, s);
  }
  // (a sum that is a power of two up to rounding, like psi_0 + psi_P = 1, counts as it)
  return (int)std::ceil(std::log2(big) - 1e-12L);
}

}  // namespace

void build_fix_tables(int P, int Q, FixTab& f) {
  std::memset(&f, 0, sizeof(f));
  const int N = P + 1;
  std::vector<ld> x(Q), w(Q), bw(Q);
  for (int i = 0; i < Q; ++i) {
    ld z = -std::cos(LD_PI * (i + 0.75L) / (Q + 0.5L)), d = 1;
    for (int it = 0; it < 8; ++it) {  // (quadratic from two digits: six suffice)
      ld p0 = 1, p1 = z;
      for (int k = 2; k <= Q; ++k) {
        const ld p2 = ((2 * k - 1) * z * p1 - (k - 1) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      d = Q * (z * p1 - p0) / (z * z - 1);
      z -= p1 / d;
    }
    x[i] = z;
    w[i] = 2 / ((1 - z * z) * d * d);
  }
  const auto psi = modified_polys(P);
  std::vector<ld> B(Q * N), DB(Q * N), D(Q * Q), Dh(Q * Q), A(N * Q), BW(N * Q), lh(2 * Q), le(2 * Q), dp(2 * N);
  for (int k = 0; k < N; ++k) {
    const auto d = poly_diff(psi[k]);
    for (int q = 0; q < Q; ++q) {
      B[q * N + k] = poly_at(psi[k], x[q]);
      DB[q * N + k] = poly_at(d, x[q]);
    }
    dp[k] = poly_at(d, -1);
    dp[N + k] = poly_at(d, 1);
  }
  for (int k = 0; k < Q; ++k) {
    ld p = 1;
    for (int j = 0; j < Q; ++j)
      if (j != k) p *= x[k] - x[j];
    bw[k] = 1 / p;
  }
  for (int i = 0; i < Q; ++i) {
    ld diag = 0;
    for (int k = 0; k < Q; ++k) {
      if (k == i) continue;
      D[i * Q + k] = bw[k] / bw[i] / (x[i] - x[k]);
      diag -= D[i * Q + k];
    }
    D[i * Q + i] = diag;
  }
  for (int s = 0; s < 2; ++s) {
    const ld z = s ? 1 : -1;
    for (int k = 0; k < Q; ++k) {
      ld p = 1;
      for (int j = 0; j < Q; ++j)
        if (j != k) p *= (z - x[j]) / (x[k] - x[j]);
      lh[s * Q + k] = p;
    }
    // l_q'(z) = sum_k l_k(z) D[k][q]
    for (int q = 0; q < Q; ++q) {
      ld d = 0;
      for (int k = 0; k < Q; ++k) d += lh[s * Q + k] * D[k * Q + q];
      le[s * Q + q] = d / w[q];
    }
    for (int k = 0; k < Q; ++k) lh[s * Q + k] /= w[k];
  }
  for (int q = 0; q < Q; ++q)
    for (int k = 0; k < Q; ++k) Dh[q * Q + k] = D[k * Q + q] * w[k] / w[q];
  // M1 A = B^T W by Gauss-Jordan elimination with partial pivoting
  const int C = N + Q;
  std::vector<ld> M(N * C, 0);
  for (int a = 0; a < N; ++a) {
    for (int q = 0; q < Q; ++q) {
      M[a * C + N + q] = B[q * N + a] * w[q];
      for (int b = 0; b < N; ++b) M[a * C + b] += B[q * N + a] * w[q] * B[q * N + b];
    }
  }
  for (int c = 0; c < N; ++c) {
    int piv = c;
    for (int r = c + 1; r < N; ++r)
      if (std::fabs(M[r * C + c]) > std::fabs(M[piv * C + c])) piv = r;
    for (int k = 0; k < C; ++k) std::swap(M[c * C + k], M[piv * C + k]);
    const ld d = M[c * C + c];
    for (int k = 0; k < C; ++k) M[c * C + k] /= d;
    for (int r = 0; r < N; ++r) {
      const ld m = r == c ? 0 : M[r * C + c];
      for (int k = 0; k < C; ++k) M[r * C + k] -= m * M[c * C + k];
    }
  }
  for (int a = 0; a < N; ++a)
    for (int q = 0; q < Q; ++q) {
      A[a * Q + q] = M[a * C + N + q];
      BW[a * Q + q] = B[q * N + a] * w[q];
    }
  for (int q = 0; q < Q; ++q) f.iw[q] = (double)(1 / w[q]);
  auto ends = [&](const std::vector<ld>& v) {  // largest |v(-1)| + |v(+1)| over the points
    ld big = 0;
    for (int q = 0; q < Q; ++q) big = std::max(big, std::fabs(v[q]) + std::fabs(v[Q + q]));
    return (int)std::ceil(std::log2(big));
  };
  f.eB = row_exponent(B.data(), Q, N);
  f.eDB = row_exponent(DB.data(), Q, N);
  f.eD = row_exponent(D.data(), Q, Q);
  f.eDh = row_exponent(Dh.data(), Q, Q) + 1;
  f.eA = row_exponent(A.data(), N, Q);
  f.elh = ends(lh) + 2;
  f.eld = ends(le) + 2;
  f.edp = row_exponent(dp.data(), 2, N);
  store(B.data(), Q, N, f.eB, f.B);
  store(DB.data(), Q, N, f.eDB, f.DB);
  store(D.data(), Q, Q, f.eD, f.D);
  store(Dh.data(), Q, Q, f.eDh, f.Dh);
  store(A.data(), N, Q, f.eA, f.A);
  for (int a = 0; a < N; ++a) {
    f.aw[a] = -row_exponent(&BW[a * Q], 1, Q);
    store(&BW[a * Q], 1, Q, -f.aw[a], f.BW + a * Q);
  }
  for (int s = 0; s < 2; ++s) {
    store(&lh[s * Q], 1, Q, f.elh, f.lh[s]);
    store(&le[s * Q], 1, Q, f.eld, f.ld[s]);
    store(&dp[s * N], 1, N, f.edp, f.dp[s]);
  }
}

}  // namespace dg
