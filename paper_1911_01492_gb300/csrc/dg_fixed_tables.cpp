// Host construction of the fixed-point 1D tables (dg_fixed.cuh) for n Gauss
// points, from Legendre polynomials in extended precision (at least 64
// mantissa bits on both x86 and Arm), rounded to 60 binary places.
//
// With q[a][i] = sqrt(w_a) L_i(xi_a) (orthogonal, since the n-point Gauss rule
// integrates L_i L_j exactly) the scaled point values u = q x give
//   value at 0:            sum_a l_a u_a,  l_a = sum_i L_i(0) q[a][i],
//   half derivative at 0:  sum_a d_a u_a,  d_a = sum_i L_i'(0) q[a][i] / 2,
//   scaled derivative at point f: sum_a Dh[f][a] u_a,
//                          Dh[f][a] = sqrt(w_f) sum_i L_i'(xi_f) q[a][i];
// at 1: l_{n-1-a} and -d_{n-1-a}.
#include <cmath>
#include <cstring>

#include "dg_internal.cuh"

namespace {

typedef long double ld;

FxPair pair_of(ld t) {  // t 2^60 = h 2^30 + l
  const long long v = (long long)llrintl(ldexpl(t, 60));
  const long long h = (v + (1ll << 29)) >> 30;
  return {(int)h, (int)(v - (h << 30))};
}

int ceil_log2(ld v) {  // smallest e with v <= 2^e
  int e;
  const ld m = frexpl(v, &e);
  return m == 0.5L ? e - 1 : e;
}

}  // namespace

bool dg_build_fixed_tables(int n, double h, DGTabX* t, DGTabXSetup* s, DGTabXGrad* g) {
  std::memset(t, 0, sizeof(*t));
  std::memset(s, 0, sizeof(*s));
  std::memset(g, 0, sizeof(*g));
  ld xi[DG_MAXN], w[DG_MAXN];
  // Legendre values and derivatives on [-1, 1], degrees 0..n
  auto legendre = [n](ld x, ld* P, ld* dP) {
    P[0] = 1;
    dP[0] = 0;
    P[1] = x;
    dP[1] = 1;
    for (int j = 1; j < n; ++j) {
      P[j + 1] = ((2 * j + 1) * x * P[j] - j * P[j - 1]) / (j + 1);
      dP[j + 1] = dP[j - 1] + (2 * j + 1) * P[j];
    }
  };
  ld P[DG_MAXN + 1], dP[DG_MAXN + 1];
  for (int a = 0; a < n; ++a) {
    if (2 * a + 1 > n) break;
    ld x = -std::cos(3.14159265358979323846 * (a + 0.75) / (n + 0.5));
    for (int it = 0; it < 12; ++it) {
      legendre(x, P, dP);
      x -= P[n] / dP[n];
    }
    if (2 * a + 1 == n) x = 0;
    legendre(x, P, dP);
    xi[a] = x;
    xi[n - 1 - a] = -x;
    w[a] = w[n - 1 - a] = 1 / ((1 - x * x) * dP[n] * dP[n]);  // weight on [0, 1]
  }
  ld q[DG_MAXN][DG_MAXN], dq[DG_MAXN][DG_MAXN], E0[DG_MAXN], D0[DG_MAXN];
  for (int a = 0; a <= n; ++a) {  // a = n: the end point 0
    legendre(a < n ? xi[a] : -1.0L, P, dP);
    for (int i = 0; i < n; ++i) {
      const ld c = sqrtl(2.0L * i + 1);
      if (a < n) {
        q[a][i] = sqrtl(w[a]) * c * P[i];
        dq[a][i] = sqrtl(w[a]) * 2 * c * dP[i];
      } else {
        E0[i] = c * P[i];
        D0[i] = 2 * c * dP[i];
      }
    }
  }
  ld l[DG_MAXN], d[DG_MAXN], Dh[DG_MAXN][DG_MAXN];
  for (int a = 0; a < n; ++a) {
    l[a] = d[a] = 0;
    for (int i = 0; i < n; ++i) {
      l[a] += E0[i] * q[a][i];
      d[a] += D0[i] * q[a][i] / 2;
    }
    for (int f = 0; f < n; ++f) {
      Dh[f][a] = 0;
      for (int i = 0; i < n; ++i) Dh[f][a] += dq[f][i] * q[a][i];
    }
  }
  const ld sigma = 2.0L * n * n;
  // bounds in units of the largest point value: trace value V, trace
  // combination A = sigma value +- half derivative; test factors lm, dm
  ld V = 0, A = 0, lm = 0, dm = 0;
  for (int a = 0; a < n; ++a) {
    V += fabsl(l[a]);
    A += fabsl(sigma * l[a] + d[a]);
    lm = fmaxl(lm, fabsl(l[a]));
    dm = fmaxl(dm, fabsl(d[a]));
  }
  const int cv = ceil_log2(V), ca = ceil_log2(A), cl = ceil_log2(lm) - 1;
  t->cg = ca + cl;
  // one face adds at most gamma (lm A + dm V) max|u| with gamma below half of its
  // exponent's unit; six of them, each 2^bump below the common exponent, stay
  // within 1.45 of the own terms' bound
  const ld kappa = (lm * A + dm * V) / ldexpl(1, ca + cl);
  t->bump = ceil_log2(3 * kappa / 1.45L);
  for (int a = 0; a < n; ++a)
    for (int i = 0; i < n; ++i) t->q[a][i] = pair_of(q[a][i]);
  bool ok = true;
  auto put = [&ok](ld v) {
    ok = ok && fabsl(v) < 2 - 0x1p-30L;  // a pair ends just below 2
    return pair_of(v);
  };
  for (int a = 0; a < (n + 1) / 2; ++a) {
    const int b = n - 1 - a;
    const ld le = a == b ? l[a] : (l[a] + l[b]) / 2, lo = a == b ? 0 : (l[a] - l[b]) / 2;
    const ld de = a == b ? d[a] : (d[a] + d[b]) / 2, dd = a == b ? 0 : (d[a] - d[b]) / 2;
    t->ve[a] = put(ldexpl(le, -cv));
    t->vo[a] = put(ldexpl(lo, -cv));
    t->ae[a] = put(ldexpl(sigma * le + de, -ca));
    t->ao[a] = put(ldexpl(sigma * lo + dd, -ca));
    t->le[a] = put(ldexpl(le, -cl));
    t->lo[a] = put(ldexpl(lo, -cl));
    t->de[a] = put(-ldexpl(de, cv - ca - cl));
    t->dn[a] = put(-ldexpl(dd, cv - ca - cl));
  }
  // line operators: h sum_f K_f Dh[f][i] Dh[f][j] + h gamma F[i][j] per face,
  // F = sigma l l^T + c (l d^T + d l^T) on the lower face (c = 1 inside, 2 on
  // the boundary), mirrored on the upper one; each of the two under its own scale
  const ld hl = (ld)h;
  ld big[2] = {0, 0}, Ff[2][DG_MAXP];
  for (int i = 0, k = 0; i < n; ++i)
    for (int j = i; j < n; ++j, ++k) {
      ld sum = 0;
      for (int f = 0; f < n; ++f) sum += fabsl(hl * Dh[f][i] * Dh[f][j]);
      big[0] = fmaxl(big[0], sum);
      for (int m = 0; m < 2; ++m) {
        Ff[m][k] = sigma * l[i] * l[j] + (m + 1) * (l[i] * d[j] + d[i] * l[j]);
        big[1] = fmaxl(big[1], fabsl(Ff[m][k]));
      }
    }
  s->cV = ceil_log2(big[0]);
  s->cF = ceil_log2(big[1]);
  for (int i = 0, k = 0; i < n; ++i)
    for (int j = i; j < n; ++j, ++k) {
      for (int f = 0; f < n; ++f)
        s->DD[f][k] = put(ldexpl(hl * Dh[f][i] * Dh[f][j], -s->cV));
      for (int m = 0; m < 2; ++m) s->F[m][k] = put(ldexpl(Ff[m][k], -s->cF));
    }
  // the scaled derivative: Dh[n-1-f][n-1-a] = -Dh[f][a], so its even and odd
  // halves over the mirror pairs give both points of a pair
  ld row = 0;
  for (int f = 0; f < n; ++f) {
    ld sum = 0;
    for (int a = 0; a < n; ++a) sum += fabsl(Dh[f][a]);
    row = fmaxl(row, sum);
    sum = 0;  // and of the transpose
    for (int a = 0; a < n; ++a) sum += fabsl(Dh[a][f]);
    row = fmaxl(row, sum);
  }
  g->cD = ceil_log2(row);
  for (int f = 0; f < (n + 1) / 2; ++f)
    for (int a = 0; a < (n + 1) / 2; ++a) {
      const int b = n - 1 - a;
      const ld e = a == b ? Dh[f][a] : (Dh[f][a] + Dh[f][b]) / 2;
      const ld o = a == b ? 0 : (Dh[f][a] - Dh[f][b]) / 2;
      g->De[f][a] = put(ldexpl(f == n - 1 - f ? 0 : e, -g->cD));
      g->Do[f][a] = put(ldexpl(o, -g->cD));
    }
  g->cj[0] = put(ldexpl(sigma / 2, cv - ca - 2));
  g->cj[1] = put(ldexpl(3 * sigma / 2, cv - ca - 2));
  g->cva = cv + ca;
  g->cv = cv;
  g->cl = cl;
  for (int a = 0; a < n; ++a) {
    g->w[a] = (double)w[a];
    g->iw[a] = (double)(1 / w[a]);
  }
  return ok;
}
