// Host run of the fixed-point GRP of an interface (csrc/grp_fixed.cuh) against
// the same formulas in quad precision and against the FP64 path (grp_euler),
// over seeded states: slopes, Mach numbers on both sides of one, resting gas,
// kinks, units over 40 binary orders.  Prints one line per regime:
//   degree from_traces gamma slope share_in_fixed_point rms_error max_error rms_error_fp64 max_error_fp64 wrong
// wrong: interfaces the fixed path accepted although a field is sonic or the
// series is cut at a Gauss node.  Errors are relative to rho a^k, a = |u| + c.
#include <cstdio>
#include <cstdlib>
#include <quadmath.h>
#include <random>

#include "grp_fixed.cuh"

using namespace grp;
typedef __float128 T;

// Exact Riemann state at x / t = 0, gamma = 7/5 (Newton on the star pressure);
// near: a decision of the sampling within 1e-9 of its threshold
static void quad_riemann(const T QL[3], const T QR[3], T Q0[3], T& u0, T& p0, bool& near_)
{
  const T g = (T)1.4 - (T)1.4 + (T)7 / 5, gm1 = (T)(1.4 - 1.0);
  T r[2] = {QL[0], QR[0]}, u[2] = {QL[1] / QL[0], QR[1] / QR[0]}, p[2], c[2];
  p[0] = gm1 * (QL[2] - QL[1] * u[0] / 2); p[1] = gm1 * (QR[2] - QR[1] * u[1] / 2);
  for (int k = 0; k < 2; ++k) c[k] = sqrtq((T)1.4 * p[k] / r[k]);
  T ps = (p[0] + p[1]) / 2, f[2], d[2], us = 0;
  for (int it = 0; it < 60; ++it) {
    for (int k = 0; k < 2; ++k) {
      if (ps > p[k]) {
        const T A = 2 / ((g + 1) * r[k]), B = (g - 1) / (g + 1) * p[k], s = sqrtq(A / (ps + B));
        f[k] = (ps - p[k]) * s; d[k] = s * (1 - (ps - p[k]) / (ps + B) / 2);
      } else {
        const T x = ps / p[k], w = powq(x, (T)1 / 7);
        f[k] = 5 * c[k] * (w - 1); d[k] = w / x / (r[k] * c[k]);
      }
    }
    const T st = -(f[0] + f[1] + u[1] - u[0]) / (d[0] + d[1]);
    us = (u[0] + u[1] + f[1] - f[0]) / 2;
    ps += st;
    if (fabsq(st) < (T)1e-30 * ps && it > 2) break;
  }
  const T tie = (T)1e-10 * (c[0] + c[1]);
  near_ = fabsq(us + tie) < (T)1e-13 * c[0];
  const int k = us >= -tie ? 0 : 1;
  const T sg = k ? -1 : 1, x = ps / p[k], um = sg * us, uk = sg * u[k];
  bool own = false;
  T rho;
  if (ps > p[k]) {
    const T S = uk - c[k] * sqrtq((g + 1) / (2 * g) * x + (g - 1) / (2 * g));
    own = S >= 0; near_ = near_ || fabsq(S) < (T)1e-9 * c[k];
    rho = r[k] * (x + (T)1 / 6) / (x / 6 + 1);
  } else {
    own = uk - c[k] >= 0; near_ = near_ || fabsq(uk - c[k]) < (T)1e-9 * c[k];
    rho = r[k] * powq(x, (T)5 / 7);
    const T tail = um - c[k] * powq(x, (T)1 / 7);
    near_ = near_ || (!own && tail > -(T)1e-9 * c[k]);             // in or next to a fan
  }
  u0 = own ? u[k] : us; p0 = own ? p[k] : ps; rho = own ? r[k] : rho;
  Q0[0] = rho; Q0[1] = rho * u0; Q0[2] = p0 / gm1 + rho * u0 * u0 / 2;
}

// general: a field is sonic, or a state at a node or at dt is inadmissible
template <int M>
static bool quad_grp(double gamma, double nu_, const T tl[3][M + 1], const T tr[3][M + 1],
                     T out[6], bool* skip)
{
  const T gm1 = (T)(gamma - 1.0), gam = gamma, nu = nu_;
  T Q[3] = {tl[0][0], tl[1][0], tl[2][0]}, u = Q[1] / Q[0], p = gm1 * (Q[2] - Q[1] * u / 2);
  bool general = false;
  if (tl[0][0] != tr[0][0] || tl[1][0] != tr[1][0] || tl[2][0] != tr[2][0]) {
    const T QL[3] = {tl[0][0], tl[1][0], tl[2][0]}, QR[3] = {tr[0][0], tr[1][0], tr[2][0]};
    quad_riemann(QL, QR, Q, u, p, general);
    if (general) { *skip = true; return true; }
  }
  const T c2 = gam * p / Q[0], c = sqrtq(c2), H = (Q[2] + p) / Q[0];
  const T lam[3] = {u - c, u, u + c}, tie = (T)1e-10 * (fabsq(u) + c), b1 = gm1 / c2, b2 = b1 * u * u / 2;
  const T l[3][3] = {{(b2 + u / c) / 2, -(b1 * u + 1 / c) / 2, b1 / 2}, {1 - b2, b1 * u, -b1},
                     {(b2 - u / c) / 2, -(b1 * u - 1 / c) / 2, b1 / 2}};
  const T r[3][3] = {{1, u - c, H - u * c}, {1, u, u * u / 2}, {1, u + c, H + u * c}};
  T q[3][M + 1][M + 1], F[3][M + 1][M + 1], U[M + 1][M + 1], P[M + 1][M + 1];
  for (int c2_ = 0; c2_ < 3; ++c2_) q[c2_][0][0] = Q[c2_];
  for (int k = 1; k <= M; ++k) {
    T D[3];
    for (int i = 0; i < 3; ++i) D[i] = tl[i][k];
    for (int j = 0; j < 3; ++j) {
      const T th = lam[j] > tie ? (T)0 : (lam[j] < -tie ? (T)1 : (T)0.5);
      if (j != 1 && th == (T)0.5) general = true;
      T w = 0;
      for (int i = 0; i < 3; ++i) w += l[j][i] * (tl[i][k] - tr[i][k]);
      for (int i = 0; i < 3; ++i) D[i] -= th * w * r[j][i];
    }
    for (int i = 0; i < 3; ++i) q[i][k][0] = D[i];
  }
  for (int b = 0; b < M; ++b) {
    for (int a = 0; a + b <= M; ++a) {
      T acc = q[1][a][b], mm = 0, f = 0;
      for (int i = 0; i <= a; ++i) for (int j = 0; j <= b; ++j) if (i || j) acc -= q[0][i][j] * U[a - i][b - j];
      U[a][b] = acc / Q[0];
      for (int i = 0; i <= a; ++i) for (int j = 0; j <= b; ++j) mm += q[1][i][j] * U[a - i][b - j];
      const T pp = gm1 * (q[2][a][b] - mm / 2);
      P[a][b] = q[2][a][b] + pp;
      for (int i = 0; i <= a; ++i) for (int j = 0; j <= b; ++j) f += U[i][j] * P[a - i][b - j];
      F[0][a][b] = q[1][a][b]; F[1][a][b] = mm + pp; F[2][a][b] = f;
    }
    for (int a = 0; a + b + 1 <= M; ++a)
      for (int i = 0; i < 3; ++i) q[i][a][b + 1] = -(T)(a + 1) / (T)(b + 1) * F[i][a + 1][b];
  }
  for (int k = 0; k < 6; ++k) out[k] = 0;
  constexpr int G = Gauss<M>::G;
  for (int n = 0; n <= G; ++n) {
    const T a = G == 2 ? sqrtq((T)1 / 12) : sqrtq((T)3 / 20), w = G == 1 ? (T)1 : G == 2 ? (T)0.5 : (n == 1 ? (T)4 / 9 : (T)5 / 18);
    const T t = (n == G ? (T)1 : G == 1 ? (T)0.5 : n == 0 ? (T)0.5 - a : n == G - 1 ? (T)0.5 + a : (T)0.5) * nu;
    T v[3];
    for (int i = 0; i < 3; ++i) { v[i] = q[i][0][M]; for (int k = M - 1; k >= 0; --k) v[i] = v[i] * t + q[i][0][k]; }
    const T s = v[1] / v[0], pp = gm1 * (v[2] - v[1] * s / 2);
    if (!(v[0] > 0 && pp > 0)) general = true;
    if (n < G) { out[0] += w * v[1]; out[1] += w * (v[1] * s + pp); out[2] += w * s * (v[2] + pp); }
    else for (int i = 0; i < 3; ++i) out[3 + i] = v[i];
  }
  return general;
}

// Taylor coefficients at the edge of p = b0 + b1 xi + b2 (xi^2 - 1/12) + b3 xi^3 + b4 (xi^4 - 1/80)
template <int M>
static void quad_edges(const double* x, const double gl, const double gr, int side, T t[M + 1])
{
  T b[5] = {x[1], 0, 0, 0, 0};
  const T q = x[1], g0 = gl, g1 = gr, dg = g1 - g0, qm = x[0], qp = x[2];
  if (M <= 2) b[1] = dg;
  if (M == 2) b[2] = 3 * (g0 + g1 - 2 * q);
  if (M >= 3) { b[1] = (10 * dg - (qp - qm)) / 8; b[3] = (qp - qm) / 2 - dg; }
  if (M == 3) b[2] = 3 * (g0 + g1 - 14 * q + 6 * (qm + qp)) / 37;
  if (M == 4) { b[2] = (30 * (g0 + g1) - 58 * q - (qm + qp)) / 8; b[4] = -5 * (6 * (g0 + g1) - 10 * q - (qm + qp)) / 12; }
  const T s = side * (T)0.5;
  T e[5];
  e[0] = M % 2 == 0 ? (side > 0 ? g1 : g0) : b[0] + b[1] * s + b[2] * (s * s - (T)1 / 12) + b[3] * s * s * s;
  e[1] = b[1] + 2 * b[2] * s + 3 * b[3] * s * s + 4 * b[4] * s * s * s;
  e[2] = b[2] + 3 * b[3] * s + 6 * b[4] * s * s;
  e[3] = b[3] + 4 * b[4] * s;
  e[4] = b[4];
  for (int k = 0; k <= M; ++k) t[k] = e[k];
}

// traces: the interface is given by its traces (grp_traces), with a jump of the
// slopes' size; else by averages and interface data (grp_linear)
template <int M, bool TR>
static void run(int count)
{
  std::mt19937_64 rng(2602);
  auto U = [&](double a, double b) { return a + (b - a) * (double)(rng() >> 11) * (1.0 / 9007199254740992.0); };
  const double gammas[4] = {1.4, 1.3, 5.0 / 3.0, 1.9}, slopes[5] = {0.0, 1e-3, 0.05, 0.3, 1.0};
  constexpr bool EQ = !TR && M % 2 == 0;
  constexpr int NQ = M <= 2 ? 2 : 4;
  for (int gi = 0; gi < (EQ ? 4 : 1); ++gi)
    for (double amp : slopes) {
      const double gamma = gammas[gi];
      const Phys ph = make_phys(1.0, gamma, 1e-12, 50, 0);
      const fixed::Consts K = fixed::make_consts(gamma);
      double sf = 0, sd = 0, mf = 0, md = 0;
      int n = 0, took = 0, wrong = 0;
      while (n < count) {
        const double S = exp2(floor(U(-40, 40))) * U(1, 2), V = exp2(floor(U(-20, 20))) * U(1, 2);
        const double rho = exp(U(-1, 1)), p = exp(U(-1, 1)), c = sqrt(gamma * p / rho);
        const double u = n % 5 == 0 ? 0.0 : (n % 5 == 1 ? U(-6, 6) : U(-1.2, 1.2)) * c;
        const double size[3] = {rho, c, p};
        // points x = -3/2, -1, ..., 3/2: averages at even places, interface data between
        double v[7][3], Q[7][3];
        bool good = true;
        for (int j = 0; j < 3; ++j) {
          const double s = U(-amp, amp) * size[j], k = U(-amp, amp) * size[j], z = 0.3 * U(-amp, amp) * size[j];
          for (int i = 0; i < 7; ++i) {
            const double x = 0.5 * (i - 3);
            v[i][j] = (j == 0 ? rho : j == 1 ? u : p);
            if (!(j == 1 && n % 10 == 0)) v[i][j] += s * x + 0.5 * k * x * x + (x > 0 ? z * x : 0);
          }
        }
        for (int i = 0; i < 7; ++i) {
          good = good && v[i][0] > 0 && v[i][2] > 0;
          Q[i][0] = v[i][0] * S; Q[i][1] = v[i][0] * v[i][1] * S * V;
          Q[i][2] = (v[i][2] / ph.gm1 + 0.5 * v[i][0] * v[i][1] * v[i][1]) * S * V * V;
        }
        if (!good) continue;
        ++n;
        // cells at x = -1/2 and 1/2 (places 2, 4), beyond at 0, 6; data at -1, 0, 1 (places 1, 3, 5)
        double q[NQ][3], g[3][3], F[3], gn[3], Fd[3], gd[3], tL[3][M + 1], tR[3][M + 1];
        T ql[3][M + 1], qr[3][M + 1];
        for (int j = 0; j < 3; ++j) {
          for (int k = 0; k < NQ; ++k) q[k][j] = Q[M <= 2 ? 2 + 2 * k : 2 * k][j];
          for (int k = 0; k < 3; ++k) g[k][j] = Q[1 + 2 * k][j];
          const double xl[3] = {Q[0][j], Q[2][j], Q[4][j]}, xr[3] = {Q[2][j], Q[4][j], Q[6][j]};
          double b[5];
          grprec_coeffs<M>(xl[0], xl[1], xl[2], g[0][j], g[1][j], b);
          edge_taylor<M>(b, 1.0, tL[j]);
          grprec_coeffs<M>(xr[0], xr[1], xr[2], g[1][j], g[2][j], b);
          edge_taylor<M>(b, -1.0, tR[j]);
          if (EQ) tL[j][0] = tR[j][0] = g[1][j];
          if (TR) { tL[j][0] = 0.5 * (g[0][j] + g[1][j]); tR[j][0] = 0.5 * (g[2][j] + g[1][j]); }
          if (TR) {
            for (int k = 0; k <= M; ++k) { ql[j][k] = tL[j][k]; qr[j][k] = tR[j][k]; }
          } else {
            quad_edges<M>(xl, g[0][j], g[1][j], 1, ql[j]);
            quad_edges<M>(xr, g[1][j], g[2][j], -1, qr[j]);
          }
        }
        const double a = (fabs(u) + c) * V, nu = U(0.1, 0.9) / a;
        bool newton;
        const bool ok = TR ? fixed::grp_traces<M>(K, ph.gm1, nu, tL, tR, F, gn, newton)
                           : fixed::grp_linear<M>(K, ph.gm1, nu, q, g, F, gn, newton);
        if (!ok) continue;
        T ref[6];
        bool skip = false;
        if (quad_grp<M>(gamma, nu, ql, qr, ref, &skip)) { wrong += skip ? 0 : 1; continue; }
        int it;
        bool cut;
        grp_euler<M, EQ ? false : true>(ph, nu, tL, tR, Fd, gd, it, cut);
        ++took;
        const double rs = rho * S, unit[6] = {rs * a, rs * a * a, rs * a * a * a, rs, rs * a, rs * a * a};
        for (int k = 0; k < 6; ++k) {
          const double ef = fabs((double)((k < 3 ? F[k] : gn[k - 3]) - ref[k])) / unit[k];
          const double ed = fabs((double)((k < 3 ? Fd[k] : gd[k - 3]) - ref[k])) / unit[k];
          sf += ef * ef; sd += ed * ed;
          mf = ef > mf ? ef : mf; md = ed > md ? ed : md;
        }
      }
      printf("%d %d %.3f %.3f %.5f %.3e %.3e %.3e %.3e %d\n", M, TR ? 1 : 0, gamma, amp, (double)took / n,
             sqrt(sf / (6.0 * took)), mf, sqrt(sd / (6.0 * took)), md, wrong);
    }
}

int main(int argc, char** argv)
{
  const int count = argc > 1 ? atoi(argv[1]) : 20000;
  run<2, false>(count);
  run<4, false>(count);
  run<1, false>(count);
  run<3, false>(count);
  run<1, true>(count);
  run<2, true>(count);
  run<3, true>(count);
  return 0;
}
