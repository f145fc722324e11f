// Host run of the fixed-point GRP of an interface (csrc/grp_fixed.cuh) against
// the same formulas in quad precision and against the FP64 path (grp_euler),
// over seeded states: slopes, Mach numbers on both sides of one, resting gas,
// kinks, units over 40 binary orders.  Prints one line per regime:
//   gamma slope share_in_fixed_point rms_error max_error rms_error_fp64 max_error_fp64 wrong
// wrong: interfaces the fixed path accepted although a field is sonic or the
// series is cut at a Gauss node.  Errors are relative to rho a^k, a = |u| + c.
#include <cstdio>
#include <cstdlib>
#include <quadmath.h>
#include <random>

#include "grp_fixed.cuh"

using namespace grp;
typedef __float128 T;

// general: a field is sonic, or a state at a node or at dt is inadmissible
static bool quad_grp(double gamma, double nu_, const double q[2][3], const double g[3][3], T out[6])
{
  const T gm1 = (T)(gamma - 1.0), gam = gamma, nu = nu_;
  T L[2][3], R[2][3], Q[3];
  for (int c = 0; c < 3; ++c) {
    const T g0 = g[0][c], g1 = g[1][c], g2 = g[2][c], ql = q[0][c], qr = q[1][c];
    L[1][c] = 3 * (g0 + g1 - 2 * ql); L[0][c] = g1 - g0 + L[1][c];
    R[1][c] = 3 * (g1 + g2 - 2 * qr); R[0][c] = g2 - g1 - R[1][c];
    Q[c] = g1;
  }
  const T u = Q[1] / Q[0], p = gm1 * (Q[2] - Q[1] * u / 2), c2 = gam * p / Q[0], c = sqrtq(c2), H = (Q[2] + p) / Q[0];
  const T lam[3] = {u - c, u, u + c}, tie = (T)1e-10 * (fabsq(u) + c), b1 = gm1 / c2, b2 = b1 * u * u / 2;
  const T l[3][3] = {{(b2 + u / c) / 2, -(b1 * u + 1 / c) / 2, b1 / 2}, {1 - b2, b1 * u, -b1},
                     {(b2 - u / c) / 2, -(b1 * u - 1 / c) / 2, b1 / 2}};
  const T r[3][3] = {{1, u - c, H - u * c}, {1, u, u * u / 2}, {1, u + c, H + u * c}};
  bool general = false;
  T D[2][3];
  for (int o = 0; o < 2; ++o) {
    for (int k = 0; k < 3; ++k) D[o][k] = L[o][k];
    for (int j = 0; j < 3; ++j) {
      const T th = lam[j] > tie ? (T)0 : (lam[j] < -tie ? (T)1 : (T)0.5);
      if (j != 1 && th == (T)0.5) general = true;
      T w = 0;
      for (int k = 0; k < 3; ++k) w += l[j][k] * (L[o][k] - R[o][k]);
      for (int k = 0; k < 3; ++k) D[o][k] -= th * w * r[j][k];
    }
  }
  const T m0 = Q[1], ir = 1 / Q[0], r1 = D[0][0], m1 = D[0][1], E1 = D[0][2], r2 = D[1][0], m2 = D[1][1], E2 = D[1][2];
  const T Ep0 = Q[2] + p, u1 = (m1 - r1 * u) * ir, u2 = (m2 - r2 * u - r1 * u1) * ir;
  const T mu1 = m1 * u + m0 * u1, mu2 = m2 * u + m1 * u1 + m0 * u2;
  const T p1 = gm1 * (E1 - mu1 / 2), p2 = gm1 * (E2 - mu2 / 2), Ep1 = E1 + p1, Ep2 = E2 + p2;
  const T rt = -m1, mt = -(mu1 + p1), Et = -(u * Ep1 + u1 * Ep0);
  const T rx = -2 * m2, mx = -2 * (mu2 + p2), Ex = -2 * (u * Ep2 + u1 * Ep1 + u2 * Ep0);
  const T ut = (mt - rt * u) * ir, Ept = Et + gm1 * (Et - (mt * u + m0 * ut) / 2);
  const T ux = (mx - r1 * ut - rt * u1 - rx * u) * ir, mux = mx * u + m1 * ut + mt * u1 + m0 * ux;
  const T px = gm1 * (Ex - mux / 2), fx = u * (Ex + px) + u1 * Ept + ut * Ep1 + ux * Ep0;
  const T s1[3] = {rt, mt, Et}, s2[3] = {-mx / 2, -(mux + px) / 2, -fx / 2};
  for (int k = 0; k < 6; ++k) out[k] = 0;
  for (int n = 0; n < 3; ++n) {
    const T a = 1 / sqrtq((T)12), t = (n == 0 ? (T)0.5 - a : n == 1 ? (T)0.5 + a : (T)1) * nu;
    T v[3];
    for (int k = 0; k < 3; ++k) v[k] = Q[k] + t * (s1[k] + t * s2[k]);
    const T w = v[1] / v[0], pp = gm1 * (v[2] - v[1] * w / 2);
    if (!(v[0] > 0 && pp > 0)) general = true;
    if (n < 2) { out[0] += v[1] / 2; out[1] += (v[1] * w + pp) / 2; out[2] += w * (v[2] + pp) / 2; }
    else for (int k = 0; k < 3; ++k) out[3 + k] = v[k];
  }
  return general;
}

int main(int argc, char** argv)
{
  const int count = argc > 1 ? atoi(argv[1]) : 20000;
  std::mt19937_64 rng(2602);
  auto U = [&](double a, double b) { return a + (b - a) * (double)(rng() >> 11) * (1.0 / 9007199254740992.0); };
  const double gammas[4] = {1.2, 1.4, 5.0 / 3.0, 1.9}, slopes[5] = {0.0, 1e-3, 0.05, 0.3, 1.0};
  for (double gamma : gammas)
    for (double amp : slopes) {
      const Phys ph = make_phys(1.0, gamma, 1e-12, 50, 0);
      const fixed::fx gm1 = fixed::to_format(ph.gm1), hg = fixed::to_format(0.5 * gamma);
      double sf = 0, sd = 0, mf = 0, md = 0;
      int n = 0, took = 0, wrong = 0;
      while (n < count) {
        const double S = exp2(floor(U(-40, 40))) * U(1, 2), V = exp2(floor(U(-20, 20))) * U(1, 2);
        const double rho = exp(U(-1, 1)), p = exp(U(-1, 1)), c = sqrt(gamma * p / rho);
        const double u = n % 5 == 0 ? 0.0 : (n % 5 == 1 ? U(-6, 6) : U(-1.2, 1.2)) * c;
        const double size[3] = {rho, c, p};
        double v[5][3], Q[5][3];
        bool good = true;
        for (int j = 0; j < 3; ++j) {
          const double s = U(-amp, amp) * size[j], k = U(-amp, amp) * size[j], z = 0.3 * U(-amp, amp) * size[j];
          for (int i = 0; i < 5; ++i) {
            const double x = 0.5 * (i - 2);
            v[i][j] = (j == 0 ? rho : j == 1 ? u : p);
            if (!(j == 1 && n % 10 == 0)) v[i][j] += s * x + 0.5 * k * x * x + (x > 0 ? z * x : 0);
          }
        }
        for (int i = 0; i < 5; ++i) {
          good = good && v[i][0] > 0 && v[i][2] > 0;
          Q[i][0] = v[i][0] * S; Q[i][1] = v[i][0] * v[i][1] * S * V;
          Q[i][2] = (v[i][2] / ph.gm1 + 0.5 * v[i][0] * v[i][1] * v[i][1]) * S * V * V;
        }
        if (!good) continue;
        ++n;
        double q[2][3], g[3][3], F[3], gn[3], Fd[3], gd[3], tL[3][3], tR[3][3];
        for (int j = 0; j < 3; ++j) {
          g[0][j] = Q[0][j]; q[0][j] = Q[1][j]; g[1][j] = Q[2][j]; q[1][j] = Q[3][j]; g[2][j] = Q[4][j];
          double b[5], t[3];
          grprec_coeffs<2>(0.0, q[0][j], 0.0, g[0][j], g[1][j], b);
          edge_taylor<2>(b, 1.0, t);
          tL[j][0] = g[1][j]; tL[j][1] = t[1]; tL[j][2] = t[2];
          grprec_coeffs<2>(0.0, q[1][j], 0.0, g[1][j], g[2][j], b);
          edge_taylor<2>(b, -1.0, t);
          tR[j][0] = g[1][j]; tR[j][1] = t[1]; tR[j][2] = t[2];
        }
        const double a = (fabs(u) + c) * V, nu = U(0.1, 0.9) / a;
        if (!fixed::grp_equal2(ph.gm1, gm1, hg, nu, q, g, F, gn)) continue;
        T ref[6];
        if (quad_grp(gamma, nu, q, g, ref)) { ++wrong; continue; }
        int it;
        bool cut;
        grp_euler<2, false>(ph, nu, tL, tR, Fd, gd, it, cut);
        ++took;
        const double rs = rho * S, unit[6] = {rs * a, rs * a * a, rs * a * a * a, rs, rs * a, rs * a * a};
        for (int k = 0; k < 6; ++k) {
          const double ef = fabs((double)((k < 3 ? F[k] : gn[k - 3]) - ref[k])) / unit[k];
          const double ed = fabs((double)((k < 3 ? Fd[k] : gd[k - 3]) - ref[k])) / unit[k];
          sf += ef * ef; sd += ed * ed;
          mf = ef > mf ? ef : mf; md = ed > md ? ed : md;
        }
      }
      printf("%.3f %.3f %.5f %.3e %.3e %.3e %.3e %d\n", gamma, amp, (double)took / n, sqrt(sf / (6.0 * took)), mf,
             sqrt(sd / (6.0 * took)), md, wrong);
    }
  return 0;
}
