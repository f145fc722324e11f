// Host run of the fixed-point Riemann problems (csrc/grp_fixed.cuh, gamma = 7/5)
// over independent left and right states, against quad precision and against
// the FP64 path.  Prints one line per regime:
//   kind degree spread share_in_fixed_point rms_error max_error rms_error_fp64 max_error_fp64 wrong
// kind 0: riemann_flux (state and flux of the leading problem); 1: the same of
// data inadmissible on one side; 2: grp_traces with slopes up to `spread` times the
// states' size; 3: grp_linear of rough data; 4: grp_traces of inadmissible constant data.  wrong: problems the fixed path accepted although a
// side is inadmissible, the contact's side or the wave at x / t = 0 is not decided,
// a field is sonic or the series is cut.  Errors are relative to rho a^k,
// a = |u| + c, of the larger of the two sides.
#define main smooth_main
#include "fixed_point_check.cu"
#undef main

// The exact Riemann state at x / t = 0 in quad precision.  Newton's iteration from
// below (the velocity function is concave: no overshoot), two rarefactions in
// closed form.  false: vacuum, or a decision of the sampling within 1e-9 of its
// threshold (in or next to a fan among them).
static bool exact_state(const T QL[3], const T QR[3], T Q0[3], T& u0, T& p0)
{
  const T z = (T)1 / 7, gm1 = (T)(1.4 - 1.0);
  T r[2] = {QL[0], QR[0]}, u[2] = {QL[1] / QL[0], QR[1] / QR[0]}, p[2], c[2], ps, f[2] = {0, 0};
  for (int k = 0; k < 2; ++k) {
    p[k] = gm1 * ((k ? QR : QL)[2] - (k ? QR : QL)[1] * u[k] / 2);
    c[k] = sqrtq((T)1.4 * p[k] / r[k]);
  }
  const T du = u[1] - u[0];
  if (du >= 5 * (c[0] + c[1])) return false;
  ps = p[0] < p[1] ? p[0] : p[1];
  for (int it = 0; it < 200; ++it) {
    T d[2];
    for (int k = 0; k < 2; ++k) {
      if (ps > p[k]) {
        const T A = (T)5 / (6 * r[k]), B = p[k] / 6, s = sqrtq(A / (ps + B));
        f[k] = (ps - p[k]) * s; d[k] = s * (1 - (ps - p[k]) / (ps + B) / 2);
      } else {
        const T x = ps / p[k], w = powq(x, z);
        f[k] = 5 * c[k] * (w - 1); d[k] = w / x / (r[k] * c[k]);
      }
    }
    const T g = f[0] + f[1] + du;
    if (it == 0 && g > 0) {                                        // two rarefactions
      const T w = (c[0] + c[1] - du / 5) / (c[0] * powq(p[0], -z) + c[1] * powq(p[1], -z));
      ps = powq(w, 7);
      for (int k = 0; k < 2; ++k) f[k] = 5 * c[k] * (w * powq(p[k], -z) - 1);
      break;
    }
    const T st = -g / (d[0] + d[1]);
    ps += st;
    if (it > 2 && fabsq(st) < (T)1e-32 * ps) break;
  }
  const T us = (u[0] + u[1] + f[1] - f[0]) / 2, tie = (T)1e-10 * (c[0] + c[1]), eps = (T)1e-9;
  if (fabsq(us + tie) < (T)1e-13 * c[0]) return false;
  const int k = us >= -tie ? 0 : 1;
  const T sg = k ? -1 : 1, x = ps / p[k], um = sg * us, uk = sg * u[k];
  T rho;
  bool own;
  if (ps > p[k]) {
    const T S = uk - c[k] * sqrtq((6 * x + 1) / 7);
    if (fabsq(S) < eps * c[k]) return false;
    own = S >= 0;
    rho = r[k] * (x + (T)1 / 6) / (x / 6 + 1);
  } else {
    if (fabsq(uk - c[k]) < eps * c[k]) return false;
    own = uk >= c[k];
    rho = r[k] * powq(x, (T)5 / 7);
    if (!own && um - c[k] * powq(x, z) > -eps * c[k]) return false;
  }
  u0 = own ? u[k] : us; p0 = own ? p[k] : ps; rho = own ? r[k] : rho;
  Q0[0] = rho; Q0[1] = rho * u0; Q0[2] = p0 / gm1 + rho * u0 * u0 / 2;
  return true;
}

struct Errors {
  double sf = 0, sd = 0, mf = 0, md = 0;
  long long took = 0;
  int n = 0, wrong = 0, terms = 6;
  void add(double fixed, double fp64, const T& ref, double unit)
  {
    const double ef = fabs((double)(fixed - ref)) / unit, ed = fabs((double)(fp64 - ref)) / unit;
    sf += ef * ef; sd += ed * ed;
    mf = ef > mf || ef != ef ? ef : mf; md = ed > md ? ed : md;
  }
  void print(int kind, int M, double spread) const
  {
    const double k = took ? (double)terms * took : 1.0;
    printf("%d %d %.2f %.5f %.3e %.3e %.3e %.3e %d\n", kind, M, spread, (double)took / n, sqrt(sf / k), mf, sqrt(sd / k),
           md, wrong);
  }
};

struct Draw {
  std::mt19937_64 rng;
  explicit Draw(int seed) : rng(seed) {}
  double U(double a, double b) { return a + (b - a) * (double)(rng() >> 11) * (1.0 / 9007199254740992.0); }
  // units of mass and speed, far from one in every other draw
  void units(int i, double& S, double& V)
  {
    S = i & 1 ? exp2(floor(U(-60, 60))) * U(1, 2) : 1.0;
    V = i & 1 ? exp2(floor(U(-30, 30))) * U(1, 2) : 1.0;
  }
  // two states; densities and pressures within exp(+-spread), velocities within 1.2 spread
  void states(double spread, double S, double V, double W[2][3], double Q[2][3])
  {
    const double u = U(-1.5, 1.5);
    for (int k = 0; k < 2; ++k) {
      W[k][0] = exp(U(-spread, spread)); W[k][1] = u + U(-1.2, 1.2) * spread; W[k][2] = exp(U(-spread, spread));
      Q[k][0] = W[k][0] * S; Q[k][1] = W[k][0] * W[k][1] * S * V;
      Q[k][2] = (2.5 * W[k][2] + 0.5 * W[k][0] * W[k][1] * W[k][1]) * S * V * V;
    }
  }
};

static void size_of(const double W[2][3], double& rho, double& a)
{
  rho = fmax(W[0][0], W[1][0]);
  a = 0.0;
  for (int k = 0; k < 2; ++k) a = fmax(a, fabs(W[k][1]) + sqrt(1.4 * W[k][2] / W[k][0]));
}

static void run_flux(int count, double spread)
{
  Draw D(2602);
  const Phys ph = make_phys(1.0, 1.4, 1e-12, 50, 0);
  const fixed::Consts K = fixed::make_consts(1.4);
  Errors e;
  for (; e.n < count; ++e.n) {
    double S, V, W[2][3], Q[2][3], Q0[3], F[3], Qd[3], Fd[3], rho, a;
    D.units(e.n, S, V);
    D.states(spread, S, V, W, Q);
    bool newton;
    if (!fixed::riemann_flux(K, ph.gm1, Q[0], Q[1], Q0, F, newton)) continue;
    T q[2][3], ref[3], u, p;
    for (int k = 0; k < 6; ++k) q[k / 3][k % 3] = Q[k / 3][k % 3];
    if (!exact_state(q[0], q[1], ref, u, p)) { ++e.wrong; continue; }
    Prim w;
    int it;
    riemann_state<true>(ph, Q[0], Q[1], false, Qd, w, it);
    euler_flux(1.4, Qd[0], Qd[1], Qd[2], Fd);
    ++e.took;
    size_of(W, rho, a);
    rho *= S; a *= V;
    const double unit[3] = {rho, rho * a, rho * a * a};
    const T fr[3] = {ref[1], ref[1] * u + p, u * (ref[2] + p)};
    for (int k = 0; k < 3; ++k) {
      e.add(Q0[k], Qd[k], ref[k], unit[k]);
      e.add(F[k], Fd[k], fr[k], unit[k] * a);
    }
  }
  e.print(0, 0, spread);
}

// The GRP (kind 2: of given traces, 3: of averages and interface data, all of them
// independent states, as on a rough grid) against the same formulas in quad
// precision, the leading problem solved by exact_state.
template <int M, bool TR>
static void run_grp(int count, double spread)
{
  Draw D(100 * M + (TR ? 1 : 0));
  const Phys ph = make_phys(1.0, 1.4, 1e-12, 50, 0);
  const fixed::Consts K = fixed::make_consts(1.4);
  constexpr int NQ = M <= 2 ? 2 : 4;
  Errors e;
  for (; e.n < count; ++e.n) {
    double S, V, W[2][3], Q[2][3], P[2][3], q[NQ][3], g[3][3], tL[3][M + 1], tR[3][M + 1], F[3], gn[3], Fd[3], gd[3];
    T ql[3][M + 1], qr[3][M + 1];
    D.units(e.n, S, V);
    D.states(TR ? 1.1 : spread, S, V, W, Q);
    double rho, a;
    size_of(W, rho, a);
    if (TR) {
      for (int c = 0; c < 3; ++c)
        for (int k = 0; k <= M; ++k) {
          const double size = rho * S * (c ? a * V : 1.0) * (c == 2 ? a * V : 1.0);
          tL[c][k] = k ? D.U(-spread, spread) * size : Q[0][c];
          tR[c][k] = k ? D.U(-spread, spread) * size : Q[1][c];
          ql[c][k] = tL[c][k]; qr[c][k] = tR[c][k];
        }
    } else {
      for (int k = 0; k < 4; k += 2) {                             // cells: beyond, left, right, beyond
        D.states(spread, S, V, W, k ? P : Q);
        double r2, a2;
        size_of(W, r2, a2);
        rho = fmax(rho, r2); a = fmax(a, a2);
      }
      double cell[4][3];
      for (int c = 0; c < 3; ++c) { cell[1][c] = Q[0][c]; cell[2][c] = Q[1][c]; cell[0][c] = P[0][c]; cell[3][c] = P[1][c]; }
      for (int k = 0; k < 2; ++k) {
        D.states(spread, S, V, W, P);
        double r2, a2;
        size_of(W, r2, a2);
        rho = fmax(rho, r2); a = fmax(a, a2);
        for (int c = 0; c < 3; ++c) { g[k][c] = P[0][c]; g[2][c] = P[1][c]; }
      }
      for (int c = 0; c < 3; ++c) {
        for (int k = 0; k < NQ; ++k) q[k][c] = cell[M <= 2 ? 1 + k : k][c];
        const double xl[3] = {cell[0][c], cell[1][c], cell[2][c]}, xr[3] = {cell[1][c], cell[2][c], cell[3][c]};
        double b[5];
        grprec_coeffs<M>(xl[0], xl[1], xl[2], g[0][c], g[1][c], b);
        edge_taylor<M>(b, 1.0, tL[c]);
        grprec_coeffs<M>(xr[0], xr[1], xr[2], g[1][c], g[2][c], b);
        edge_taylor<M>(b, -1.0, tR[c]);
        quad_edges<M>(xl, g[0][c], g[1][c], 1, ql[c]);
        quad_edges<M>(xr, g[1][c], g[2][c], -1, qr[c]);
      }
    }
    rho *= S; a *= V;
    const double nu = D.U(0.1, 0.9) / a;
    bool newton;
    if (!(TR ? fixed::grp_traces<M>(K, ph.gm1, nu, tL, tR, F, gn, newton)
             : fixed::grp_linear<M>(K, ph.gm1, nu, q, g, F, gn, newton)))
      continue;
    T a0[3] = {ql[0][0], ql[1][0], ql[2][0]}, b0[3] = {qr[0][0], qr[1][0], qr[2][0]}, Q0[3], u, p, ref[6];
    const bool adm = a0[0] > 0 && 2 * a0[2] * a0[0] > a0[1] * a0[1] && b0[0] > 0 && 2 * b0[2] * b0[0] > b0[1] * b0[1];
    if (!adm || !exact_state(a0, b0, Q0, u, p)) { ++e.wrong; continue; }
    for (int c = 0; c < 3; ++c) ql[c][0] = qr[c][0] = Q0[c];
    bool skip = false;
    if (quad_grp<M>(1.4, nu, ql, qr, ref, &skip)) { ++e.wrong; continue; }
    int it;
    bool cut;
    if (grp_euler<M, true>(ph, nu, tL, tR, Fd, gd, it, cut) != ST_OK) { ++e.wrong; continue; }
    ++e.took;
    const double unit[6] = {rho * a, rho * a * a, rho * a * a * a, rho, rho * a, rho * a * a};
    for (int k = 0; k < 6; ++k) e.add(k < 3 ? F[k] : gn[k - 3], k < 3 ? Fd[k] : gd[k - 3], ref[k], unit[k]);
  }
  e.print(TR ? 2 : 3, M, spread);
}

// Data with 2 E rho <= m^2 on one side: momenta from just beyond that to twice it, and
// velocities up to 24 times the other side's sqrt(E / rho).
static void run_inadmissible(int count, double spread, bool traces)
{
  Draw D(21911);
  const Phys ph = make_phys(1.0, 1.4, 1e-12, 50, 0);
  const fixed::Consts K = fixed::make_consts(1.4);
  Errors e;
  for (; e.n < count; ++e.n) {
    double S, V, W[2][3], Q[2][3], Q0[3], F[3];
    D.units(e.n, S, V);
    D.states(spread, S, V, W, Q);
    double *q = Q[e.n % 4 == 0 ? 0 : 1], *o = Q[e.n % 4 == 0 ? 1 : 0];
    const double bound = sqrt(2.0 * q[2] * q[0]), fast = q[0] * sqrt(o[2] / o[0]) * D.U(1.0, 24.0);
    q[1] = (e.n % 3 && fast > bound ? fast : bound * D.U(1.0 + 1e-12, 2.0)) * (D.U(-1, 1) < 0 ? -1 : 1);
    bool newton;
    if (!traces) {
      e.wrong += fixed::riemann_flux(K, ph.gm1, Q[0], Q[1], Q0, F, newton) ? 1 : 0;
      continue;
    }
    double tL[3][2], tR[3][2];
    for (int c = 0; c < 3; ++c) { tL[c][0] = Q[0][c]; tR[c][0] = Q[1][c]; tL[c][1] = tR[c][1] = 0.0; }
    e.wrong += fixed::grp_traces<1>(K, ph.gm1, 0.1 / V, tL, tR, F, Q0, newton) ? 1 : 0;
  }
  e.print(traces ? 4 : 1, 0, spread);
}

int main(int argc, char** argv)
{
  const int count = argc > 1 ? atoi(argv[1]) : 20000;
  for (double s : {0.1, 0.5, 1.1, 2.5}) run_flux(count, s);
  for (double s : {0.1, 0.5, 1.1, 2.5}) run_inadmissible(20 * count, s, false);
  for (double s : {0.1, 0.5, 1.1, 2.5}) run_inadmissible(20 * count, s, true);
  for (double s : {0.1, 0.5, 1.5, 4.0}) {
    run_grp<1, true>(count, s);
    run_grp<2, true>(count, s);
    run_grp<3, true>(count, s);
  }
  for (double s : {0.1, 0.5, 1.1, 2.5}) {
    run_grp<1, false>(count, s);
    run_grp<3, false>(count, s);
  }
  return 0;
}
