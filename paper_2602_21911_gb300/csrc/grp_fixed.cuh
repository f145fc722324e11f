// The GRP at an interface with equal data (degrees 2 and 4 of the linear
// reconstruction) in 64-bit fixed point, on the integer pipes.
//
// Why: an SM of this GPU retires 2 FP64 lane-operations per cycle and 64
// 32 x 32 -> 64 multiply-adds; one 64-bit fixed-point product costs three of
// them and a sum two 32-bit additions, so a product-sum runs about 4 times and
// a sum about 20 times as fast as its FP64 instruction (measured: 7.5 products
// and 42 sums per SM and cycle against 1.73 FP64 instructions).
//
// Precision.  Every interface has its own powers of two for length, time and
// mass (exact scalings), so that its state sits at the top of the format: a
// number x of the scaled problem is the integer x 2^61.  With V^2 a power of
// four and x = E/(rho V^2) in [1/8, 1/2):
//   density  rho 2^-(er+2)          in [1/8, 1/4)   2^58..2^59 units
//   momentum rho V as unit of rho   |m| < rho
//   energy   2 E (twice the unit)   in [rho/4, rho) at least 2^56 units
//   velocity u / V                  |u| < 1
// A double of the interface's state converts exactly (its last bit is worth 8
// units or more), a product is off by at most 2 units (its low x low partial
// product is left out), so an operation's error is 2^-56 or less of the state
// where an FP64 operation's is 2^-53.  Nothing wraps unseen: every operand of a
// product is tested against its bound, and an interface that leaves the range
// (a jump of more than about 4 between neighbours, sonic fields, a state near
// vacuum) is solved in FP64 by the second pass instead.
#pragma once
#include "grp_device.cuh"

namespace grp {
namespace fixed {

typedef long long fx;                       // x 2^61
constexpr fx ONE = 1ll << 61;

GRP_HD __forceinline__ fx mad(int a, int b, fx c)
{
#ifdef __CUDA_ARCH__
  fx r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (fx)a * b + c;
#endif
}
GRP_HD __forceinline__ fx shl(fx x, int s) { return (fx)((unsigned long long)x << s); }
GRP_HD __forceinline__ fx add(fx a, fx b) { return (fx)((unsigned long long)a + (unsigned long long)b); }
GRP_HD __forceinline__ fx sub(fx a, fx b) { return (fx)((unsigned long long)a - (unsigned long long)b); }

// balanced limbs: x = h 2^32 + l with l signed, so that every partial product
// is a signed 32 x 32 one
struct Op { int h, l; };
GRP_HD __forceinline__ Op op(fx x)
{
  const int l = (int)(unsigned)(unsigned long long)x;
  return Op{(int)(x >> 32) + (int)((unsigned)l >> 31), l};
}

// bits of the high word that differ from the sign, where |x| >= 2^lim is to be seen
GRP_HD __forceinline__ unsigned over(fx x, int lim)
{
  const int h = (int)(x >> 32);
  return (unsigned)(h ^ (int)((unsigned)h << 1)) & ~((2u << (lim - 32)) - 1u);
}

// Sum of products.  hi carries 2^64, mid 2^32; with operands below 2^61 a
// product adds at most 2^61 to mid, so mid is moved up after three.
struct Dot {
  fx hi, mid;
  int n;                                    // products in mid (a compile-time constant after unrolling)
  GRP_HD __forceinline__ Dot() : hi(0), mid(0), n(0) {}
  GRP_HD __forceinline__ void mac(Op a, Op b)
  {
    if (n == 3) { hi = fixed::add(hi, mid >> 32); mid = (fx)(unsigned)mid; n = 0; }
    hi = mad(a.h, b.h, hi);
    mid = mad(a.h, b.l, mid);
    mid = mad(a.l, b.h, mid);
    ++n;
  }
  GRP_HD __forceinline__ void mac(fx a, fx b) { mac(op(a), op(b)); }
  // the sum / 2^S; bad collects a result of 2^lim or more
  template <int S>
  GRP_HD __forceinline__ fx value(unsigned& bad, int lim = 61) const
  {
    bad |= over(hi, lim - (64 - S));
    return fixed::add(shl(hi, 64 - S), mid >> (S - 32));
  }
  template <int S>
  GRP_HD __forceinline__ fx value() const { return fixed::add(shl(hi, 64 - S), mid >> (S - 32)); }
};

// one product / 2^S
template <int S>
GRP_HD __forceinline__ fx mul(fx a, fx b)
{
  Dot d;
  d.mac(a, b);
  return d.value<S>();
}
template <int S>
GRP_HD __forceinline__ fx mul(fx a, fx b, unsigned& bad, int lim = 61)
{
  Dot d;
  d.mac(a, b);
  return d.value<S>(bad, lim);
}
// ... with the low x low partial product, for results shifted up
template <int S>
GRP_HD __forceinline__ fx mul_full(fx a, fx b, unsigned& bad)
{
  const Op x = op(a), y = op(b);
  Dot d;
  d.hi = mad(x.h, y.h, 0);
  d.mid = mad(x.h, y.l, mad(x.l, y.l, 0) >> 32);
  d.mid = mad(x.l, y.h, d.mid);
  return d.value<S>(bad);
}
// a value tested against 2^lim on its way to a product
GRP_HD __forceinline__ fx chk(fx x, unsigned& bad, int lim = 61)
{
  bad |= over(x, lim);
  return x;
}

// 1/(32 rho) for rho in [1/16, 1/2) (R in [2^57, 2^60)): FP32 seed (relative
// error e < 2^-22) and one step iv (1 + e + e^2), error e^3
GRP_HD __forceinline__ fx recip32(fx R)
{
  const float f = (float)(int)(R >> 32);
#ifdef __CUDA_ARCH__
  float g;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(g) : "f"(f));
#else
  const float g = 1.0f / f;
#endif
  const int h = (int)(g * 9007199254740992.0f);                    // 2^53
  const Op r = op(R);
  // 32 R (h 2^32) / 2^61 = R h / 2^24
  const fx e = sub(ONE, add(shl(mad(r.h, h, 0), 8), mad(r.l, h, 0) >> 24));
  const int es = (int)(e >> 10);
  const Op c = op(add(e, mad(es, es, 0) >> 41));
  return add(shl((fx)h, 32), add(shl(mad(h, c.h, 0), 3), mad(h, c.l, 0) >> 29));
}

// 1/(8 c) from c^2 in [1/64, 1): FP32 seed and one step y (1 + e/2 + 3 e^2/8)
GRP_HD __forceinline__ fx rsqrt8(fx c2)
{
  const float f = (float)(int)(c2 >> 32);
#ifdef __CUDA_ARCH__
  float g;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(g) : "f"(f));
#else
  const float g = 1.0f / sqrtf(f);
#endif
  const int h = (int)(g * 1554944255988.0f);                       // 2^40.5
  unsigned none = 0;
  const fx e = sub(ONE, mul_full<55>(c2, shl(mad(h, h, 0), 3), none));    // 1 - 64 c^2 y^2
  const int es = (int)(e >> 10);
  const fx e2 = mad(es, es, 0) >> 41;
  const Op c = op(add(e >> 1, (3 * e2) >> 3));
  return add(shl((fx)h, 32), add(shl(mad(h, c.h, 0), 3), mad(h, c.l, 0) >> 29));
}

// ---------------------------------------------------------------- conversions
GRP_HD __forceinline__ int hiword(double x)
{
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  long long b;
  __builtin_memcpy(&b, &x, 8);
  return (int)(b >> 32);
#endif
}
GRP_HD __forceinline__ int loword(double x)
{
#ifdef __CUDA_ARCH__
  return __double2loint(x);
#else
  long long b;
  __builtin_memcpy(&b, &x, 8);
  return (int)b;
#endif
}
GRP_HD __forceinline__ double from_words(int h, int l)
{
#ifdef __CUDA_ARCH__
  return __hiloint2double(h, l);
#else
  const long long b = ((long long)h << 32) | (unsigned)l;
  double x;
  __builtin_memcpy(&x, &b, 8);
  return x;
#endif
}

// One component's scale 2^k: a double x becomes the integer x 2^k.  lo, hi:
// the high words below which x 2^k rounds to zero and from which it is 2^61
// or more.
struct Scale {
  int k20, lo, hi;
};
GRP_HD __forceinline__ Scale make_scale(int k)
{
  Scale s;
  s.k20 = (int)((unsigned)k << 20);
  const int lo = 1023 - 1 - k, hi = 1023 + 61 - k;          // exponent fields of 2^-1 and 2^61 units
  s.lo = lo < 1 ? 1 << 20 : lo << 20;
  s.hi = (hi > 2046 ? 2047 : hi < 1 ? 1 : hi) << 20;        // (infinities and NaN never pass)
  if (lo > 2046) s.lo = 2047 << 20;
  return s;
}
GRP_HD __forceinline__ fx to_fixed(double x, const Scale& s, bool& ok)
{
  const int h = hiword(x), a = h & 0x7fffffff;
  ok = ok && a < s.hi;
  const int hs = a >= s.lo ? (int)((unsigned)h + (unsigned)s.k20) : 0;
  const double y = from_words(hs, loword(x));
#ifdef __CUDA_ARCH__
  return __double2ll_rn(y);
#else
  return (fx)nearbyint(fabs(y) < 9e18 ? y : 0.0);
#endif
}
// 2^k as a double (k in the normal range)
GRP_HD __forceinline__ double pow2(int k) { return from_words((1023 + k) << 20, 0); }

// The range of gamma the bounds are worked out for (c^2 / V^2 within [1/64, 1)
// in subsonic flow).
GRP_HD inline bool gamma_ok(double g) { return g >= 1.2 && g <= 1.9; }
inline fx to_format(double x) { return (fx)ldexp(x, 61); }          // a constant below one, on the host

// ---------------------------------------------------------------------------
// The GRP of an interface with equal data g[1] on both sides, degree 2.
// q[0], q[1]: averages of the left and right cell; g[0], g[1], g[2]: the
// interface data left of the left cell, here, right of the right cell.
// dgm1: gamma - 1; gm1, hgam: gamma - 1 and gamma / 2 in the format.  Returns false, with no
// output, when the interface leaves the format's range or needs the general
// path (a sonic field, a state of the series near vacuum).
// ---------------------------------------------------------------------------
GRP_HD __forceinline__ bool grp_equal2(double dgm1, fx gm1, fx hgam, double nu, const double q[2][3], const double g[3][3],
                                       double F[3], double gnew[3])
{
  // ---- the interface's units
  const int hr = hiword(g[1][0]), hE = hiword(g[1][2]);
  const int xr = hr >> 20, xE = hE >> 20;                      // biased exponents (of positive numbers)
  bool ok = xr >= 1 && xr < 2046 && xE >= 1 && xE < 2046;
  // rho = r 2^er, r in [1/2, 1); E / rho = f 2^eq, f in [1/2, 1); V = 2^ev
  const int er = xr - 1022, eq = xE - xr + ((hE & 0xfffff) >= (hr & 0xfffff) ? 1 : 0), ev = (eq + 2) >> 1;
  const int sr = er + 2, sm = sr + ev, sE = sm + ev - 1;       // units 2^s of the three components
  ok = ok && sr > -400 && sr < 400 && ev > -150 && ev < 150;   // (every power of two below is a normal double)
  unsigned bad = 0;
  // ---- reconstruction of both cells: derivative coefficients of the traces,
  // b1 = gR - gL, b2 = 3 (gL + gR - 2 q); right edge b1 + b2, left edge b1 - b2
  fx Q0[3], L1[3], L2[3], R1[3], R2[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const Scale s = make_scale(61 - (c == 0 ? sr : c == 1 ? sm : sE));
    const fx ql = to_fixed(q[0][c], s, ok), qr = to_fixed(q[1][c], s, ok);
    const fx g0 = to_fixed(g[0][c], s, ok), g1 = to_fixed(g[1][c], s, ok), g2 = to_fixed(g[2][c], s, ok);
    Q0[c] = g1;
    const fx al = chk(sub(add(g0, g1), add(ql, ql)), bad, 60), ar = chk(sub(add(g1, g2), add(qr, qr)), bad, 60);
    L2[c] = chk(add(al, add(al, al)), bad, 60);
    R2[c] = chk(add(ar, add(ar, ar)), bad, 60);
    L1[c] = chk(add(sub(g1, g0), L2[c]), bad, 60);
    R1[c] = chk(sub(sub(g2, g1), R2[c]), bad, 60);
  }
  const fx r0 = Q0[0], m0 = Q0[1];
  // ---- the constant leading state
  const fx iv = recip32(r0);                                   // 1 / (32 rho)
  const fx u = mul_full<56>(m0, iv, bad);
  const fx mu0 = mul<61>(m0, u), p0 = mul<61>(gm1, sub(Q0[2], mu0));   // 2 p = (gamma - 1)(2 E - m u)
  const fx Ep0 = add(Q0[2], p0);
  bad |= p0 < (1ll << 20) ? 1u : 0u;
  // c^2 = gamma p / rho, kept at 1/64 or more: below that the flow is supersonic
  const fx c2p = mul_full<56>(mul<61>(hgam, p0), iv, bad);
  const fx c2 = c2p < (ONE >> 6) ? (ONE >> 6) : c2p;
  const fx y = rsqrt8(c2), cs = mul<58>(c2, y, bad);           // 1 / (8 c), c
  // ---- derivative Riemann problems: D = D_L - sum over the fields that take
  // right data of w r.  Subsonic flow takes one such field from the left (u > 0:
  // D = D_L - w_1 r_1) or its complement from the right (u < 0: D = D_R + w_3 r_3);
  // a resting contact averages both, supersonic flow takes a side whole.
  // Strengths w = (dp / c -+ rho du) / (2 c).
  const bool right = u < 0;
  const fx au = right ? sub(0, u) : u;
  // TIE (|u| + c), from the high word: TIE 2^32 = 1844674407 / 2^32
  const fx tie = (fx)(((unsigned long long)(unsigned)(int)(add(au, cs) >> 32) * 1844674407ull) >> 32);
  const fx gap = sub(au, cs);
  bad |= gap <= tie && gap >= -tie ? 1u : 0u;                  // a sonic field
  fx D[2][3];
#pragma unroll
  for (int c = 0; c < 3; ++c) { D[0][c] = right ? R1[c] : L1[c]; D[1][c] = right ? R2[c] : L2[c]; }
  if (gap < 0) {
    const fx k = mul<62>(u, u), H = mul_full<57>(Ep0, iv, bad), uc = mul<61>(au, cs);   // u^2 / 2, (E + p) / rho, |u| c
    const fx un = sub(0, u);
    const fx sc = right ? sub(0, cs) : cs;
    const bool rest = au <= tie;
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      fx J[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) J[c] = o == 0 ? sub(L1[c], R1[c]) : sub(L2[c], R2[c]);
      Dot dp;
      dp.mac(k, J[0]);
      dp.mac(un, J[1]);
      // the jumps of p / c and of rho times u, the latter towards the flow's side
      const fx Jp = mul<61>(gm1, chk(add(dp.value<61>(bad), J[2] >> 1), bad)), Jc = mul<58>(Jp, y, bad);
      const fx Jv = add(J[1], mul<61>(un, J[0], bad)), Ju = right ? sub(0, Jv) : Jv;
      // the field of speed |u| - c seen from the flow's side
      const fx w1 = mul<59>(chk(sub(Jc, Ju), bad), y, bad, 60), w = right ? sub(0, w1) : w1;
      D[o][0] = sub(D[o][0], w);
      D[o][1] = sub(D[o][1], mul<61>(w, sub(u, sc)));
      D[o][2] = sub(D[o][2], mul<60>(w, sub(H, uc), bad));
      if (rest) {                                              // and half of the other side, with its field
        const fx w3 = mul<59>(chk(add(Jc, Ju), bad), y, bad, 60), v = right ? w3 : sub(0, w3);
        fx B[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) B[c] = o == 0 ? (right ? L1[c] : R1[c]) : (right ? L2[c] : R2[c]);
        D[o][0] = add(D[o][0], sub(B[0], v)) >> 1;
        D[o][1] = add(D[o][1], sub(B[1], mul<61>(v, add(u, sc)))) >> 1;
        D[o][2] = add(D[o][2], sub(B[2], mul<60>(v, add(H, uc), bad))) >> 1;
      }
    }
  }
  // ---- Cauchy-Kovalevskaya series to degree 2: x-derivatives (1, 2), t (t), x t (x)
  const fx r1 = chk(D[0][0], bad), m1 = chk(D[0][1], bad), E1 = chk(D[0][2], bad);
  const fx r2 = chk(D[1][0], bad), m2 = chk(D[1][1], bad, 60), E2 = chk(D[1][2], bad);
  const fx u1 = mul_full<56>(chk(sub(m1, mul<61>(r1, u, bad)), bad), iv, bad);
  Dot d;
  d.mac(r2, u);
  d.mac(r1, u1);
  const fx u2 = mul_full<56>(chk(sub(m2, d.value<61>(bad)), bad), iv, bad);
  d = Dot();
  d.mac(m1, u);
  d.mac(m0, u1);
  const fx mu1 = d.value<61>(bad);
  d = Dot();
  d.mac(m2, u);
  d.mac(m1, u1);
  d.mac(m0, u2);
  const fx mu2 = d.value<61>(bad);
  const fx p1 = mul<61>(gm1, chk(sub(E1, mu1), bad)), p2 = mul<61>(gm1, chk(sub(E2, mu2), bad));
  const fx Ep1 = chk(add(E1, p1), bad), Ep2 = chk(add(E2, p2), bad);
  d = Dot();
  d.mac(u, Ep1);
  d.mac(u1, Ep0);
  const fx f1 = d.value<61>(bad);
  d = Dot();
  d.mac(u, Ep2);
  d.mac(u1, Ep1);
  d.mac(u2, Ep0);
  const fx f2 = d.value<61>(bad, 60);
  const fx h1 = chk(add(mu1, p1 >> 1), bad), h2 = chk(add(mu2, p2 >> 1), bad, 60);     // momentum flux
  const fx rt = sub(0, m1), mt = sub(0, h1), Et = sub(0, f1);
  const fx rx = sub(0, add(m2, m2)), mx = sub(0, add(h2, h2)), Ex = sub(0, add(f2, f2));
  const fx ut = mul_full<56>(chk(sub(mt, mul<61>(rt, u, bad)), bad), iv, bad);
  d = Dot();
  d.mac(mt, u);
  d.mac(m0, ut);
  const fx at = chk(sub(Et, d.value<61>(bad)), bad), Ept = chk(add(Et, mul<61>(gm1, at)), bad);
  d = Dot();
  d.mac(r1, ut);
  d.mac(rt, u1);
  d.mac(rx, u);
  const fx ux = mul_full<56>(chk(sub(mx, d.value<61>(bad)), bad), iv, bad);
  d = Dot();
  d.mac(m0, ux);
  d.mac(m1, ut);
  d.mac(mt, u1);
  d.mac(mx, u);
  const fx mux = d.value<61>(bad), px = mul<61>(gm1, chk(sub(Ex, mux), bad)), Epx = chk(add(Ex, px), bad);
  d = Dot();
  d.mac(u, Epx);
  d.mac(u1, Ept);
  d.mac(ut, Ep1);
  d.mac(ux, Ep0);
  const fx fxt = d.value<61>(bad), hx = chk(add(mux, px >> 1), bad);
  // ---- states at the two Gauss nodes and at dt: with y_k = s_k nu^k,
  // Q(1/2 -+ a) = s0 + y1 / 2 + y2 / 3 -+ a (y1 + y2), a^2 = 1/12
  const fx n4 = to_fixed(nu, make_scale(59 + ev), ok);         // nu V / 4
  const fx n16 = mul_full<61>(n4, n4, bad);                    // (nu V)^2 / 16
  constexpr fx THIRD = 768614336404564651ll, NODE = 665639541039271463ll;      // 1/3, 1/sqrt(12)
  const fx s1[3] = {rt, mt, Et}, s2[3] = {sub(0, mx) >> 1, sub(0, hx) >> 1, sub(0, fxt) >> 1};
  fx A[3], B[3], Z[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const fx y1 = mul_full<59>(s1[c], n4, bad), y2 = mul_full<57>(s2[c], n16, bad);
    const fx w = chk(add(y1, y2), bad), o = mul<61>(w, NODE);
    const fx mid = add(Q0[c], add(y1 >> 1, mul<61>(y2, THIRD)));
    A[c] = chk(sub(mid, o), bad, 60);
    B[c] = chk(add(mid, o), bad, 60);
    Z[c] = chk(add(Q0[c], w), bad, 60);
  }
  // densities in the range of the reciprocal
  const fx rlo = 1ll << 57, rhi = 1ll << 60;
  bad |= A[0] < rlo || A[0] >= rhi || B[0] < rlo || B[0] >= rhi ? 1u : 0u;
  const fx ua = mul_full<56>(A[1], recip32(A[0]), bad), ub = mul_full<56>(B[1], recip32(B[0]), bad);
  const fx ma = mul<61>(A[1], ua), mb = mul<61>(B[1], ub);
  const fx pa = mul<61>(gm1, chk(sub(A[2], ma), bad)), pb = mul<61>(gm1, chk(sub(B[2], mb), bad));
  bad |= pa < (1ll << 20) || pb < (1ll << 20) ? 1u : 0u;
  // admissible at dt: rho > 0 and 2 E rho - m^2 > 0
  d = Dot();
  d.mac(Z[2], Z[0]);
  d.mac(sub(0, Z[1]), Z[1]);
  bad |= Z[0] <= 0 || d.value<61>() < (1ll << 20) ? 1u : 0u;
  d = Dot();
  d.mac(ua, chk(add(A[2], pa), bad));
  d.mac(ub, chk(add(B[2], pb), bad));
  const fx f = d.value<61>(bad);
  if (!ok || bad) return false;
  // the nodes' weight 1/2 is in the powers of two
  F[0] = (double)add(A[1], B[1]) * pow2(sm - 62);
  F[1] = (double)add(add(ma, mb), add(pa, pb) >> 1) * pow2(sm + ev - 62);
  // Gas at rest: the momentum flux is the pressure alone.  Interfaces of equal
  // pressure have equal fluxes only if its rounding does not depend on their
  // units, so it is formed in FP64 (a resting contact stays at rest exactly).
  if ((A[1] | B[1]) == 0 && A[2] == Q0[2] && B[2] == Q0[2]) F[1] = dgm1 * g[1][2];
  F[2] = (double)f * pow2(sE + ev - 62);
  gnew[0] = (double)Z[0] * pow2(sr - 61);
  gnew[1] = (double)Z[1] * pow2(sm - 61);
  gnew[2] = (double)Z[2] * pow2(sE - 61);
  return true;
}

}  // namespace fixed
}  // namespace grp
