// The GRP at an interface in 64-bit fixed point, on the integer pipes: with equal
// data (degrees 2 and 4 of the linear reconstruction), and for gamma = 7/5 with a
// leading Riemann problem (degrees 1 and 3, GRPrecNL up to degree 3, and the
// interface problems of the DET solver, which are that problem alone).
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
// four and x = E/(rho V^2) in [1/8, 1/2) for the state that sets the units (the
// interface datum of equal data, otherwise the left cell's average or trace):
//   density  rho 2^-(er+2)          in [1/8, 1/4)   2^58..2^59 units
//   momentum rho V as unit of rho   |m| < rho
//   energy   2 E (twice the unit)   in [rho/4, rho) at least 2^56 units
//   velocity u / V                  |u| < 1
// A double of that state converts exactly (its last bit is worth 8 units or
// more), a product is off by at most 2 units (its low x low partial product is
// left out), so an operation's error is 2^-56 or less of the state where an FP64
// operation's is 2^-53.  Every operand of a product is tested against its bound,
// or bounded by tests before it, and an interface that leaves the range (a jump of
// more than about 4 between neighbours, sonic fields, sound slower than V/8, an
// iteration that has not converged, a state near vacuum or inadmissible) is solved
// in FP64 instead: by the second pass, or in place (DET).
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

// Range tests.  see<L>(x) collects the bits of the high word that differ from
// their neighbour; any of them at 2^L or above means |x| >= 2^L.  One word per
// bound (unused ones vanish), compared once at the end.
struct Guard {
  unsigned b[16];
  bool out;                                 // a test that is not a bound
  GRP_HD __forceinline__ Guard() : out(false)
  {
#pragma unroll
    for (int i = 0; i < 16; ++i) b[i] = 0;
  }
  template <int L>
  GRP_HD __forceinline__ void see(fx x)
  {
    static_assert(L > 46 && L < 62, "bound");
    const int h = (int)(x >> 32);
    b[61 - L] |= (unsigned)(h ^ (int)((unsigned)h << 1));
  }
  template <int L = 61>
  GRP_HD __forceinline__ fx chk(fx x) { see<L>(x); return x; }
  GRP_HD __forceinline__ bool bad() const
  {
    unsigned o = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) o |= b[i] & ~((2u << (61 - i - 32)) - 1u);
    return o != 0 || out;
  }
};

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
  // ... with the low x low partial product (first in the sum)
  GRP_HD __forceinline__ void mac_full(fx a, fx b)
  {
    const Op x = op(a), y = op(b);
    hi = mad(x.h, y.h, hi);
    mid = mad(x.h, y.l, mad(x.l, y.l, 0) >> 32);
    mid = mad(x.l, y.h, mid);
    n = 1;
  }
  // the sum / 2^S
  template <int S>
  GRP_HD __forceinline__ fx value() const { return fixed::add(shl(hi, 64 - S), mid >> (S - 32)); }
  // ... and a result of 2^L or more is seen
  template <int S, int L = 61>
  GRP_HD __forceinline__ fx value(Guard& g) const
  {
    g.see<L - (64 - S)>(hi);
    return value<S>();
  }
};

// one product / 2^S
template <int S>
GRP_HD __forceinline__ fx mul(fx a, fx b)
{
  Dot d;
  d.mac(a, b);
  return d.value<S>();
}
template <int S, int L = 61>
GRP_HD __forceinline__ fx mul(fx a, fx b, Guard& g)
{
  Dot d;
  d.mac(a, b);
  return d.value<S, L>(g);
}
// ... with the low x low partial product, for results shifted up
template <int S>
GRP_HD __forceinline__ fx mul_full(fx a, fx b)
{
  Dot d;
  d.mac_full(a, b);
  return d.value<S>();
}
template <int S, int L = 61>
GRP_HD __forceinline__ fx mul_full(fx a, fx b, Guard& g)
{
  Dot d;
  d.mac_full(a, b);
  return d.value<S, L>(g);
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
  const fx e = sub(ONE, mul_full<55>(c2, shl(mad(h, h, 0), 3)));   // 1 - 64 c^2 y^2
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
// An integer times 2^k, rounded to a double (0, or k in a range that keeps it
// normal).
GRP_HD __forceinline__ double to_double(fx x, int k)
{
  const double y = (double)x;
  const int h = hiword(y);
  return from_words(h == 0 ? 0 : h + (int)((unsigned)k << 20), loword(y));
}
// The range of gamma the bounds are worked out for (c^2 / V^2 within [1/64, 1)
// in subsonic flow).
GRP_HD inline bool gamma_ok(double g) { return g >= 1.3 && g <= 1.9; }
inline fx to_format(double x) { return (fx)ldexp(x, 61); }          // a constant below one, on the host

// The format's constants of a problem (host-built, in the kernel's arguments).
struct Consts {
  fx gm1, hgam;                              // gamma - 1, gamma / 2
};
inline Consts make_consts(double gamma)
{
  Consts c;
  c.gm1 = to_format(gamma - 1.0);
  c.hgam = to_format(0.5 * gamma);
  return c;
}

// Powers of two of an interface: units 2^s of the three components, V = 2^ev.
struct Units {
  int sr, sm, sE, ev;
};
GRP_HD __forceinline__ Units make_units(double rho, double E, bool& ok)
{
  const int hr = hiword(rho), hE = hiword(E);
  const int xr = hr >> 20, xE = hE >> 20;                      // biased exponents (of positive numbers)
  // rho = r 2^er, r in [1/2, 1); E / rho = f 2^eq, f in [1/2, 1)
  const int er = xr - 1022, eq = xE - xr + ((hE & 0xfffff) >= (hr & 0xfffff) ? 1 : 0);
  Units v;
  v.ev = (eq + 2) >> 1;
  v.sr = er + 2;
  v.sm = v.sr + v.ev;
  v.sE = v.sm + v.ev - 1;
  // (every power of two used is then that of a normal double)
  ok = ok && xr >= 1 && xr < 2046 && xE >= 1 && xE < 2046 && v.sr > -400 && v.sr < 400 && v.ev > -150 && v.ev < 150;
  return v;
}

// Reconstruction (linear GRPrec, Section 3.1) of a cell from q_{i-1}, q_i,
// q_{i+1}, g_{i-1/2}, g_{i+1/2} of one component: the Taylor coefficients
// t[0..M-1] of orders 1..M at its right (side = 1) or left (side = -1) edge, and
// at degrees 1 and 3 the values there (near) and at the other edge (far).
template <int M, int SIDE>
GRP_HD __forceinline__ void edge(fx qm, fx q, fx qp, fx gl, fx gr, fx t[M], Guard& G, fx* near_ = nullptr,
                                 fx* far_ = nullptr)
{
  const fx dg = sub(gr, gl), a = sub(add(gl, gr), add(q, q));
  if (M == 1) {
    const fx h = dg >> 1;
    t[0] = G.chk<60>(dg);
    *near_ = SIDE > 0 ? add(q, h) : sub(q, h);
    *far_ = SIDE > 0 ? sub(q, h) : add(q, h);
  } else if (M == 2) {
    // b1 = dg, b2 = 3 a; orders 1, 2 at the edge: b1 +- b2, b2
    const fx b2 = add(G.chk<58>(a), add(a, a));
    t[0] = G.chk<60>(SIDE > 0 ? add(dg, b2) : sub(dg, b2));
    t[1] = b2;
  } else {
    const fx dq = sub(qp, qm), d2 = sub(add(qm, qp), add(q, q));
    G.see<58>(dg); G.see<58>(a); G.see<58>(dq); G.see<58>(d2);
    // b1 = (10 dg - dq) / 8, b3 = dq / 2 - dg
    const fx b1 = sub(10 * dg, dq) >> 3, b3 = sub(dq >> 1, dg), s3 = SIDE > 0 ? b3 : sub(0, b3);
    if (M == 3) {
      // b2 = 3 (a + 6 d2) / 37
      constexpr fx C337 = 186960243990299510ll, C6 = 384307168202282325ll;      // 3/37, 1/6
      const fx b2 = mul<61>(add(a, 6 * d2), C337), s2 = SIDE > 0 ? b2 : sub(0, b2);
      const fx even = add(q, mul<61>(b2, C6)), odd = add(b1 >> 1, b3 >> 3);
      *near_ = SIDE > 0 ? add(even, odd) : sub(even, odd);
      *far_ = SIDE > 0 ? sub(even, odd) : add(even, odd);
      t[0] = G.chk<60>(add(add(b1, s2), (3 * b3) >> 2));
      t[1] = G.chk<60>(add(b2, (3 * s3) >> 1));
      t[M - 1] = G.chk<60>(b3);
    } else {
      // b2 = (30 a - d2) / 8, b4 = -5 (6 a - d2) / 12
      constexpr fx C512 = 960767920505705813ll;                 // 5/12
      const fx b2 = sub(30 * a, d2) >> 3, b4 = sub(0, mul<61>(sub(6 * a, d2), C512));
      const fx s2 = SIDE > 0 ? b2 : sub(0, b2), s4 = SIDE > 0 ? b4 : sub(0, b4);
      // in twice the length (order k times 2^k), which keeps the rounding of the
      // high orders from growing with (nu V)^k
      t[0] = shl(G.chk<59>(add(add(b1, s2), add((3 * b3) >> 2, s4 >> 1))), 1);
      t[M > 1 ? 1 : 0] = shl(G.chk<58>(add(b2, (3 * add(s3, b4)) >> 1)), 2);
      t[M > 2 ? 2 : 0] = shl(G.chk<57>(add(b3, add(s4, s4))), 3);
      t[M - 1] = shl(G.chk<56>(b4), 4);
    }
  }
}

// The constant leading state of an interface and what its derivative Riemann
// problems need of it.
struct State {
  fx Q[3];                     // rho, m, 2 E
  fx iv, u, p, Ep, c, y;       // 1/(32 rho), velocity, 2 p, 2 (E + p), sound speed, 1/(8 c)
};
// ... the velocity and pressure of its conserved values.  In the state's own units
// an admissible one has |u| < 1 (m^2 < 2 E rho); FOREIGN: in units that may be
// another state's, and not known to be admissible, the product is tested before it
// can wrap (|m| < 1/2 and rho >= 1/16 leave |u| up to 8).
template <bool FOREIGN>
GRP_HD __forceinline__ void primitive(const Consts& K, State& w, Guard& G)
{
  w.iv = recip32(w.Q[0]);
  w.u = FOREIGN ? mul_full<56>(w.Q[1], w.iv, G) : mul_full<56>(w.Q[1], w.iv);
  w.p = mul<61>(K.gm1, sub(w.Q[2], mul<61>(w.Q[1], w.u)));      // 2 p = (gamma - 1)(2 E - m u)
}
// ... the rest, from those
GRP_HD __forceinline__ void acoustic(const Consts& K, State& w, Guard& G)
{
  w.Ep = add(w.Q[2], w.p);
  G.out = G.out || w.p < (1ll << 20);
  // c^2 = gamma p / rho, kept at 1/64 or more.  In the state's own units the flow is
  // supersonic below that (|u| > 0.4), and takes a side whole; in another state's (the
  // star state of an expansion in those of its left trace) it need not be, and is left
  const fx c2 = mul_full<56>(mul<61>(K.hgam, w.p), w.iv, G), lo = ONE >> 6;
  G.out = G.out || (c2 < lo && w.u < (ONE >> 3) && w.u > -(ONE >> 3));
  const fx c2l = c2 < lo ? lo : c2;
  w.y = rsqrt8(c2l);
  w.c = mul<58>(c2l, w.y);
}

// Derivative Riemann problems (Section 2): D = D_L - sum over the fields that
// take right data of w r.  Subsonic flow takes one such field from the left
// (u > 0: D = D_L - w_1 r_1) or its complement from the right (u < 0:
// D = D_R + w_3 r_3); a resting contact averages both, supersonic flow takes a
// side whole.  Strengths w = (dp / c -+ rho du) / (2 c).  A sonic field is left
// to the general path.
template <int M>
GRP_HD __forceinline__ void derivatives(const Consts& K, const State& s, const fx L[M][3], const fx R[M][3],
                                        fx D[M][3], Guard& G)
{
  const fx u = s.u, cs = s.c, y = s.y;
  const bool right = u < 0;
  const fx au = right ? sub(0, u) : u;
  // TIE (|u| + c), from the high word: TIE 2^32 = 1844674407 / 2^32
  const fx tie = (fx)(((unsigned long long)(unsigned)(int)(add(au, cs) >> 32) * 1844674407ull) >> 32);
  const fx gap = sub(au, cs);
  G.out = G.out || (gap <= tie && gap >= -tie);
#pragma unroll
  for (int o = 0; o < M; ++o)
#pragma unroll
    for (int c = 0; c < 3; ++c) D[o][c] = right ? R[o][c] : L[o][c];
  if (gap < 0) {
    const fx k = mul<62>(u, u), H = mul_full<57>(s.Ep, s.iv), uc = mul<61>(au, cs);   // u^2/2, (E+p)/rho, |u| c
    const fx un = sub(0, u), sc = right ? sub(0, cs) : cs;
    const bool rest = au <= tie;
#pragma unroll
    for (int o = 0; o < M; ++o) {
      fx J[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) J[c] = sub(L[o][c], R[o][c]);
      Dot dp;
      dp.mac(k, J[0]);
      dp.mac(un, J[1]);
      // the jumps of p / c and of rho times u, the latter towards the flow's side
      const fx Jp = mul<61>(K.gm1, G.chk(add(dp.value<61>(), J[2] >> 1))), Jc = mul<58>(Jp, y, G);
      const fx Jv = add(J[1], mul<61>(un, J[0])), Ju = right ? sub(0, Jv) : Jv;
      // the field of speed |u| - c seen from the flow's side
      const fx w1 = mul<59, 60>(G.chk(sub(Jc, Ju)), y, G), w = right ? sub(0, w1) : w1;
      D[o][0] = sub(D[o][0], w);
      D[o][1] = sub(D[o][1], mul<61>(w, sub(u, sc)));
      D[o][2] = sub(D[o][2], mul<60>(w, sub(H, uc)));
      if (rest) {                                              // and half of the other side, with its field
        const fx w3 = mul<59, 60>(G.chk(add(Jc, Ju)), y, G), v = right ? w3 : sub(0, w3);
        fx B[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) B[c] = right ? L[o][c] : R[o][c];
        D[o][0] = add(D[o][0], sub(B[0], v)) >> 1;
        D[o][1] = add(D[o][1], sub(B[1], mul<61>(v, add(u, sc)))) >> 1;
        D[o][2] = add(D[o][2], sub(B[2], mul<60, 61>(v, add(H, uc), G))) >> 1;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Leading Riemann problem, gamma = 7/5, of data without strong waves.  The star
// velocity is the unknown: with d the velocity by which the gas of a side is
// pulled away from it, its pressure is p_K (1 - d / (5 c))^7 through a rarefaction
// (d > 0), and p_K + rho |d| w, w = 0.6 |d| + sqrt(0.36 d^2 + c^2) the speed of
// the shock into the side, otherwise: no roots but that one.  Three steps of
// Newton's iteration in FP32 leave about 2^-21; two steps follow with the pressures
// in the format and the FP32 slopes of the last point, which are off by 2^-20 and by
// a few times the first of these steps.  That one is held below 2^-16 and the second
// below 2^-40, so what is left is below 2^-53, and 2^-57 once FP32 has converged.
// (Slopes of the point before the last, and no bound of the second step, left up to
// 4e-8 of the state.)
// ---------------------------------------------------------------------------
GRP_HD __forceinline__ float to_f32(fx x) { return (float)x * 0x1p-61f; }

struct Side32 { float p, r, c, i5c; };                          // 2 p, rho, c, 1/(5 c)
GRP_HD __forceinline__ float pressure32(const Side32& s, float d, float& k)
{
  const float q = fmaf(-d, s.i5c, 1.0f), q2 = q * q, q6 = q2 * q2 * q2;
  const float aD = -0.6f * d, sq = sqrtf(fmaf(aD, aD, s.c * s.c)), w = aD + sq, r2 = s.r + s.r;
  k = d > 0.0f ? r2 * s.c * q6 : r2 * w * w / sq;
  return d > 0.0f ? s.p * q6 * q : fmaf(-r2 * d, w, s.p);
}

// 2 p of a side at d; i10c = 1/(10 c)
GRP_HD __forceinline__ fx pressure(const State& s, fx c2, fx i10c, fx d, Guard& G)
{
  if (d > 0) {
    const fx q = sub(ONE, mul<60>(d, i10c)), q2 = mul<61>(q, q), q4 = mul<61>(q2, q2);
    return mul<61>(s.p, mul<61>(mul<61>(q4, q2), q));
  }
  constexpr fx C06 = 1383505805528216371ll;                      // 0.6
  const fx D = sub(0, d), aD = mul<61>(D, C06);
  const fx s2 = G.chk(add(mul<61>(aD, aD), c2)), w = G.chk(add(aD, mul<58>(s2, rsqrt8(s2))));
  return add(s.p, mul<60>(s.Q[0], mul<61>(D, w)));
}

// The Godunov state of L | R at x / t = 0 into w (Q, u, p).  L and R hold the
// conserved values; their other members are formed here.
GRP_HD __forceinline__ void riemann(const Consts& K, State& L, State& R, State& w, Guard& G)
{
  primitive<true>(K, L, G);
  primitive<true>(K, R, G);
  const bool equal = L.Q[0] == R.Q[0] && L.Q[1] == R.Q[1] && L.Q[2] == R.Q[2];
  fx c2[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    State& s = k ? R : L;
    G.out = G.out || s.Q[0] < (1ll << 57) || s.Q[0] >= (1ll << 60);
    c2[k] = mul_full<56, 61>(mul<61>(K.hgam, s.p), s.iv, G);
    // slower sound than 1/8: general path, unless there is no wave
    G.out = G.out || s.p < (1ll << 20) || (c2[k] < (ONE >> 6) && !equal);
    c2[k] = c2[k] < (ONE >> 6) ? (ONE >> 6) : c2[k];
    s.y = rsqrt8(c2[k]);
    s.c = mul<58>(c2[k], s.y);
  }
  constexpr fx C08 = 1844674407370955162ll;                      // 0.8
  const fx iL = mul<61>(L.y, C08), iR = mul<61>(R.y, C08);       // 1/(10 c)
  // FP32, from the acoustic estimate
  const fx du = G.chk(sub(R.u, L.u));
  const float fdu = to_f32(du);
  const Side32 l = {to_f32(L.p), to_f32(L.Q[0]), to_f32(L.c), 2.0f * to_f32(iL)};
  const Side32 r = {to_f32(R.p), to_f32(R.Q[0]), to_f32(R.c), 2.0f * to_f32(iR)};
  const float zl = 2.0f * l.r * l.c, zr = 2.0f * r.r * r.c;
  float x = fmaf(zr, fdu, to_f32(sub(L.p, R.p))) / (zl + zr), kl = zl, kr = zr;      // u* - u_L
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float pl = pressure32(l, x, kl), pr = pressure32(r, fdu - x, kr);
    x += (pl - pr) / (kl + kr);
  }
  pressure32(l, x, kl);                                          // the slopes there
  pressure32(r, fdu - x, kr);
  // the side's gas must stay away from vacuum (q > 1/2) and the iteration finite
  G.out = G.out || !(x * l.i5c < 0.5f && (fdu - x) * r.i5c < 0.5f && fabsf(x) < 0.5f && fabsf(fdu - x) < 0.5f);
  const float xs = fabsf(x) < 0.5f ? x : 0.0f;
  fx d = (fx)(xs * 0x1p61f);
  const float inv = 1.0f / (kl + kr);
  const fx g1 = sub(pressure(L, c2[0], iL, d, G), pressure(R, c2[1], iR, sub(du, d), G));
  // a step of 2^-16 or more: FP32 did not converge
  const float s1 = to_f32(g1) * inv;
  G.out = G.out || !(fabsf(s1) < 0x1p-16f);
  d = add(d, (fx)(fabsf(s1) < 0x1p-16f ? s1 * 0x1p61f : 0.0f));
  const fx pl = pressure(L, c2[0], iL, d, G), pr = pressure(R, c2[1], iR, sub(du, d), G);
  const float s2 = to_f32(sub(pl, pr)) * inv;
  // the last step along the tangents; p* from both sides alike, so that a mirrored
  // problem in the same units gives the mirrored state.  (The units are the left
  // side's: the mirror image of an interface agrees to the format's rounding, and
  // near the bounds one of the two may be left to FP64 alone.)
  G.out = G.out || !(fabsf(s2) < 0x1p-40f);
  const float t2 = fabsf(s2) < 0x1p-40f ? s2 : 0.0f;
  const fx ps = add(add(pl >> 1, pr >> 1), (fx)(0.5f * (kr - kl) * t2 * 0x1p61f));
  d = add(d, (fx)(t2 * 0x1p61f));
  const fx us = add(L.u, d);
  // ---- the state at x / t = 0: the side of the contact, mirrored to the left
  const fx cc = add(L.c, R.c);
  const fx tie = (fx)(((unsigned long long)(unsigned)(int)(cc >> 32) * 1844674407ull) >> 32);
  const bool right = us < sub(0, tie);
  const State& k = right ? R : L;
  const fx dk = right ? sub(du, d) : d, i10c = right ? iR : iL, ck2 = right ? c2[1] : c2[0];
  const fx uk = right ? sub(0, k.u) : k.u, um = right ? sub(0, us) : us;
  fx rho;
  bool own;
  if (dk > 0) {
    const fx q = sub(ONE, mul<60>(dk, i10c)), q2 = mul<61>(q, q);
    rho = mul<61>(k.Q[0], mul<61>(mul<61>(q2, q2), q));
    own = uk >= k.c;                                             // the head moves away
    const fx tail = sub(um, mul<61>(k.c, q));
    G.out = G.out || (!own && !equal && tail >= 0);              // x = 0 inside the fan
  } else {
    constexpr fx C06 = 1383505805528216371ll;
    const fx D = sub(0, dk), aD = mul<61>(D, C06), s2 = G.chk(add(mul<61>(aD, aD), ck2));
    const fx wk = add(aD, mul<58>(s2, rsqrt8(s2))), m = sub(wk, D);
    G.out = G.out || ((m < (1ll << 57) || m >= (1ll << 60)) && !equal);
    const fx j = mul<61>(k.Q[0], wk);                            // rho* = rho w / (w - D)
    rho = equal ? k.Q[0] : mul_full<56, 60>(j, recip32(m), G);
    own = uk >= wk;
  }
  // a side's own state, and equal data, as they are
  own = own || equal;
  constexpr fx C58 = 1441151880758558720ll;                      // 5/8
  const fx m = mul<61>(rho, us);
  w.Q[0] = own ? k.Q[0] : rho;
  w.Q[1] = own ? k.Q[1] : m;
  w.Q[2] = own ? k.Q[2] : add(mul<59>(ps, C58), mul<61>(m, us));
  w.u = own ? k.u : us;
  w.p = own ? k.p : ps;
  G.see<60>(w.Q[2]);
  G.see<61>(w.u);
  G.out = G.out || w.Q[0] < (1ll << 57) || w.Q[0] >= (1ll << 60);
  w.iv = recip32(w.Q[0]);
}

// Cauchy-Kovalevskaya series in time at the interface from its x-derivatives
// D[k - 1] of order k = 1..M: s[b][c] of T^b, b = 1..M, with the scheme of
// ck_euler.  Operands are kept below one, x-derivatives below 1/2.
template <int M>
GRP_HD __forceinline__ void series(const Consts& K, const State& w, const fx D[M][3], fx s[M][3], Guard& G)
{
  using T = Tri<M>;
  fx r[T::N], m[T::N], E[T::N], u[T::N], Ep[T::N];
  r[0] = w.Q[0]; m[0] = w.Q[1]; E[0] = w.Q[2]; u[0] = w.u; Ep[0] = w.Ep;
#pragma unroll
  for (int k = 1; k <= M; ++k) {
    const int i = T::idx(k, 0);
    r[i] = G.chk<60>(D[k - 1][0]); m[i] = G.chk<60>(D[k - 1][1]); E[i] = G.chk<60>(D[k - 1][2]);
  }
#pragma unroll
  for (int b = 0; b < M; ++b) {
#pragma unroll
    for (int a = 0; a + b <= M; ++a) {
      const int k = T::idx(a, b);
      if (k == 0) continue;
      Dot du;
#pragma unroll
      for (int i = 0; i <= a; ++i)
#pragma unroll
        for (int j = 0; j <= b; ++j)
          if (i || j) du.mac(r[T::idx(i, j)], u[T::idx(a - i, b - j)]);
      u[k] = mul_full<56>(G.chk(sub(m[k], du.value<61>(G))), w.iv, G);
      Dot dm;
#pragma unroll
      for (int i = 0; i <= a; ++i)
#pragma unroll
        for (int j = 0; j <= b; ++j) dm.mac(m[T::idx(i, j)], u[T::idx(a - i, b - j)]);
      const fx mu = dm.value<61>(G), p = mul<61>(K.gm1, G.chk(sub(E[k], mu)));
      Ep[k] = G.chk(add(E[k], p));
      if (a >= 1) {
        // q[a - 1][b + 1] = -(a / (b + 1)) F[a][b]
        Dot df;
#pragma unroll
        for (int i = 0; i <= a; ++i)
#pragma unroll
          for (int j = 0; j <= b; ++j) df.mac(u[T::idx(i, j)], Ep[T::idx(a - i, b - j)]);
        const int dst = T::idx(a - 1, b + 1);
        constexpr fx THIRD = 768614336404564651ll;
        const fx f[3] = {m[k], add(mu, p >> 1), df.value<61>(G)};
        fx q[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          fx v = f[c];
          if (a == 2) { v = G.chk<60>(v); v = add(v, v); }
          if (a == 3) { v = G.chk<59>(v); v = add(v, add(v, v)); }
          if (a == 4) { v = G.chk<59>(v); v = shl(v, 2); }
          if (b == 1) v = v >> 1;
          if (b == 2) v = mul<61>(G.chk(v), THIRD);
          if (b == 3) v = v >> 2;
          q[c] = G.chk(sub(0, v));
        }
        r[dst] = q[0]; m[dst] = q[1]; E[dst] = q[2];
      }
    }
  }
#pragma unroll
  for (int b = 1; b <= M; ++b) { s[b - 1][0] = r[T::idx(0, b)]; s[b - 1][1] = m[T::idx(0, b)]; s[b - 1][2] = E[T::idx(0, b)]; }
}

// The flux of a state at a Gauss node: f[1] = m u + p, f[2] = 2 u (E + p).
GRP_HD __forceinline__ void node_flux(const Consts& K, const fx A[3], fx& f1, fx& f2, Guard& G)
{
  G.out = G.out || A[0] < (1ll << 57) || A[0] >= (1ll << 60);   // the reciprocal's range
  const fx u = mul_full<56>(A[1], recip32(A[0]), G), mu = mul<61>(A[1], u);
  const fx p = mul<61>(K.gm1, G.chk(sub(A[2], mu)));
  G.out = G.out || p < (1ll << 20);
  f1 = add(mu, p >> 1);
  f2 = mul<61>(u, G.chk(add(A[2], p)));
}

// ---------------------------------------------------------------------------
// The GRP from its leading state w and the traces' derivative coefficients L, R:
// the flux and the datum at dt.  still_p: gamma - 1 times the total energy, the
// pressure of gas at rest in FP64 (see below).  false: out of range, no output.
// ---------------------------------------------------------------------------
template <int M>
GRP_HD __forceinline__ bool evolve(const Consts& K, const Units& v, State& w, const fx L[M][3], const fx R[M][3],
                                   double nu, double still_p, Guard& G, bool ok, double F[3], double gnew[3])
{
  acoustic(K, w, G);
  fx D[M][3], s[M][3];
  derivatives<M>(K, w, L, R, D, G);
  series<M>(K, w, D, s, G);
  // ---- states at the Gauss nodes and at dt
  const fx n4 = to_fixed(nu, make_scale(59 + v.ev), ok);        // nu V / 4
  constexpr int NG = Gauss<M>::G;
  fx A[NG][3], Z[3];
  if (NG <= 2 && M <= 2) {
    // with y_k = s_k nu^k: Q(1/2 -+ a) = s0 + y1 / 2 + y2 / 3 -+ a (y1 + y2), a^2 = 1/12 (degree 1: the midpoint)
    const fx n16 = mul_full<61>(n4, n4);                        // (nu V)^2 / 16
    constexpr fx THIRD = 768614336404564651ll, NODE = 665639541039271463ll;      // 1/3, 1/sqrt(12)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const fx y1 = mul_full<59, 60>(s[0][c], n4, G);
      if (M == 1) {
        A[0][c] = add(w.Q[c], y1 >> 1);
        Z[c] = add(w.Q[c], y1);
        continue;
      }
      const fx y2 = mul_full<57, 60>(s[M - 1][c], n16, G);
      const fx t = add(y1, y2), o = mul<61>(t, NODE), mid = add(w.Q[c], add(y1 >> 1, mul<61>(y2, THIRD)));
      A[0][c] = sub(mid, o);
      A[NG - 1][c] = add(mid, o);
      Z[c] = add(w.Q[c], t);
    }
  } else {
    // Horner's rule at the nodes and at dt, in T / 4 (degree 4: T / 2, of twice
    // the length: twice the time)
    constexpr fx H = 1ll << 60, N2 = 665639541039271463ll, N30 = 259872347241503775ll, N32 = 2045970661972190177ll;
#pragma unroll
    for (int al = 0; al <= NG; ++al) {
      const fx node = M == 3 ? (al == 0 ? H - N2 : H + N2) : (al == 0 ? N30 : al == 1 ? H : N32);   // 1/2 -+ 1/sqrt(12), sqrt(0.15)
      const fx t = al == NG ? n4 : mul_full<61>(n4, node);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        fx x = s[M - 1][c];
#pragma unroll
        for (int k = M - 2; k >= 0; --k) x = G.chk(add(s[k][c], mul_full<M == 3 ? 59 : 60>(x, t, G)));
        x = G.chk(add(w.Q[c], mul_full<M == 3 ? 59 : 60>(x, t, G)));
        if (al == NG) Z[c] = x;
        else A[al][c] = x;
      }
    }
  }
  fx f1[NG], f2[NG];
  bool still = true;                                            // gas at rest (below)
#pragma unroll
  for (int al = 0; al < NG; ++al) {
    node_flux(K, A[al], f1[al], f2[al], G);
    still = still && A[al][1] == 0 && A[al][2] == w.Q[2];
  }
  // admissible at dt: rho > 0 and 2 E rho - m^2 > 0
  Dot d;
  d.mac(G.chk(Z[2]), G.chk(Z[0]));
  d.mac(sub(0, G.chk(Z[1])), Z[1]);
  G.out = G.out || Z[0] <= 0 || d.value<61>() < (1ll << 20);
  if (!ok || G.bad()) return false;
  if (M == 4) {
    constexpr fx W0 = 640511947003803876ll, W1 = 1024819115206086201ll;              // 5/18, 4/9
    constexpr int MID = NG / 2;
    F[0] = to_double(add(add(mul<61>(A[0][1], W0), mul<61>(A[MID][1], W1)), mul<61>(A[NG - 1][1], W0)), v.sm - 61);
    F[1] = to_double(add(add(mul<61>(f1[0], W0), mul<61>(f1[MID], W1)), mul<61>(f1[NG - 1], W0)), v.sm + v.ev - 61);
    F[2] = to_double(add(add(mul<61>(f2[0], W0), mul<61>(f2[MID], W1)), mul<61>(f2[NG - 1], W0)), v.sE + v.ev - 61);
  } else {
    // one node, or two whose weight 1/2 is in the powers of two
    constexpr int E = NG == 1 ? 61 : 62;
    F[0] = to_double(NG == 1 ? A[0][1] : add(A[0][1], A[NG - 1][1]), v.sm - E);
    F[1] = to_double(NG == 1 ? f1[0] : add(f1[0], f1[NG - 1]), v.sm + v.ev - E);
    F[2] = to_double(NG == 1 ? f2[0] : add(f2[0], f2[NG - 1]), v.sE + v.ev - E);
  }
  // Gas at rest: the momentum flux is the pressure alone.  Interfaces of equal
  // pressure have equal fluxes only if its rounding does not depend on their
  // units, so it is formed in FP64 (a resting contact stays at rest exactly).
  if (still) F[1] = still_p;
  gnew[0] = to_double(Z[0], v.sr - 61);
  gnew[1] = to_double(Z[1], v.sm - 61);
  gnew[2] = to_double(Z[2], v.sE - 61);
  return true;
}

// ---------------------------------------------------------------------------
// The GRP of an interface from the averages q of the cells around it (degrees 1
// and 2: left and right; 3 and 4: with the cells beyond) and the interface data
// g[0], g[1], g[2] left of the left cell, here, right of the right cell.  dgm1:
// gamma - 1.  Degrees 2 and 4: equal data g[1] on both sides.  Degrees 1 and 3
// (gamma = 7/5): the leading Riemann problem of the two traces; the cells must
// keep their polynomials (admissible at both edges).  Returns false, with no
// output, when the interface leaves the format's range or needs the general path
// (strong waves, a sonic field or fan, a state near vacuum).  newton: whether the
// traces differ.
// ---------------------------------------------------------------------------
template <int M>
GRP_HD __forceinline__ bool grp_linear(const Consts& K, double dgm1, double nu, const double q[M <= 2 ? 2 : 4][3],
                                       const double g[3][3], double F[3], double gnew[3], bool& newton)
{
  constexpr bool EQ = M == 2 || M == 4;
  constexpr int NQ = M <= 2 ? 2 : 4, IL = M <= 2 ? 0 : 1;        // the left cell's place
  bool ok = true;
  Guard G;
  const Units v = EQ ? make_units(g[1][0], g[1][2], ok) : make_units(q[IL][0], q[IL][2], ok);
  State w;
  fx L[M][3], R[M][3], nl[3], fl[3], nr[3], fr[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const Scale s = make_scale(61 - (c == 0 ? v.sr : c == 1 ? v.sm : v.sE));
    fx x[NQ], y[3], tl[M], tr[M];
#pragma unroll
    for (int k = 0; k < NQ; ++k) x[k] = to_fixed(q[k][c], s, ok);
#pragma unroll
    for (int k = 0; k < 3; ++k) y[k] = to_fixed(g[k][c], s, ok);
    w.Q[c] = y[1];
    edge<M, 1>(x[0], x[IL], x[NQ - 1 - IL], y[0], y[1], tl, G, &nl[c], &fl[c]);
    edge<M, -1>(x[IL], x[IL + 1], x[NQ - 1], y[1], y[2], tr, G, &nr[c], &fr[c]);
#pragma unroll
    for (int k = 0; k < M; ++k) { L[k][c] = tl[k]; R[k][c] = tr[k]; }
  }
  newton = false;
  double still_p;
  if (EQ) {
    primitive<false>(K, w, G);
    still_p = dgm1 * g[1][2];
  } else {
    // admissible at the far edges (rho > 0, 2 E rho - m^2 > 0); at the near ones the Riemann problem sees to it
    Dot dl, dr;
    dl.mac(G.chk(fl[2]), G.chk(fl[0]));
    dl.mac(sub(0, G.chk(fl[1])), fl[1]);
    dr.mac(G.chk(fr[2]), G.chk(fr[0]));
    dr.mac(sub(0, G.chk(fr[1])), fr[1]);
    G.out = G.out || fl[0] <= 0 || fr[0] <= 0 || dl.value<61>() < (1ll << 20) || dr.value<61>() < (1ll << 20);
    State a, b;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      a.Q[c] = G.chk<60>(nl[c]);
      b.Q[c] = G.chk<60>(nr[c]);
    }
    newton = !(nl[0] == nr[0] && nl[1] == nr[1] && nl[2] == nr[2]);
    riemann(K, a, b, w, G);
    still_p = dgm1 * to_double(w.Q[2], v.sE - 61);
  }
  return evolve<M>(K, v, w, L, R, nu, still_p, G, ok, F, gnew);
}

// The same from traces given as Taylor coefficients tL, tR in FP64 (gamma = 7/5;
// degrees 1 to 3).
template <int M>
GRP_HD __forceinline__ bool grp_traces(const Consts& K, double dgm1, double nu, const double tL[3][M + 1],
                                       const double tR[3][M + 1], double F[3], double gnew[3], bool& newton)
{
  bool ok = true;
  Guard G;
  const Units v = make_units(tL[0][0], tL[2][0], ok);
  State w, a, b;
  fx L[M][3], R[M][3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const Scale s = make_scale(61 - (c == 0 ? v.sr : c == 1 ? v.sm : v.sE));
    a.Q[c] = G.chk<60>(to_fixed(tL[c][0], s, ok));
    b.Q[c] = G.chk<60>(to_fixed(tR[c][0], s, ok));
#pragma unroll
    for (int k = 1; k <= M; ++k) {
      L[k - 1][c] = G.chk<60>(to_fixed(tL[c][k], s, ok));
      R[k - 1][c] = G.chk<60>(to_fixed(tR[c][k], s, ok));
    }
  }
  newton = !(a.Q[0] == b.Q[0] && a.Q[1] == b.Q[1] && a.Q[2] == b.Q[2]);
  riemann(K, a, b, w, G);
  return evolve<M>(K, v, w, L, R, nu, dgm1 * to_double(w.Q[2], v.sE - 61), G, ok, F, gnew);
}

// Godunov state Q0 and its flux F of QL | QR in FP64 (gamma = 7/5).  false: outside
// the format's range (inadmissible data among it), nothing to be used.
GRP_HD __forceinline__ bool riemann_flux(const Consts& K, double dgm1, const double QL[3], const double QR[3],
                                         double Q0[3], double F[3], bool& newton)
{
  bool ok = true;
  Guard G;
  const Units v = make_units(QL[0], QL[2], ok);
  State w, a, b;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const Scale s = make_scale(61 - (c == 0 ? v.sr : c == 1 ? v.sm : v.sE));
    a.Q[c] = G.chk<60>(to_fixed(QL[c], s, ok));
    b.Q[c] = G.chk<60>(to_fixed(QR[c], s, ok));
  }
  newton = !(a.Q[0] == b.Q[0] && a.Q[1] == b.Q[1] && a.Q[2] == b.Q[2]);
  riemann(K, a, b, w, G);
  Q0[0] = to_double(w.Q[0], v.sr - 61);
  Q0[1] = to_double(w.Q[1], v.sm - 61);
  Q0[2] = to_double(w.Q[2], v.sE - 61);
  const double u = to_double(w.u, v.ev - 61);
  // (at rest the pressure must not depend on the interface's units)
  const double ps = w.u == 0 ? dgm1 * Q0[2] : to_double(w.p, v.sE - 61);
  F[0] = Q0[1];
  F[1] = fma(Q0[1], u, ps);
  F[2] = u * (Q0[2] + ps);
  return ok && !G.bad();
}

}  // namespace fixed
}  // namespace grp
