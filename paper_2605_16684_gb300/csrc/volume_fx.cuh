// volume_fx.cuh -- the FP64 path's two-point pair in 60-bit fixed point.
//
// What bounds the FP64 volume kernel is the FP64 pipe: it takes one lane's
// instruction every half cycle and SM (64 cycles for a warp on its quarter of
// the SM), while an integer multiply-add of 32 x 32 + 64 bits takes a warp two
// cycles and an addition one (throughput loops on this GPU).  The 61 FP64
// instructions of a pair cost a warp 3900 cycles; the same pair in two-limb
// fixed point, about 350 integer instructions, costs 640.  The node fields of
// an element are scaled by powers of two to the element's own largest values
// and held as value = h 2^30 + l, and the pair pass runs on the integer pipes.
//
// A common scale holds a value of the largest size to 2^-59, six bits finer than an FP64
// significand, and a smaller one to as many bits less as it is smaller.  What one sum adds
// up therefore has to be of one size: the components of the metric and of the velocity
// have a scale each, stretched against one another so that u_c Ja^d_c keeps its value
// (metric_stretch).  With one scale for all, an element of 100 km x 100 km x 20 m lost
// three digits of its horizontal fluxes.  The geopotential is relative to the element's
// first node (the energy's interface terms as well; the kernel restores it from the mass
// sum), and the pressure's scale stands above the energies' where they are much larger
// (FxScale::dp): gamma near 1 and meshes far above z = 0 lost up to five bits of it.
// Right-hand side without dissipation against long double, error over that of the FP64
// pair by variable, N = 2 to 7: cubes to 100 m/s 0.4 to 0.95, boxes of 1:1 to 1:1e5 0.4 to
// 0.96, elements of 3 to 11 km 0.4 to 1.1, gamma 1.05 to 2 0.4 to 0.95, a mesh 10 to
// 1000 km above z = 0 0.4 to 1.0; N = 1 up to 1.1.
//
// Whole kernel, before (FP64 pairs) and after, one launch: 32^3 N = 4 warped bubble
// 3.400 -> 1.164 ms (narrow path), 16^3 N = 7 2.77 -> 0.79 ms, 16^3 N = 4 on a 2 km
// box 0.494 -> 0.209 ms (wide path), 60 x 12 x 6 N = 4 channel 0.566 -> 0.233 ms
// (tall path); with the launches of volume_fp64.cuh 0.966, 0.767 and 0.190 ms, and
// 80 x 16 x 8 N = 4 channel 0.485 ms.
//
// Which elements take it (fx_path, fx_scales), decided per element so that a
// result does not depend on the tile: all densities and 1/b = 2p/rho positive and
// within 0.95 % (narrow) or 12 % (wide) of the first node's, or densities between
// 0.21 and 1.12 of it (tall: a stratified element whose first node is its
// lowest); metric terms in a sane range, gamma <= 2, velocities up to about 0.4 of the
// speed of sound.  An element with stretched components, or whose energies stand well
// above p/rho, takes the tall path too, the only one for any scales.  The lines lie
// where the correction series leave 2^-51 (narrow), 2^-55 (wide, tall); all other
// elements take pair64.  The wide path costs a pair about 900 cycles, the tall one
// 1050.  The coefficients of odd_poly and coth_poly are those of the polynomials in w = y^2
// that interpolate (f(y)/y - 1)/w at the Chebyshev points of the path's interval, computed
// in 50 digits and rounded to the scales they are used at.
//
// The pair is pair64's in a form that needs no reciprocal: with the node
// fields x = ln(rho)/2, y = ln(b)/2 (relative to the element's first node) and
// differences over the pair (A minus B),
//   f_b = (b_A - b_B)/(b_A + b_B) = tanh(dy),
//   <rho>_log   = {{rho}} - (d rho / 2)(coth dx - 1/dx),
//   1/<b>_log   = {{1/b}} + (d(1/b)/3) f_b (1 + f_b^2/5 + 3 f_b^4/35 + ...),
//   p*          = {{rho}}/(2{{b}}) = {{p}} + f_b dp / 2,
//   {{b}}/b_A   = 1/(1 + f_b) = 1 + sinh^2 dy - sinh(2 dy)/2,  {{b}}/b_B with the sign changed,
// each correction a product of two differences over the pair.  The
// quadrature-weighted derivative matrix Q_il = w_i Dt_il is antisymmetric, so Q
// multiplies the metric average once and node B subtracts what node A adds; each
// node's sum is scaled by 1/w_i at its end.
#pragma once
#ifdef __CUDACC__
#define ESDG_HD __host__ __device__ __forceinline__
#else
#define ESDG_HD inline
#endif

namespace esdg_fx {

struct Fx {  // h 2^30 + l
  int h, l;
};
ESDG_HD Fx operator+(Fx a, Fx b) { return Fx{a.h + b.h, a.l + b.l}; }
ESDG_HD Fx operator-(Fx a, Fx b) { return Fx{a.h - b.h, a.l - b.l}; }

typedef long long i64;
typedef unsigned long long u64;

// a b + c: one integer multiply-add of 32 x 32 + 64 bits
ESDG_HD i64 madw(int a, int b, i64 c) {
#ifdef __CUDA_ARCH__
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(c) : "r"(a), "r"(b), "l"(c));
  return c;
#else
  return (i64)a * b + c;
#endif
}

// limbs of p, |p| < 2^61, |l| <= 2^29; limbs_b takes p + 2^29
ESDG_HD Fx limbs_b(i64 p) {
  return Fx{(int)(p >> 30), (int)((unsigned)p & 0x3fffffffu) - (1 << 29)};
}
ESDG_HD Fx limbs(i64 p) { return limbs_b(p + (1ll << 29)); }
// limbs of p/4, any p (the two low bits are dropped): 0 <= l < 2^30
ESDG_HD Fx limbs4(i64 p) { return Fx{(int)(p >> 32), (int)((unsigned)p >> 2)}; }
// Products over 2^60 (the low limbs' product, of mean zero and below a unit, is
// left out).  k rounds the shift (RND), or rounds it and adds the 2^29 of
// limbs_b (RNDL); it comes from the kernel's parameters, so that the
// multiply-add reads it there.
struct Round {
  i64 v, l;
};
constexpr i64 RND = 1ll << 29, RNDL = RND + (1ll << 59);
ESDG_HD i64 mul(Fx a, Fx b, i64 k) {
  i64 c = madw(a.h, b.l, k);
  c = madw(a.l, b.h, c);
  return madw(a.h, b.h, c >> 30);
}
ESDG_HD i64 mul2(Fx a, Fx b, Fx c, Fx d, i64 k) {  // a b + c d
  i64 x = madw(a.h, b.l, k);
  x = madw(a.l, b.h, x);
  x = madw(c.h, d.l, x);
  x = madw(c.l, d.h, x);
  return madw(c.h, d.h, madw(a.h, b.h, x >> 30));
}
ESDG_HD i64 mul3(Fx a, Fx b, Fx c, Fx d, Fx e, Fx f, i64 k) {
  i64 x = madw(a.h, b.l, k);
  x = madw(a.l, b.h, x);
  x = madw(c.h, d.l, x);
  x = madw(c.l, d.h, x);
  x = madw(e.h, f.l, x);
  x = madw(e.l, f.h, x);
  return madw(e.h, f.h, madw(c.h, d.h, madw(a.h, b.h, x >> 30)));
}
ESDG_HD unsigned hi32(unsigned a, unsigned b) { return (unsigned)(((u64)a * b) >> 32); }

// One element's scales: a field of value v is held as v 2^s.
struct FxScale {
  int ok;              // the element takes the fixed-point path
  int sr, sk, su, sn;  // density (halved), bracket and geopotential, velocity, metric
  int k[3];            // stretch of the components, the largest 0: u_c is held at su + k_c,
                       // Ja^d_c at sn - k_c (metric_stretch)
  ESDG_HD bool flat() const { return k[0] + k[1] + k[2] < 0; }
  ESDG_HD bool tall() const { return flat() || dp; }  // only the tall path has such scales
  int dp;              // bits by which the pressure's scale is above the bracket's
  int s1[3];           // 2 (su + k_c) - sk - dp - 60 >= 1: kinetic terms against the pressure terms
  ESDG_HD int sp() const { return sr + sk + dp - 60; }              // pressure
  ESDG_HD int sF() const { return sr + su + sn - 121; }             // mass flux times Q
  ESDG_HD int sM(int c) const { return sp() + sn - k[c] - 61; }     // momentum flux
  ESDG_HD int sE() const { return sF() + sk - 60; }                 // energy flux
};

struct FxNode {  // rho/2, p/2, 1/(6 (gamma-1) b), ln(rho)/6, ln(b)/2, phi/2 (at sk + dp),
                 // phi/2 + 1/(4 (gamma-1) b), u/2, Ja^d/2
  Fx r, p, c, x, y, f, g, u0, u1, u2, n0, n1, n2;
};

// y + y w (c0 + w (c1 + w (c2 + w (c3 + w c4)))) with w = y^2 (w37: w in scale
// 37): c0 and c1 in scale 60, the rest in scale 31.
ESDG_HD Fx odd_poly(Fx y, Fx w, int w37, i64 c0, i64 c1, int c2, int c3, int c4) {
  int t = c4 ? c3 + (int)(madw(w37, c4, 0) >> 37) : c3;
  t = c2 + (int)(madw(w37, t, 0) >> 37);
  const i64 u = c1 + (madw(w37, t, 0) >> 8);
  const i64 v = c0 + mul(w, limbs(u), RND);
  return y + limbs(mul(y, limbs(mul(w, limbs(v), RND)), RND));
}

// coth(3y) - 1/(3y) with 3y up to 0.85: nine coefficients, five in two limbs
ESDG_HD Fx coth_poly(Fx y, Fx w) {
  const int w34 = (w.h << 4) + (w.l >> 26);  // scale 34
  int t = 601955888 + (int)(madw(w34, -412417561, 0) >> 34);
  t = -682763608 + (int)(madw(w34, t, 0) >> 34);
  t = 750614701 + (int)(madw(w34, t, 0) >> 34);
  i64 u = -442049323941814575ll + (madw(w34, t, 0) >> 5);
  u = 485125393383650676ll + mul(w, limbs(u), RND);
  u = -533637953412707857ll + mul(w, limbs(u), RND);
  u = 592931059511645589ll + mul(w, limbs(u), RND);
  u = -691752902764107963ll + mul(w, limbs(u), RND);
  return y + limbs(mul(y, limbs(mul(w, limbs(u), RND)), RND));
}

// One unordered pair (A = node i, B = node l) of a pencil; q = Q_il 2^59.
// ai += Q F(A, B), al -= Q F(B, A) in units 2^-sF, 2^-sM (3), 2^-sE.  Sums and
// differences of limbs need no carries: |l| stays below 2^31.
// The corrections' arguments, with y = dy and dx = 3 x' (scale 60):
//   fb = tanh y, sg = sinh(2y)/2, ch = (3/2)(1 - 2y/sinh 2y)/tanh y, xx = coth dx - 1/dx.
// Narrow: each is the difference plus its cube times a linear polynomial in its
// square, in 30 bits (|y| < 0.0098; what is left out stays below 2^-51).
// Wide: |y|, |dx| < 0.1225, polynomials fitted to 2^-55, the leading terms in two
// limbs.  Tall: |dx| < 0.85, and any scales: components stretched against one another
// (s1 by component), the pressure's above the bracket's (dp).
enum { FX_NARROW = 0, FX_WIDE = 1, FX_TALL = 2, FX_GENERAL = 3 };
template <int PATH>
ESDG_HD void pair_fx(const FxNode& A, const FxNode& B, Fx q, const int* s1, int dp, const Round& K,
                     i64* ai, i64* al) {
  constexpr bool TALL = PATH == FX_TALL;
  if (!TALL) dp = 0;
  const Fx dy = A.y - B.y, dx = A.x - B.x;
  Fx fb, sg, ch, xx;
  if (PATH != FX_NARROW) {
    const Fx wy = limbs(mul(dy, dy, K.v)), wx = limbs(mul(dx, dx, K.v));
    const int y37 = (wy.h << 7) + (wy.l >> 23);
    fb = odd_poly(dy, wy, y37, -384307168202276263ll, 153722867260710440ll, -115895923, 46960618, -18747093);
    sg = odd_poly(dy, wy, y37, 768614336404552924ll, 153722867305918083ll, 27269618, 1516634, 0);
    ch = odd_poly(dy, wy, y37, -153722867280895198ll, 21960409573745069ll, -5453903, 686122, 0);
    xx = PATH == FX_TALL ? coth_poly(dx, wx)
                         : odd_poly(dx, wx, (wx.h << 7) + (wx.l >> 23), -691752902764081575ll, 592931059001350324ll, -993975292, 900876470, 0);
  } else {
    const int ys = (dy.h << 7) + (dy.l >> 23);    // scale 37
    const int y2 = (int)(madw(ys, ys, 0) >> 30);  // scale 44
    const int y3 = (int)(madw(ys, y2, 0) >> 32);  // scale 49
    const int tb = 0x55555555 - (int)hi32((unsigned)y2, 139810u);  // (1/3 - 2/15 y^2) 2^32
    const int tg = 0x2aaaaaab + (int)hi32((unsigned)y2, 34953u);   // (2/3 + 2/15 y^2) 2^30
    const int tc = 0x22222222 - (int)hi32((unsigned)y2, 19972u);   // (2/15 - 2/105 y^2) 2^32
    auto small = [](i64 v) { return Fx{(int)(v >> 30), (int)((unsigned)v & 0x3fffffffu)}; };
    fb = dy - small(madw(y3, tb, 0) >> 21);
    sg = dy + small(madw(y3, tg, 0) >> 19);
    ch = dy - small(madw(y3, tc, 0) >> 21);
    const int xs = (dx.h << 8) + (dx.l >> 22);    // scale 38
    const int x2 = (int)(madw(xs, xs, 0) >> 30);  // scale 46
    const int x3 = (int)(madw(xs, x2, 0) >> 32);  // scale 52
    const int tx = 0x4ccccccd - (int)hi32((unsigned)x2, 67413u);  // (0.6 - 0.5143 x'^2) 2^31
    xx = dx - small(madw(x3, tx, 0) >> 23);
  }
  // <rho>_log
  const Fx rl = (A.r + B.r) - limbs_b(mul(A.r - B.r, xx, K.l));
  // u . Q n and the mass flux
  const Fx n0 = limbs_b(mul(q, A.n0 + B.n0, K.l)), n1 = limbs_b(mul(q, A.n1 + B.n1, K.l)),
           n2 = limbs_b(mul(q, A.n2 + B.n2, K.l));
  const Fx u0 = A.u0 + B.u0, u1 = A.u1 + B.u1, u2 = A.u2 + B.u2;
  const Fx un = limbs_b(mul3(u0, n0, u1, n1, u2, n2, K.l));
  const i64 F = mul(rl, un, K.v);
  ai[0] += F;
  al[0] -= F;
  // pressure mean and gravity
  const Fx T = limbs_b(mul(rl, B.f - A.f, K.l));  // <rho>_log [[phi]] / 2
  const Fx V = limbs_b(mul(T, sg, K.l));
  const Fx S = T + limbs_b(mul(V, fb, K.l));  // T / (1 - fb^2)
  const Fx pt = (A.p + B.p) - limbs_b(mul(B.p - A.p, fb, K.l));
  const Fx pm = pt - V;
  // energy
  const int t = dp - 1;
  const i64 ke = TALL ? (mul(A.u0, B.u0, K.v) >> (s1[0] + t)) + (mul(A.u1, B.u1, K.v) >> (s1[1] + t)) +
                            (mul(A.u2, B.u2, K.v) >> (s1[2] + t))
                      : mul3(A.u0, B.u0, A.u1, B.u1, A.u2, B.u2, K.v) >> (s1[0] + t);
  const Fx br = (A.g + B.g) - limbs_b(mul(B.c - A.c, ch, K.l) - ke);
  const i64 E = TALL ? mul(limbs(F), br, K.v) + (mul(pt, un, K.v) >> dp)
                     : mul2(limbs(F), br, pt, un, K.v);
  ai[4] += E;
  al[4] -= E;
  // momentum
  const Fx F0 = limbs(F >> s1[0]), F1 = TALL ? limbs(F >> s1[1]) : F0,
           F2 = TALL ? limbs(F >> s1[2]) : F0;
  const i64 b0 = mul2(F0, u0, pm, n0, K.v), b1 = mul2(F1, u1, pm, n1, K.v),
            b2 = mul2(F2, u2, pm, n2, K.v);
  const i64 g0 = mul(S, n0, K.v), g1 = mul(S, n1, K.v), g2 = mul(S, n2, K.v);
  ai[1] += b0 + g0;
  al[1] -= b0 - g0;
  ai[2] += b1 + g1;
  al[2] -= b1 - g1;
  ai[3] += b2 + g2;
  al[3] -= b2 - g2;
}

}  // namespace esdg_fx

namespace esdg_fx {

// ln(x/x0) in units of 2^-58 from x and x0 (units of any scale, x0 in
// [2^58, 2^59)) and inv = 2^118/x0, |x/x0 - 1| < 0.0096:
//   ln(1 + a) = a - a^2/2 + a^3 (1/3 - a/4 + a^2/5 - a^3/6 + a^4/7),
// a and a^2 in two limbs, the cubic part (below 2^-21) in 31 bits.
ESDG_HD i64 log_ratio(i64 x, i64 x0, Fx inv) {
  const Fx a = limbs(mul(limbs(x - x0), inv, RND));  // scale 58
  const int as = (a.h << 9) + (a.l >> 21);                // scale 37
  const int a2 = (int)(madw(as, as, 0) >> 30);             // scale 44
  const int a3 = (int)(madw(as, a2, 0) >> 32);             // scale 49
  int t = 0x15555555 - (int)(madw(as, 0x12492492, 0) >> 37);  // (1/6 - a/7) 2^31
  t = 0x1999999a - (int)(madw(as, t, 0) >> 37);               // 1/5 - ...
  t = 0x20000000 - (int)(madw(as, t, 0) >> 37);               // 1/4 - ...
  t = 0x2aaaaaab - (int)(madw(as, t, 0) >> 37);               // 1/3 - ...
  return (i64)a.h * (1 << 30) + a.l - (mul(a, a, RND) << 1) + (madw(a3, t, 0) >> 22);
}

}  // namespace esdg_fx

#ifdef __CUDACC__
#include "esdg_internal.cuh"

namespace esdg_fx {

// v 2^s in limbs (|v 2^s| < 2^60; bits below one unit are dropped)
__device__ __forceinline__ i64 to_fx64(double v, int s) {
  const int hi = __double2hiint(v);
  const int e = (hi >> 20) & 0x7ff;
  u64 m = ((u64)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
  m <<= 7;
  const unsigned r = e ? (unsigned)(1082 - s - e) : 64u;
  asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m), "r"(r));  // shifts past 63 give 0
  return hi < 0 ? -(i64)m : (i64)m;
}
__device__ __forceinline__ Fx to_fx(double v, int s) { return limbs(to_fx64(v, s)); }
// v 2^-s, |s| < 700 (a sum's scale lies between -250 and 620): the power of two goes
// on the exponent field of the converted sum, which is zero or at least 1.  On the
// factor that multiplies it (-dt/J) it would not do: a step of zero, a subnormal or an
// infinite one has no exponent to add to.
__device__ __forceinline__ double from_fx(i64 v, int s) {
  const double d = (double)v;
  int hi = __double2hiint(d);
  if (hi) hi -= s * (1 << 20);
  return __hiloint2double(hi, __double2loint(d));
}
// does v 2^s leave the limbs' range by 2^-b? (infinities and NaNs do)
__device__ __forceinline__ bool fx_over(double v, int s, int b) {
  return ((__double2hiint(v) >> 20) & 0x7ff) > 1082 - s - b;
}
__device__ __forceinline__ Fx ld_fx(const double* p) {
  const int2 v = *reinterpret_cast<const int2*>(p);
  return Fx{v.x, v.y};
}
__device__ __forceinline__ void st_fx(double* p, Fx v) {
  *reinterpret_cast<int2*>(p) = make_int2(v.h, v.l);
}

// An element's metric terms Ja/2 are kept in limbs (rows 0-8 of its geometry
// block, 8 bytes each as the doubles they stand for) with the scales sn - k_c of their
// three components behind the last element's block; FX_NO_METRIC marks an element whose
// terms stay doubles (none or out of the sane range).
constexpr int FX_NO_METRIC = -1000000;
__host__ __device__ __forceinline__ int* metric_scales(const double* vgeo, size_t E, int np) {
  return const_cast<int*>(reinterpret_cast<const int*>(vgeo + E * ESDG_NVGEO * np));
}
// The stretch k_c <= 0 of the components from the high words of the largest |Ja^d_c/2|
// of each: stretched to a common size, a flat element looks like a cube (u_c Ja^d_c, and
// with it every mass flux, stays the same).  None where the largest terms of the
// components lie within a factor of two to four: that costs at most two of the six
// spare bits and keeps the element off the tall path.
__device__ __forceinline__ void metric_stretch(const unsigned* hi, int* k) {
  const int e0 = (int)(hi[0] >> 20), e1 = (int)(hi[1] >> 20), e2 = (int)(hi[2] >> 20);
  const int top = max(e0, max(e1, e2)), none = min(e0, min(e1, e2)) >= top - 1;
  k[0] = none ? 0 : e0 - top;
  k[1] = none ? 0 : e1 - top;
  k[2] = none ? 0 : e2 - top;
}
// sn of an element whose largest squared norm of Ja^d/2 (stretched) has this high word:
// the norm of Ja^d is below 2^(60 - sn)
__device__ __forceinline__ int metric_scale(unsigned hi, const int* k) {
  const int e = (int)((hi >> 20) & 0x7ff) - 1022;  // |Ja^d/2|^2 < 2^e
  return e > -240 && e < 240 && min(k[0], min(k[1], k[2])) > -60 ? 60 - (((e + 1) >> 1) + 1)
                                                                : FX_NO_METRIC;
}

// What a tile keeps per element: the scales, the first node's rho and 1/b
// (the logarithms' reference), the scales of the five sums as they leave the
// pencils, and the running maxima (high words) of the prologue: the stretched
// velocity's components and the geopotential.
struct FxElement {
  FxScale sc;
  int out[5];
  int mu;
  unsigned mf;
  double rq0, ib0;  // the first node's rho/4 and 1/b, as in log_ratio r0, b0,
  i64 r0, b0;
  Fx ir0, inb0;     // and their reciprocals
  int sb;           // scale of b0
  double phi0;      // the first node's geopotential: the pairs' is relative to it
};

// the stored scales of an element's metric, for its tile
__device__ __forceinline__ void fx_metric(FxElement& E, const int* scales) {
  const int s0 = scales[0], s1 = scales[1], s2 = scales[2];
  E.sc.sn = min(s0, min(s1, s2));
  E.sc.k[0] = E.sc.sn - s0;
  E.sc.k[1] = E.sc.sn - s1;
  E.sc.k[2] = E.sc.sn - s2;
}
// high word of |u 2^k|, not positive where that is too small to matter
__device__ __forceinline__ int stretched(double u, int k) {
  return (__double2hiint(u) & 0x7fffffff) + k * (1 << 20);
}
// The scales of an element from its first node and the maxima; ok = 0 where a
// field leaves the representation or loses more than the spare bits: velocities of about
// half the speed of sound (a stretched element: the largest u_c Ja_c over the smallest
// Ja_c above a tenth of it), gamma > 2 or below 1.005, geopotential differences above the
// energies.
__device__ __forceinline__ void fx_scales(FxElement& E, double rq0, double ib0, double phi0,
                                          double gm1, double igm1, int wm) {
  auto expo = [](unsigned hi) { return (int)((hi >> 20) & 0x7ff) - 1022; };  // |v| < 2^expo
  auto sane = [&](unsigned hi) { return expo(hi) > -120 && expo(hi) < 120; };
  const unsigned hr = (unsigned)__double2hiint(rq0), hb = (unsigned)__double2hiint(ib0);
  FxScale s = E.sc;
  const int low = min(s.k[0], min(s.k[1], s.k[2])), eu = expo(E.mu) - low;  // any velocity / 2 < 2^eu
  bool ok = !(hr >> 31) && !(hb >> 31) && sane(hr) && sane(hb) && s.sn != FX_NO_METRIC && gm1 <= 1.0 &&
            eu < 60 && expo(E.mf) < 120;
  // bracket: 1/(2 (gamma-1) b) (12 % above the first node's) + kinetic +
  // geopotential, below 2^(60 - sk)
  const float um = ok ? __uint_as_float((unsigned)max(eu + 127, 1) << 23) : 1.0f;
  const float fm = ok ? __uint_as_float((unsigned)max(expo(E.mf) + 127, 1) << 23) : 1.0f;
  const float kin = 6.0f * um * um, rest = fmaf(2.0f, fm, 0.565f * esdg_d2f(igm1 * ib0));
  const float k = ok ? kin + rest : 1.0f;
  const int eK = (int)((__float_as_uint(k) >> 23) & 0xff) - 126;
  // The pressure p = rho / (2b) is held at the bracket's scale while that is below 3/b
  // (gamma = 1.4 at rest: 1.4 to 2.8, by the power of two); above, its scale is raised by
  // as many bits, on the tall path.
  s.dp = max(eK - ((int)(__float_as_uint(3.0f * esdg_d2f(ib0)) >> 23) - 127), 0);
  s.sr = 60 - (expo(hr) + 2);
  s.sk = 60 - eK;
  // the norm of u (stretched), at most sqrt(3) times the largest component (u/2 in mu),
  // is below 2^(60 - su)
  const int hm = (int)(E.mu & 0xfffffu) >= 0x279a7 ? 2 : 1;  // mantissa over 2/sqrt(3)
  s.su = 60 - max(expo(E.mu) + hm, -200);
  // Stretched, um is a bound that no node need come near, and what it takes from the
  // pressure's and the small components' bits shows from um = 64 m/s on (1000 x 1000 x 10 m,
  // u = 10, N = 4, error of rho u over that of the FP64 pairs: w = 0.5 0.81, w = 1 1.08,
  // w = 2 1.22): 32 m/s at the temperature of air.
  s.ok = ok && k < 1.0e30f && s.dp < 8 && expo(E.mf) + 1 + s.dp <= eK && (!s.flat() || 16.0f * kin <= rest);
  const int s1 = 2 * s.su - s.sk - s.dp - 60;
  s.ok = s.ok && s1 + 2 * low >= 1;
  for (int c = 0; c < 3; c++) {
    s.s1[c] = min(s1 + 2 * s.k[c], 55);  // a shift of s1 + dp stays below 64
    E.out[1 + c] = s.sM(c) - 2 - wm;
  }
  E.sc = s;
  E.out[0] = s.sF() - 2 - wm;
  E.out[4] = s.sE() - 2 - wm;
  E.rq0 = rq0;
  E.phi0 = phi0;
  E.ib0 = ib0;
  E.sb = 59 - expo(hb);
  if (s.ok) {
    E.r0 = to_fx64(rq0, s.sr + 1);
    E.b0 = to_fx64(ib0, E.sb);
    E.ir0 = limbs(2 * to_fx64(esdg_rcp(rq0), 117 - (s.sr + 1)));
    E.inb0 = limbs(2 * to_fx64(esdg_rcp(ib0), 117 - E.sb));
  }
}

// ln(x/x0)/2 = z (1 + z^2/3 + z^4/5 + ...) with z = (x - x0)/(x + x0), |z| < 0.064,
// the terms beyond z^4 (below 2^-26) in FP32
__device__ __forceinline__ double half_log_ratio(double x, double x0) {
  const double z = (x - x0) * esdg_rcp(x + x0), u = z * z;
  const float uf = esdg_d2f(u);
  const float t = uf * uf * fmaf(uf, fmaf(uf, fmaf(uf, 1.0f / 13.0f, 1.0f / 11.0f), 1.0f / 9.0f), 1.0f / 7.0f);
  const double p = fma(u, 0.2, 1.0 / 3.0) + esdg_f2d(t);
  return fma(z * u, p, z);
}

// The path that this node leaves to its element: may it share the first node's
// scales and the correction series?  (NaNs and values that are not positive may not.)
__device__ __forceinline__ unsigned fx_path(double rq, double ib, double rq0, double ib0) {
  // positive, finite, exponents within the float range (esdg_d2f's domain)
  const unsigned hr = (unsigned)__double2hiint(rq), hb = (unsigned)__double2hiint(ib);
  const bool sane = hr - 0x38800000u < 0x0f000000u && hb - 0x38800000u < 0x0f000000u;
  const float r0 = esdg_d2f(rq0), rn = esdg_d2f(rq);
  const float b0 = esdg_d2f(ib0), bn = esdg_d2f(ib);
  const float dr = fabsf(rn - r0), db = fabsf(bn - b0);
  if (!(sane && rn <= 1.12f * r0 && rn >= 0.21f * r0 && db <= 0.12f * b0)) return FX_GENERAL;
  if (!(dr <= 0.12f * r0)) return FX_TALL;
  return dr <= 0.0095f * r0 && db <= 0.0095f * b0 ? FX_NARROW : FX_WIDE;
}

// Slots of the node fields in a tile's S buffer (those of the FP64 fields they
// replace, one 8-byte word each): rho/4 -> r, b/2 -> y, 1/b -> c, u/2, phi/2,
// [ln rho -> x], [ln b -> p], Ja/2, and one more: g.
template <int NP>
__device__ __forceinline__ void fx_convert(double* S, int n, const FxElement& E, unsigned path, double ce) {
  const FxScale& s = E.sc;
  const double rq = S[n], ib = S[2 * NP + n], ph = S[8 * NP + n];
  const i64 r = to_fx64(rq, s.sr + 1);
  st_fx(S + n, limbs(r));
  // y = -ln(1/b)/2 and x = ln(rho)/6 in scale 60 (log_ratio: scale 58)
  if (path != FX_NARROW) {
    st_fx(S + 1 * NP + n, to_fx(half_log_ratio(E.ib0, ib), 60));
    const double h = path == FX_TALL ? 0.5 * log(rq * esdg_rcp(E.rq0)) : half_log_ratio(rq, E.rq0);
    st_fx(S + 7 * NP + n, to_fx(h * (1.0 / 3.0), 60));
  } else {
    st_fx(S + 1 * NP + n, limbs(-2 * log_ratio(to_fx64(ib, E.sb), E.b0, E.inb0)));
    st_fx(S + 7 * NP + n, limbs(mul(limbs(log_ratio(r, E.r0, E.ir0)), Fx{0x2aaaaaab, -0x15555555}, RND)));
  }
  st_fx(S + 2 * NP + n, to_fx(ib * (ce * (1.0 / 3.0)), s.sk));
#pragma unroll
  for (int k = 3; k < 6; k++) st_fx(S + k * NP + n, to_fx(S[k * NP + n], s.su + s.k[k - 3]));
  const i64 f = to_fx64(S[6 * NP + n], s.sk + s.dp);
  st_fx(S + 6 * NP + n, limbs(f));
  st_fx(S + 18 * NP + n, limbs((f >> s.dp) + to_fx64(ib * (ce * 0.5), s.sk)));
  st_fx(S + 8 * NP + n, to_fx(ph, s.sp()));
}

template <int NP>
__device__ __forceinline__ FxNode fx_load(const double* S, int n, int d) {
  FxNode a;
  a.r = ld_fx(S + n);
  a.y = ld_fx(S + NP + n);
  a.c = ld_fx(S + 2 * NP + n);
  a.u0 = ld_fx(S + 3 * NP + n);
  a.u1 = ld_fx(S + 4 * NP + n);
  a.u2 = ld_fx(S + 5 * NP + n);
  a.f = ld_fx(S + 6 * NP + n);
  a.g = ld_fx(S + 18 * NP + n);
  a.x = ld_fx(S + 7 * NP + n);
  a.p = ld_fx(S + 8 * NP + n);
  const double* nh = S + (9 + 3 * d) * NP;
  a.n0 = ld_fx(nh + n);
  a.n1 = ld_fx(nh + NP + n);
  a.n2 = ld_fx(nh + 2 * NP + n);
  return a;
}

// An interface term (a value already divided by w_end, scale out) as the
// start of its end node's sum.
__device__ __forceinline__ i64 fx_lift(double f, int out, const EsdgLGL& L) {
  return mul(to_fx(f, out), Fx{L.w0h, L.w0l}, RND) * 8;
}

}  // namespace esdg_fx
#endif
