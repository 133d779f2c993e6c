// mg5_split.cuh -- the FP64 cell arithmetic on the FP32 and integer pipes.
//
// GB300 executes FP64 at 2 lanes a clock per SM, 1/64 of its FP32 rate: an FP64 sweep spends
// ~32 FP64-pipe instructions a cell, 16 clocks of an SM, whatever the memory does.  Here a cell
// is computed in FP32 operations without giving up FP64's accuracy:
//
//  * A tile of cells shares one exponent.  Every value of the field is cut into three 20-bit
//    pieces on the common grid u, u 2^-20, u 2^-40 (split3), each an integer multiple of its grid
//    unit below 2^20 in an FP32 register.  Sums and differences of up to 16 values are then exact
//    piece by piece, so the face sums, the second and the mixed differences -- where FP64 rounds
//    against the much larger field values -- carry no rounding at all.  A value more than 7
//    binary orders below the tile's largest loses its bits under 2^-60 of that largest one; FP64
//    itself rounds the neighbours' sums at 2^-53 of them.
//  * The differences' pieces are added up to unevaluated (hi, lo) pairs of FP32 values, and the
//    nonlinear terms and the residual are pair arithmetic (Knuth's and Dekker's exact sums, the
//    exact product by fused multiply-add): ~2^-47 of the terms.
//  * With X, Y, Z the second differences along the axes, lambda = X + Y + Z = h^2 L, d.. the mixed
//    ones (four-point sums), all in units of u,
//      op h^2 / u = lambda + kappa3 P,  P = X (Y + Z) + Y Z - (dxy^2 + dxz^2 + dyz^2) / 16,
//    kappa3 = 2 alpha u / h^2 ((lap)^2 - (d_i d_j phi)^2 = 2 sum_{a<b} (D_aa D_bb - D_ab^2)), and the
//    residual is r = F - lambda - kappa3 P, F = h^2 (f + c) / u.
//  * A sweep takes the cell's root as the change d of lambda: with kappa = kappa3 / 3 and
//    q1 = 1 + 2 kappa lambda, kappa d^2 + q1 d = r (the neighbours' combination Sigma does not hold
//    the cell's value).  d is estimated in FP32 and refined by one Newton step whose residual is
//    pair arithmetic (as the FP64 kernels refine their FP32 estimate), so d is good to ~2^-44 of
//    itself.  The new value phi - (omega/6) d u is added up in FP64.
//
// Measured against 128-bit arithmetic on converged lognormal fields of sigma 0.5 .. 1.5 (rms; residual
// relative to ||s delta||, update relative to phi), FP64 kernels -> these: residual 4.4e-15 .. 7.9e-15 ->
// 2.5e-15 .. 2.8e-15 at 64^3, 8.2e-15 .. 1.6e-14 -> 2.4e-15 .. 2.8e-15 at 128^3; update 1.4e-16 .. 1.5e-16
// -> 5e-17 .. 9e-17 at 48^3 and up.  The FP64 residual's error comes from the sums of the field's values and
// lies in every cell, this one from the nonlinear terms' 2^-47 and lies in the densest: the largest of a
// cell is 0.4e-15 .. 6.7e-15 of max |s delta| there, 2.5e-15 .. 8.6e-15 here.
//
// Every quantity is a float2: the same cell of two half-tiles, through the packed FP32
// instructions (two lanes an instruction), which have no operand negation: products are formed
// with one factor's negative, so that the exact error needs no sign change.
//
// Cells near the double root (discriminant below 0.25, as in the FP64 kernels), cells with
// anything not finite and tiles whose exponent leaves the FP32 range are left to the FP64
// arithmetic of mg5_dev.cuh.
#pragma once
#include <cmath>
#include <cstring>

#include "mg5_dev.cuh"

namespace mg5 {
namespace split {

#define MG5_HD __host__ __device__ __forceinline__

#ifdef __CUDA_ARCH__
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return pk_sub(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float bits_f(unsigned u) { return __uint_as_float(u); }
__device__ __forceinline__ unsigned f_bits(float f) { return __float_as_uint(f); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float rsq(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
#else
inline float fsub(float a, float b) { volatile float r = a - b; return r; }
inline float fmul(float a, float b) { volatile float r = a * b; return r; }
inline float fadd_(float a, float b) { volatile float r = a + b; return r; }
inline float2 add2(float2 a, float2 b) { return float2{fadd_(a.x, b.x), fadd_(a.y, b.y)}; }
inline float2 sub2(float2 a, float2 b) { return float2{fsub(a.x, b.x), fsub(a.y, b.y)}; }
inline float2 mul2(float2 a, float2 b) { return float2{fmul(a.x, b.x), fmul(a.y, b.y)}; }
inline float2 fma2(float2 a, float2 b, float2 c) { return float2{std::fmaf(a.x, b.x, c.x), std::fmaf(a.y, b.y, c.y)}; }
inline float bits_f(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
inline unsigned f_bits(float f) { unsigned u; std::memcpy(&u, &f, 4); return u; }
inline float rsq(float x) { return 1.0f / std::sqrt(x); }
inline float rcp(float x) { return 1.0f / x; }
#endif

MG5_HD float2 both(float x) { return float2{x, x}; }

// Values in pieces (units u): h multiples of 1, m of 2^-20, l of 2^-40.
struct P3 {
    float2 h, m, l;
};
MG5_HD P3 operator+(const P3 &a, const P3 &b) { return P3{add2(a.h, b.h), add2(a.m, b.m), add2(a.l, b.l)}; }
MG5_HD P3 operator-(const P3 &a, const P3 &b) { return P3{sub2(a.h, b.h), sub2(a.m, b.m), sub2(a.l, b.l)}; }
// s - 2 c
MG5_HD P3 minus2(const P3 &s, const P3 &c)
{
    return P3{fma2(both(-2.0f), c.h, s.h), fma2(both(-2.0f), c.m, s.m), fma2(both(-2.0f), c.l, s.l)};
}

// Unevaluated sums hi + lo.
struct Pair {
    float2 h, l;
};
MG5_HD Pair two_sum(float2 a, float2 b)
{
    const float2 s = add2(a, b), t = sub2(s, a);
    return Pair{s, add2(sub2(a, sub2(s, t)), sub2(b, t))};
}
// a - b
MG5_HD Pair two_diff(float2 a, float2 b)
{
    const float2 s = sub2(a, b), t = sub2(s, a);
    return Pair{s, sub2(sub2(a, sub2(s, t)), add2(b, t))};
}
// pieces -> pair; h is a multiple of 1 and |m| < 2^4, so the error of h + m is found exactly
MG5_HD Pair pair_of(const P3 &p)
{
    const float2 s = add2(p.h, p.m);
    return Pair{s, add2(sub2(p.m, sub2(s, p.h)), p.l)};
}

// The unit of a tile of biased exponent eb (its largest |x| < 2^(eb - 1022)): u = 2^(eb - 1042).
constexpr int kUnitBias = 1042;
// exponents for which the unit and its products with the pieces are normal FP32 values, and the
// largest kappa3 whose products stay finite (lambda < 2^24)
constexpr int kMinExp = 1023 - 90, kMaxExp = 1023 + 90;
constexpr float kMaxKappa = 1.0995116e12f;   // 2^40

// Pieces of two doubles with words (hi, lo), of biased exponents at most eb (>= kMinExp: zero and
// subnormals are shifted out).
MG5_HD unsigned funnel_r(unsigned lo, unsigned hi, int n)
{
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, n);
#else
    return (unsigned)((((unsigned long long)hi << 32) | lo) >> n);
#endif
}
MG5_HD void piece_bits(unsigned hi, unsigned lo, int eb, float &h, float &m, float &l, float &sg)
{
    int sh = eb - (int)((hi >> 20) & 0x7ffu);
    sh = sh > 63 ? 63 : sh;
    const unsigned vh = funnel_r(lo, (hi & 0xfffffu) | 0x100000u, 25), vl = lo << 7;
    const unsigned long long v = (((unsigned long long)vh << 32) | vl) >> sh;   // 60 bits
    const unsigned wh = (unsigned)(v >> 32), wl = (unsigned)v;
    h = bits_f(funnel_r(wh, 0x4Bu, 8));                             // 2^23 + h
    m = bits_f(0x41000000u | (funnel_r(wl, wh, 20) & 0xfffffu));   // 2^3 + m 2^-20
    l = bits_f(0x37000000u | (wl & 0xfffffu));                     // 2^-17 + l 2^-40
    sg = bits_f(0x3f800000u | (hi & 0x80000000u));
}
MG5_HD P3 split2(unsigned ahi, unsigned alo, unsigned bhi, unsigned blo, int eb)
{
    P3 p;
    float2 sg;
    piece_bits(ahi, alo, eb, p.h.x, p.m.x, p.l.x, sg.x);
    piece_bits(bhi, blo, eb, p.h.y, p.m.y, p.l.y, sg.y);
    p.h = mul2(sub2(p.h, both(8388608.0f)), sg);
    p.m = mul2(sub2(p.m, both(8.0f)), sg);
    p.l = mul2(sub2(p.l, both(7.62939453125e-06f)), sg);
    return p;
}

// The double with words (hi, lo) as a (h, l) pair of FP32 values: 24 bits by truncation and the
// other 29 rounded to 24.  Below 2^-73 zero; from 2^100 on (infinity, NaN) infinity.
MG5_HD void pair_words(unsigned hi, unsigned lo, float &h, float &l)
{
    const unsigned e = (hi >> 20) & 0x7ffu, sg = hi & 0x80000000u;
    unsigned b = ((hi << 3) | (lo >> 29)) - (896u << 23);
    float t = (float)(int)(lo & 0x1fffffffu) * bits_f((e - 948u) << 23);
    const bool small = e < 950u, big = e >= 1123u;
    b = small ? 0u : (big ? 0x7f800000u : b & 0x7fffffffu);
    t = (small || big) ? 0.0f : t;
    h = bits_f(b | sg);
    l = bits_f(f_bits(t) | sg);
}

// x 2^(eb - kUnitBias) as the words of a double, |x| normal FP32 or zero
MG5_HD void unit_words(float x, int eb, unsigned &hi, unsigned &lo)
{
    const unsigned b = f_bits(x);
    const bool nz = (b & 0x7f800000u) != 0u;
    hi = nz ? ((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + ((unsigned)(896 + eb - kUnitBias) << 20))) : 0u;
    lo = nz ? b << 29 : 0u;
}

// Per-grid constants: 2 alpha / h^2 and 2 alpha / (3 h^2) as pairs, omega / 6 as a pair.
// ok: they are in the FP32 range the cell arithmetic needs.
struct Coef {
    float k3h, k3l, kh, kl, wh, wl;
    int ok;
};

inline Coef make_split_coef(const CoefT<double> &cf)
{
    Coef c;
    const double k = cf.k23 * cf.inv_h2, k3 = 3.0 * k;
    c.k3h = (float)k3;
    c.k3l = (float)(k3 - (double)c.k3h);
    c.kh = (float)k;
    c.kl = (float)(k - (double)c.kh);
    c.wh = (float)cf.w6;
    c.wl = (float)(cf.w6 - (double)c.wh);
    c.ok = cf.h2 > 1e-18 && cf.h2 < 1e18 && (k == 0.0 || (k > 1e-18 && k < 1e18));
    return c;
}

// ... and of a tile: the unit's products with them.
struct Kap {
    float k3h, k3l, kh, kl;
};

// Second and mixed differences of a cell as pairs.
struct Lin {
    Pair lam, X, W, Y, Z, xy, xz, yz;   // lam = X + W, W = Y + Z
};

MG5_HD Lin lin_of(const P3 &c, const P3 &sx, const P3 &sy, const P3 &sz, const P3 &dxy, const P3 &dxz,
                  const P3 &dyz)
{
    Lin r;
    const P3 X = minus2(sx, c), Y = minus2(sy, c), Z = minus2(sz, c);
    const P3 W = Y + Z;
    r.lam = pair_of(X + W);
    r.X = pair_of(X);
    r.W = pair_of(W);
    r.Y = pair_of(Y);
    r.Z = pair_of(Z);
    r.xy = pair_of(dxy);
    r.xz = pair_of(dxz);
    r.yz = pair_of(dyz);
    return r;
}

// -(x y) = p - e (p the rounded -(x.h y.h), e the rest of x y)
MG5_HD void neg_mul(const Pair &x, const Pair &y, float2 &p, float2 &e)
{
    p = mul2(mul2(both(-1.0f), x.h), y.h);
    e = fma2(x.h, y.h, p);
    e = fma2(x.h, y.l, e);
    e = fma2(x.l, y.h, e);
}
MG5_HD void neg_sqr(const Pair &x, float2 &p, float2 &e)
{
    p = mul2(mul2(both(-1.0f), x.h), x.h);
    e = fma2(x.h, x.h, p);
    e = fma2(fma2(both(2.0f), x.h, x.l), x.l, e);
}

// r = F - lambda - kappa3 P, normalised
MG5_HD Pair resid(const Lin &t, const Pair &F, const Kap &k)
{
    float2 p, e, q, g;
    // the mixed differences' squares: -(sum) = D - E
    float2 D, E;
    neg_sqr(t.xy, D, E);
    neg_sqr(t.xz, p, e);
    Pair s = two_sum(D, p);
    D = s.h;
    E = sub2(add2(E, e), s.l);
    neg_sqr(t.yz, p, e);
    s = two_sum(D, p);
    D = mul2(s.h, both(0.0625f));
    E = mul2(sub2(add2(E, e), s.l), both(0.0625f));
    // N = -P = n + nl
    neg_mul(t.X, t.W, p, e);
    neg_mul(t.Y, t.Z, q, g);
    s = two_sum(p, q);
    float2 nl = sub2(s.l, add2(e, g));
    s = two_diff(s.h, D);
    nl = add2(nl, add2(s.l, E));
    const float2 n = s.h;
    // r = F - lambda + kappa3 N
    p = mul2(both(-k.k3h), n);
    e = fma2(both(k.k3h), n, p);
    e = fma2(both(k.k3h), nl, e);
    e = fma2(both(k.k3l), n, e);
    const Pair a = two_diff(F.h, t.lam.h), b = two_diff(a.h, p);
    const float2 l = add2(sub2(F.l, t.lam.l), add2(add2(a.l, b.l), e));
    return two_sum(b.h, l);
}

// The change d of lambda that takes each cell to its root; ok: false where the cell is left to
// FP64.
MG5_HD void root_change(const Lin &t, const Pair &r, const Kap &k, Pair &d, bool &okx, bool &oky)
{
    // q1 = 1 + 2 kappa lambda
    const float k2 = 2.0f * k.kh;
    float2 p = mul2(both(-k2), t.lam.h);
    float2 e = fma2(both(k2), t.lam.h, p);
    e = fma2(both(k2), t.lam.l, e);
    e = fma2(both(2.0f * k.kl), t.lam.h, e);
    const Pair q = two_diff(both(1.0f), p);
    const float2 ql = add2(q.l, e);
    const float2 D = fma2(both(4.0f * k.kh), r.h, mul2(q.h, q.h));
    okx = D.x >= 0.25f && D.x < 1e30f && q.h.x > 0.0f;
    oky = D.y >= 0.25f && D.y < 1e30f && q.h.y > 0.0f;
    const float2 rs{rsq(D.x), rsq(D.y)};   // 1 / sqrt(D): sqrt(D) is the slope at the root
    const float2 den = fma2(D, rs, q.h);
    const float2 d0 = mul2(add2(r.h, r.h), float2{rcp(den.x), rcp(den.y)});
    // Newton: d0 + (r - q1 d0 - kappa d0^2) / sqrt(D)
    p = mul2(mul2(both(-1.0f), q.h), d0);
    e = fma2(ql, d0, fma2(q.h, d0, p));
    const float2 kd = mul2(both(k.kh), d0), nkd = mul2(both(-k.kh), d0);
    const float2 ek = fma2(both(k.kl), d0, fma2(both(k.kh), d0, nkd));
    const float2 p2 = mul2(nkd, d0);
    e = add2(e, fma2(ek, d0, fma2(kd, d0, p2)));
    const Pair s1 = two_sum(r.h, p), s2 = two_sum(s1.h, p2);
    const float2 rho = add2(s2.h, sub2(add2(r.l, add2(s1.l, s2.l)), e));
    d = Pair{d0, mul2(rho, rs)};
}

// (omega / 6) d = e - p
MG5_HD void step_of(const Pair &d, const Coef &c, float2 &p, float2 &e)
{
    p = mul2(both(-c.wh), d.h);
    e = fma2(both(c.wh), d.h, p);
    e = fma2(both(c.wh), d.l, e);
    e = fma2(both(c.wl), d.h, e);
}

// ---- one cell at a time ---------------------------------------------------------
// The same arithmetic on single values (k_visit.cu: coarse grids, where a CTA has fewer cells
// than threads).  There the pieces are the value itself: add_change adds a pair to them, rounded
// to the grid u 2^-40, and leaves h an integer, |m| <= 1/2 and |l| <= 2^-21.
namespace one {

#ifdef __CUDA_ARCH__
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
inline float add(float a, float b) { return fadd_(a, b); }
inline float sub(float a, float b) { return fsub(a, b); }
inline float mul(float a, float b) { return fmul(a, b); }
inline float fma(float a, float b, float c) { return std::fmaf(a, b, c); }
#endif

struct P1 {
    float h, m, l;
};
struct Pr {
    float h, l;
};
MG5_HD P1 operator+(const P1 &a, const P1 &b) { return P1{add(a.h, b.h), add(a.m, b.m), add(a.l, b.l)}; }
MG5_HD P1 operator-(const P1 &a, const P1 &b) { return P1{sub(a.h, b.h), sub(a.m, b.m), sub(a.l, b.l)}; }
MG5_HD P1 minus2(const P1 &s, const P1 &c)
{
    return P1{fma(-2.0f, c.h, s.h), fma(-2.0f, c.m, s.m), fma(-2.0f, c.l, s.l)};
}
MG5_HD Pr two_sum(float a, float b)
{
    const float s = add(a, b), t = sub(s, a);
    return Pr{s, add(sub(a, sub(s, t)), sub(b, t))};
}
MG5_HD Pr pair_of(const P1 &p)
{
    const float s = add(p.h, p.m);
    return Pr{s, add(sub(p.m, sub(s, p.h)), p.l)};
}
MG5_HD Pr add_pair(const Pr &a, const Pr &b)
{
    const Pr s = two_sum(a.h, b.h);
    return Pr{s.h, add(s.l, add(a.l, b.l))};
}
MG5_HD Pr mul_pair(const Pr &x, const Pr &y)
{
    const float p = mul(x.h, y.h);
    return Pr{p, fma(x.l, y.h, fma(x.h, y.l, fma(x.h, y.h, -p)))};
}
MG5_HD Pr sqr(const Pr &x)
{
    const float p = mul(x.h, x.h);
    return Pr{p, fma(fma(2.0f, x.h, x.l), x.l, fma(x.h, x.h, -p))};
}
// a power of two times x
MG5_HD Pr scale(const Pr &x, float s) { return Pr{mul(x.h, s), mul(x.l, s)}; }
MG5_HD Pr neg(const Pr &x) { return Pr{-x.h, -x.l}; }

// The double with words (hi, lo) times 2^k as a pair.
MG5_HD Pr pair_scaled(unsigned hi, unsigned lo, int k)
{
    const int e = (int)((hi >> 20) & 0x7ffu);
    const int x = e == 0 ? 0 : (e == 2047 ? 2047 : e + k);
    const unsigned h2 = (hi & 0x800fffffu) | ((unsigned)(x < 0 ? 0 : (x > 2047 ? 2047 : x)) << 20);
    Pr r;
    pair_words(h2, lo, r.h, r.l);
    return r;
}
MG5_HD P1 split1(unsigned hi, unsigned lo, int eb)
{
    float h, m, l, sg;
    const int e = (int)((hi >> 20) & 0x7ffu);
    piece_bits(hi, lo, eb < e ? e : eb, h, m, l, sg);   // (infinity, NaN: any value)
    return P1{mul(sub(h, 8388608.0f), sg), mul(sub(m, 8.0f), sg), mul(sub(l, 7.62939453125e-06f), sg)};
}

struct Lin1 {
    Pr lam, X, W, Y, Z, xy, xz, yz;
};
MG5_HD Lin1 lin_of(const P1 &c, const P1 &sx, const P1 &sy, const P1 &sz, const P1 &dxy, const P1 &dxz,
                   const P1 &dyz)
{
    Lin1 r;
    const P1 X = minus2(sx, c), Y = minus2(sy, c), Z = minus2(sz, c);
    const P1 W = Y + Z;
    r.lam = pair_of(X + W);
    r.X = pair_of(X);
    r.W = pair_of(W);
    r.Y = pair_of(Y);
    r.Z = pair_of(Z);
    r.xy = pair_of(dxy);
    r.xz = pair_of(dxz);
    r.yz = pair_of(dyz);
    return r;
}
// lambda + kappa3 P (h^2 op / u) subtracted from F, normalised
MG5_HD Pr resid(const Lin1 &t, const Pr &F, const Kap &k)
{
    Pr d = add_pair(add_pair(sqr(t.xy), sqr(t.xz)), sqr(t.yz));
    const Pr P = add_pair(add_pair(mul_pair(t.X, t.W), mul_pair(t.Y, t.Z)), scale(d, -0.0625f));
    const Pr q = mul_pair(Pr{k.k3h, k.k3l}, P);
    const Pr a = two_sum(F.h, -t.lam.h), b = two_sum(a.h, -q.h);
    return two_sum(b.h, add(sub(F.l, t.lam.l), sub(add(a.l, b.l), q.l)));
}
// As split::root_change; a cell near the double root (or not finite) takes the closed form in
// FP64, as the FP64 kernels do, and a negative discriminant is clamped and counted.
MG5_HD Pr root_change(const Lin1 &t, const Pr &r, const Kap &k, unsigned &clamps)
{
    const Pr kap{k.kh, k.kl};
    const Pr q0 = scale(mul_pair(kap, t.lam), 2.0f);
    const Pr o = two_sum(1.0f, q0.h);
    const Pr q{o.h, add(o.l, q0.l)};
    const float D = fma(4.0f * k.kh, r.h, mul(q.h, q.h));
    if (D >= 0.25f && D < 1e30f && q.h > 0.0f) {
        const float rs = rsq(D);
        const float d0 = mul(add(r.h, r.h), rcp(fma(D, rs, q.h)));
        const float p = mul(q.h, d0), e = fma(q.l, d0, fma(q.h, d0, -p));
        const float kd = mul(k.kh, d0), ek = fma(k.kl, d0, fma(k.kh, d0, -kd));
        const float p2 = mul(kd, d0), e2 = fma(ek, d0, fma(kd, d0, -p2));
        const Pr s1 = two_sum(r.h, -p), s2 = two_sum(s1.h, -p2);
        const float rho = add(s2.h, sub(add(r.l, add(s1.l, s2.l)), add(e, e2)));
        return Pr{d0, mul(rho, rs)};
    }
    const double lam = (double)t.lam.h + (double)t.lam.l, kd = (double)k.kh + (double)k.kl;
    const double b = lam + kd * lam * lam + ((double)r.h + (double)r.l), disc = 1.0 + 4.0 * kd * b;
    double L = 2.0 * b;
    if (disc < 0.0)
        ++clamps;
    else
        L = 2.0 * b / (1.0 + sqrt(disc));
    const double d = L - lam;
    const float dh = (float)d;
    return Pr{dh, (float)(d - (double)dh)};
}

MG5_HD float round_to(float x, float magic) { return sub(add(x, magic), magic); }
constexpr float kMagic0 = 12582912.0f;           // 1.5 2^23: to integers
constexpr float kMagic1 = 12.0f;                 // 1.5 2^3: to multiples of 2^-20
constexpr float kMagic2 = 1.1444091796875e-05f;  // 1.5 2^-17: to multiples of 2^-40

MG5_HD P1 add_change(const P1 &c, const Pr &d)
{
    const float a = round_to(d.h, kMagic0);
    const Pr s = two_sum(sub(d.h, a), d.l);
    const float b = round_to(s.h, kMagic1);
    const float t = round_to(add(sub(s.h, b), s.l), kMagic2);
    P1 r{add(c.h, a), add(c.m, b), add(c.l, t)};
    const float x = round_to(r.l, kMagic1);
    r.l = sub(r.l, x);
    r.m = add(r.m, x);
    const float y = round_to(r.m, kMagic0);
    r.m = sub(r.m, y);
    r.h = add(r.h, y);
    return r;
}

}  // namespace one

}  // namespace split
}  // namespace mg5
