// rt_split.cuh -- the double precision RK4 step of the grating cloak on the
// FP32 pipe.
//
// FP64 arithmetic runs at 1/64 of the FP32 rate on this GPU, and the FP64 step
// (rk4_step<double>) is some 600 FP64 instructions.  Nothing in the step needs
// them: a step moves the ray by a few hundredths of a period over k, so what
// it computes -- the increments of position, momentum and W0 -- enters the
// state scaled by 1e-2 to 1e-3.  Here the state is held as unevaluated sums of
// three floats (72 bits, more than a double), and the increments are computed
// as sums of two floats (48 bits) with error-free transformations: two_sum
// (Knuth 1969), fast_two_sum and two_prod by FMA (Dekker 1971; Ogita, Rump &
// Oishi 2005), so a step's rounding stays at or below that of the FP64 step.
//
// Units.  Lengths are multiplied by k = 2 pi and the momentum by k h, and
// points are held as i (x + i y) = (-y, x), the direction in which W0's argument
// moves:
//   T = k (-y, X),  Q = k h (-p_y, p_x),  Phi = k h^2 (-F_y, F_x),
// so a classical RK4 step on r'' = F(r) (rk4_step) needs no products with h:
//   D2 = Q/2,  D3 = Q/2 + Phi1/4,  D4 = Q + Phi2/2  (stage displacements),
//   D  = Q + (Phi1 + Phi2 + Phi3)/6,  T += D,
//   Q += (Phi1 + 2 Phi2 + 2 Phi3 + Phi4)/6.
//
// W0 along a displacement D.  With W = W_b exp(d), W e^W = zeta (Eq. 13) at both
// ends gives, exactly,
//   d + W_b (exp(d) - 1) = D.
// d is small, so exp(d) - 1 is a short Taylor polynomial and no argument
// reduction, library exponential or sine is needed.  The solve (split_solve)
// takes d0 in FP32 (fourth-order continuation), then one Newton step on the
// residual in two floats.  The abscissa itself never enters.
//
// What bounds it.  some 870 single and 450 packed FP32 instructions a step
// against the FP64 step's 600 FP64 instructions of 64 scheduler cycles each.
// The cloaked 512 x 512 x 4 render takes 38.0 ms (592 ms with the FP64 step),
// the FMA pipe 65 % busy; 64 x 64 x 1, bound by the latency of the longest ray's
// chain of steps, 5.8 ms (32.9).  On the way: unrolled 89 ms (a 2,700-instruction
// loop body, most issue slots waiting for instructions), rolled over the four
// evaluations with the sums on packed pairs 50 ms, the face tests out of FP64
// and the state in shared memory 44 ms, fewer normalisations 39 ms.
//
// Accuracy.  Two floats are 48 bits against FP64's 53, and the solve's errors grow
// with a high power of its |d|, so the step is no less accurate than FP64's
// only up to some step size (split_in_range).  At that range's edge, over 100
// rays of up to 300 steps, half of them from the crests upwards, against RK4 of
// the same step in 113 bits: error of (x, y, p_x, p_y), median / 90 % of the rays,
// and in parentheses of RK4 in double (tests/test_split_accuracy.py):
//   kA = 0.02   2.3e-16 / 5.1e-16  (1.2e-15 / 2.1e-15)
//   kA = 0.1    4.2e-16 / 1.6e-15  (1.1e-15 / 2.5e-15)
//   kA = 0.25   1.5e-16 / 6.3e-16  (9.8e-16 / 1.8e-15)
//   kA = 0.3    1.5e-16 / 7.9e-16  (8.8e-16 / 2.0e-15)
// (kA = 0.3 at steps half as long again, with the guess cut at t^3: 3.5e-16 /
// 4.8e-15, rms 11 times the double's.)  Dormand-Prince with its stages' W0 so, and
// steps chosen for 1e-6: the double's within 7 %.  Whole rays, the kernels'
// exits against a trace with 64-bit mantissas, 2,464 rays a scene, kA from 0.005
// to 0.3: RK4's median error 0.1 to 0.9 of the FP64 kernel's and its rms 0.3 to
// 1.0; Dormand-Prince's 0.98 to 1.02.
#pragma once

#if defined(__CUDACC__)
#define GRT_HD __device__ __forceinline__
#else
#include <cmath>
#define GRT_HD static inline
#endif

namespace grt {

// Rounded operations that the compiler may not contract or reorder.
#if defined(__CUDA_ARCH__)
GRT_HD float fadd(float a, float b) { return __fadd_rn(a, b); }
GRT_HD float fmul(float a, float b) { return __fmul_rn(a, b); }
GRT_HD float ffma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
GRT_HD float frcp(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
GRT_HD float fex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
GRT_HD void fsincos(float x, float& s, float& c) { __sincosf(x, &s, &c); }
#else
GRT_HD float fadd(float a, float b) { return a + b; }
GRT_HD float fmul(float a, float b) { return a * b; }
GRT_HD float ffma(float a, float b, float c) { return fmaf(a, b, c); }
GRT_HD float frcp(float x) { return 1.0f / x; }
GRT_HD float fex2(float x) { return exp2f(x); }
GRT_HD void fsincos(float x, float& s, float& c) { s = sinf(x); c = cosf(x); }
#endif
GRT_HD float fsub(float a, float b) { return fadd(a, -b); }
// ... and on pairs, two operations in one instruction (FADD2, FFMA2)
#if defined(__CUDA_ARCH__)
GRT_HD float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
GRT_HD float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
GRT_HD float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
GRT_HD float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
#else
#if !defined(__CUDACC__)
struct float2 { float x, y; };
#endif
GRT_HD float2 vadd(float2 a, float2 b) { return {a.x + b.x, a.y + b.y}; }
GRT_HD float2 vsub(float2 a, float2 b) { return {a.x - b.x, a.y - b.y}; }
GRT_HD float2 vfma(float2 a, float2 b, float2 c) { return {ffma(a.x, b.x, c.x), ffma(a.y, b.y, c.y)}; }
GRT_HD float2 vmul(float2 a, float2 b) { return {a.x * b.x, a.y * b.y}; }
#endif
GRT_HD float2 vneg(float2 a) { return {-a.x, -a.y}; }

// Whether scenes of amplitude kA whose steps are h at most (kh = k h) take these
// steps.  A step's displacement is D <= k h n_max, n_max = 1/(1 - kA) (a thousandth
// for the drift of |p| over a ray), and the solve's |d| up to D/(1 - kA).
// RK4: |d| <= 0.06, where the series of split_expm1_tail and the guess still
// leave it no less accurate than FP64's (the benchmark's h = Lambda/200 has
// 0.056 at kA = 0.25); up to kA = 0.1, where forces and W0 are smaller, |D| <= 1/16.
// Dormand-Prince, whose stages' W0 alone is carried, for
// one step, and enters scaled by it: |D| <= 0.56 (h_max = Lambda/16 has 0.53 at
// kA = 0.25) and kA <= 0.28 (at 0.3 a tenth of the rays end up to 30 % further off).
inline bool split_in_range(bool rk4, double kA, double kh)
{
    const double D = kh * (1.001 / (1.0 - kA));
    return rk4 ? kA <= 0.3 && D <= (kA <= 0.1 ? 1.0 / 16.0 : 0.06 * (1.0 - kA)) : kA <= 0.28 && D <= 0.56;
}

struct F2 { float h, l; };          // h + l, |l| <= ulp(h)/2 when normalised
struct Z2 { float2 h, l; };         // a pair (x, y) of those: a point, or re + i im
struct Z3 { float2 h, m, l; };      // a pair of h + m + l

GRT_HD F2 fast_two_sum(float a, float b)          // |a| >= |b| or a = 0
{
    const float s = fadd(a, b);
    return {s, fsub(b, fsub(s, a))};
}
GRT_HD F2 two_prod(float a, float b)
{
    const float p = fmul(a, b);
    return {p, ffma(a, b, -p)};
}
GRT_HD F2 mulu(F2 a, F2 b)                        // product, not normalised
{
    const F2 p = two_prod(a.h, b.h);
    return {p.h, ffma(a.l, b.h, ffma(a.h, b.l, p.l))};
}
GRT_HD F2 mul(F2 a, F2 b)
{
    const F2 p = mulu(a, b);
    return fast_two_sum(p.h, p.l);
}
GRT_HD Z2 two_sum(float2 a, float2 b)
{
    const float2 s = vadd(a, b), bb = vsub(s, a);
    return {s, vadd(vsub(a, vsub(s, bb)), vsub(b, bb))};
}
GRT_HD Z2 fast_two_sum(float2 a, float2 b)
{
    const float2 s = vadd(a, b);
    return {s, vsub(b, vsub(s, a))};
}
GRT_HD Z2 scale(Z2 a, float w)                    // w: a power of two
{
    const float2 ww = {w, w};
    return {vmul(a.h, ww), vmul(a.l, ww)};
}
GRT_HD Z2 addu(Z2 a, Z2 b)                        // not normalised
{
    const Z2 s = two_sum(a.h, b.h);
    return {s.h, vadd(s.l, vadd(a.l, b.l))};
}
GRT_HD Z2 fast_addu(Z2 a, Z2 b)                   // |a| >= |b|, not normalised
{
    const Z2 s = fast_two_sum(a.h, b.h);
    return {s.h, vadd(s.l, vadd(a.l, b.l))};
}
GRT_HD Z2 add(Z2 a, Z2 b)
{
    const Z2 s = two_sum(a.h, b.h);
    return fast_two_sum(s.h, vadd(s.l, vadd(a.l, b.l)));
}
GRT_HD Z2 mul(Z2 a, F2 b)                         // times a real
{
    const F2 p = two_prod(a.h.x, b.h), q = two_prod(a.h.y, b.h);
    const float2 t = {ffma(a.l.x, b.h, ffma(a.h.x, b.l, p.l)), ffma(a.l.y, b.h, ffma(a.h.y, b.l, q.l))};
    return fast_two_sum(float2{p.h, q.h}, t);
}
// Complex products.  The sums of the partial products run on pairs, the
// products on single floats, whose operands need no broadcast or swap.
GRT_HD Z2 zmulu(Z2 a, Z2 b)                       // not normalised
{
    const F2 p = two_prod(a.h.x, b.h.x), q = two_prod(a.h.x, b.h.y);
    const F2 u = two_prod(-a.h.y, b.h.y), v = two_prod(a.h.y, b.h.x);
    const Z2 s = two_sum(float2{p.h, q.h}, float2{u.h, v.h});
    const float tx = ffma(-a.l.y, b.h.y, ffma(-a.h.y, b.l.y, ffma(a.l.x, b.h.x, ffma(a.h.x, b.l.x, p.l))));
    const float ty = ffma(a.l.y, b.h.x, ffma(a.h.y, b.l.x, ffma(a.l.x, b.h.y, ffma(a.h.x, b.l.y, q.l))));
    return {s.h, vadd(s.l, vadd(float2{tx, ty}, float2{u.l, v.l}))};
}
GRT_HD Z2 zmulf(Z2 a, float2 b)                   // times a complex float, not normalised
{
    const F2 p = two_prod(a.h.x, b.x), q = two_prod(a.h.x, b.y);
    const F2 u = two_prod(-a.h.y, b.y), v = two_prod(a.h.y, b.x);
    const Z2 s = two_sum(float2{p.h, q.h}, float2{u.h, v.h});
    const float tx = ffma(-a.l.y, b.y, ffma(a.l.x, b.x, p.l)), ty = ffma(a.l.y, b.x, ffma(a.l.x, b.y, q.l));
    return {s.h, vadd(s.l, vadd(float2{tx, ty}, float2{u.l, v.l}))};
}
GRT_HD float2 cmul(float2 a, float2 b)            // in FP32
{
    return {ffma(a.x, b.x, -fmul(a.y, b.y)), ffma(a.x, b.y, fmul(a.y, b.x))};
}
GRT_HD float2 cfma(float2 a, float2 b, float2 c)
{
    return {ffma(a.x, b.x, ffma(-a.y, b.y, c.x)), ffma(a.x, b.y, ffma(a.y, b.x, c.y))};
}
// a + b for a three-float accumulator
GRT_HD Z3 acc(Z3 a, Z2 b)
{
    const Z2 s = two_sum(a.h, b.h), t = two_sum(a.m, b.l), u = two_sum(s.l, t.h);
    const float2 l = vadd(vadd(a.l, t.l), u.l);
    const Z2 v = fast_two_sum(s.h, u.h), w = fast_two_sum(v.l, l);
    return {v.h, w.h, w.l};
}
GRT_HD Z2 hi2(Z3 a) { return {a.h, vadd(a.m, a.l)}; }

struct F3 { float h, m, l; };
GRT_HD F3 split3(double x)
{
    const float h = (float)x;
    const double r = x - (double)h;
    const float m = (float)r;
    return {h, m, (float)(r - (double)m)};
}
GRT_HD Z3 split3(double x, double y)
{
    const F3 a = split3(x), b = split3(y);
    return {float2{a.h, b.h}, float2{a.m, b.m}, float2{a.l, b.l}};
}
GRT_HD Z2 split2(double x, double y)
{
    const float a = (float)x, b = (float)y;
    return {float2{a, b}, float2{(float)(x - (double)a), (float)(y - (double)b)}};
}
GRT_HD double join_x(Z2 a) { return (double)a.h.x + (double)a.l.x; }
GRT_HD double join_y(Z2 a) { return (double)a.h.y + (double)a.l.y; }
GRT_HD double join_x(Z3 a) { return (double)a.h.x + ((double)a.m.x + (double)a.l.x); }
GRT_HD double join_y(Z3 a) { return (double)a.h.y + ((double)a.m.y + (double)a.l.y); }

// Ray inside the cloak between steps.
struct SplitState {
    Z3 t;                 // k (-y, X)
    Z3 q;                 // k h (-p_y, p_x)
    Z3 w;                 // W0
    Z2 f;                 // k h^2 (-F_y, F_x)
    float2 r;             // 1/(1 + W0)
};

// Force at W: Phi = kappa (-Re G, Im G), G = W conj(1 + W)^2 / |1 + W|^6 (Eq. 12
// in the form of ray_force), kappa = k h^2 fk; r = 1/(1 + W) as well.
GRT_HD void split_force(Z2 w, F2 kappa, Z2& f, Z2& r)
{
    F2 a = fast_two_sum(1.0f, w.h.x);
    a = fast_two_sum(a.h, fadd(a.l, w.l.x));
    const F2 b = {w.h.y, w.l.y};
    // |1 + Re W| > 0.7 > |Im W|: the sums need no ordering
    const F2 aa = mulu(a, a), bb = mulu(b, b), m1 = fast_two_sum(aa.h, bb.h), d1 = fast_two_sum(aa.h, -bb.h);
    const F2 m = {m1.h, fadd(m1.l, fadd(aa.l, bb.l))};
    const float y = frcp(m.h);
    const float e = fsub(ffma(-m.h, y, 1.0f), fmul(m.l, y));
    const F2 inv = fast_two_sum(y, fmul(y, ffma(e, e, e)));       // 1/m
    const F2 ab = mulu(a, b);
    const Z2 d = {float2{d1.h, -2.0f * ab.h}, float2{fadd(d1.l, fsub(aa.l, bb.l)), -2.0f * ab.l}};   // conj(1 + W)^2
    const Z2 g = zmulu(w, d);
    const F2 s = mul(mul(mul(inv, inv), inv), kappa);
    f = mul(Z2{float2{-g.h.x, g.h.y}, float2{-g.l.x, g.l.y}}, s);
    r = mul(Z2{float2{a.h, -b.h}, float2{a.l, -b.l}}, inv);
}

// exp(z) - 1 = z + e for a complex float z: Taylor to the ninth order,
// z^2 (1/2 + z U), U = 1/3! + z V, V = 1/4! + z X, with X and the products that
// enter below 2^-48 of the result in FP32 -- for |z| <= 0.06; at 0.13
// (split_solve_wide) the change of W0 is off by up to 1.7e-14 of itself (rms).
GRT_HD Z2 split_expm1_tail(float2 z)
{
    const float c5l = -0x1.dddddep-32f;                            // 1/5! past its FP32 rounding
    const F2 c4 = {0x1.555556p-5f, -0x1.555556p-30f}, c3 = {0x1.555556p-3f, -0x1.555556p-28f};
    float2 t = {ffma(z.x, 1.0f / 362880.0f, 1.0f / 40320.0f), fmul(z.y, 1.0f / 362880.0f)};
    t = cfma(t, z, float2{1.0f / 5040.0f, 0.0f});
    t = cfma(t, z, float2{1.0f / 720.0f, 0.0f});
    t = cfma(t, z, float2{1.0f / 120.0f, 0.0f});
    t = cmul(t, z);
    // V
    const F2 v = fast_two_sum(c4.h, t.x);
    const float vl = fadd(v.l, ffma(z.x, c5l, c4.l)), vi = ffma(z.y, c5l, t.y);
    // U
    const F2 p = two_prod(z.x, v.h), q = two_prod(z.y, v.h), u = fast_two_sum(c3.h, p.h);
    const Z2 U = {float2{u.h, q.h}, float2{fadd(u.l, fadd(c3.l, ffma(z.x, vl, ffma(-z.y, vi, p.l)))),
                                           ffma(z.y, vl, ffma(z.x, vi, q.l))}};
    // 1/2 + z U
    Z2 h = zmulf(U, z);
    const F2 h1 = fast_two_sum(0.5f, h.h.x);
    h.h.x = h1.h;
    h.l.x = fadd(h.l.x, h1.l);
    // z^2 (1/2 + z U)
    const F2 xx = two_prod(z.x, z.x), yy = two_prod(-z.y, z.y), xy = two_prod(2.0f * z.x, z.y);
    const float ds = fadd(xx.h, yy.h), db = fsub(ds, xx.h);
    const float dl = fadd(fsub(xx.h, fsub(ds, db)), fsub(yy.h, db));
    return zmulu(Z2{float2{ds, xy.h}, float2{fadd(dl, fadd(xx.l, yy.l)), xy.l}}, h);
}

// The continuation d of W = W_b exp(d) over s in FP32: with t = s r, v = W_b r,
// d = t - v t^2 (1/2 + (1 - 3v) t/6 + (1 - 10v + 15v^2) t^2/24), good to about
// t^5/30.  (split_newton drops the third order of its error: cut at t^3 the guess
// was most of the solve's error near the crests, 5.9e-15 of W0 at W_b = -0.3 and
// |s| = 0.042 against 8.6e-16 so, for 0.4 % of the step's time.)
GRT_HD float2 split_guess(float2 v, float2 r, float2 s)
{
    const float2 t = cmul(s, r);
    const float2 u = {ffma(0.625f, v.x, -5.0f / 12.0f), 0.625f * v.y};
    const float2 g = cfma(u, v, float2{1.0f / 24.0f, 0.0f});                          // (1 - 10v + 15v^2)/24
    const float2 c = {ffma(-0.5f, v.x, 1.0f / 6.0f), -0.5f * v.y};                   // (1 - 3v)/6
    const float2 a = cmul(v, cfma(cfma(g, t, c), t, float2{0.5f, 0.0f}));
    const float2 b = cmul(a, t);
    return cfma(float2{-b.x, -b.y}, t, t);
}

// Newton step of the solve at d0 = z with E = exp(z) - 1: P = W_b E and the
// residual s - z - P, then P and W = W_b + P with the step taken.
GRT_HD void split_newton(Z2 wb, float2 z, Z2 e, Z2 s, Z2& p, Z2& w)
{
    // the leading parts nearly cancel, their remainders are of the residual's size
    p = zmulu(wb, e);
    const Z2 r1 = two_sum(s.h, vneg(z)), r2 = two_sum(r1.h, vneg(p.h));
    const Z2 R = {r2.h, vadd(vadd(r1.l, r2.l), vsub(s.l, p.l))};
    // D = R/(1 + W1), W1 = W_b exp(z): an FP32 reciprocal q, corrected by
    // c = 1 - q (1 + W1), whose leading parts cancel exactly
    const Z2 w1 = add(wb, p);
    const F2 a1 = fast_two_sum(1.0f, w1.h.x);
    const float ax = a1.h, ay = w1.h.y, bx = fadd(a1.l, w1.l.x), by = w1.l.y;
    const float inv = frcp(ffma(ax, ax, fmul(ay, ay)));
    const float2 q = {fmul(ax, inv), -fmul(ay, inv)};
    const F2 c1 = two_prod(q.x, ax), c2 = two_prod(q.x, ay);
    const float2 c = {ffma(q.y, by, ffma(-q.x, bx, fsub(ffma(q.y, ay, fsub(1.0f, c1.h)), c1.l))),
                      -ffma(q.y, bx, ffma(q.x, by, fadd(ffma(q.y, ax, c2.h), c2.l)))};
    Z2 d = zmulf(R, q);
    // exp(d) - exp(z) = exp(z) (D + D^2 q/2): the second order of both the root
    // and the exponential
    const float2 g = cfma(d.h, float2{0.5f * q.x, 0.5f * q.y}, c);
    d.l = vadd(d.l, cmul(d.h, g));
    const Z2 wd = zmulu(w1, d);
    p = fast_addu(p, wd);
    w = fast_addu(w1, wd);
}

// Full solve: base W_b with v = W_b/(1 + W_b) and r = 1/(1 + W_b) in FP32,
// displacement s.  Returns P = W_b (exp(d) - 1), so that W = W_b + P, and W.
GRT_HD void split_solve(Z2 wb, float2 v, float2 r, Z2 s, Z2& p, Z2& w)
{
    const float2 z = split_guess(v, r, s.h);
    const Z2 e = split_expm1_tail(z), e1 = two_sum(z, e.h);
    split_newton(wb, z, Z2{e1.h, vadd(e1.l, e.l)}, s, p, w);
}

// The solve for |s| up to 0.6 (Dormand-Prince stages), from the FP32 guess z,
// which Newton steps in FP32 improve and leave in z: exp(z) - 1 from z/8, by
// E <- 2 E + E^2 three times.  Returns P.
GRT_HD Z2 split_solve_wide(Z2 wb, Z2 s, float2& z)
{
    for (int it = 0; it < 8; ++it) {
        const float m = fex2(fmul(z.x, 1.44269504f));
        float sn, cs;
        fsincos(z.y, sn, cs);
        const float2 E = {ffma(m, cs, -1.0f), fmul(m, sn)};
        const float2 u = cmul(wb.h, E);
        const float2 R = {fsub(fsub(s.h.x, z.x), u.x), fsub(fsub(s.h.y, z.y), u.y)};
        const float ax = fadd(1.0f + wb.h.x, u.x), ay = fadd(wb.h.y, u.y);
        const float inv = frcp(ffma(ax, ax, fmul(ay, ay)));
        const float2 d = {fmul(ffma(R.x, ax, fmul(R.y, ay)), inv), fmul(ffma(R.y, ax, -fmul(R.x, ay)), inv)};
        z = vadd(z, d);
        if (!(ffma(d.x, d.x, fmul(d.y, d.y)) > 1e-8f)) break;      // the next step would be 1e-8 at most
    }
    const float2 x = {0.125f * z.x, 0.125f * z.y};
    const Z2 t = split_expm1_tail(x), e1 = two_sum(x, t.h);
    Z2 e = {e1.h, vadd(e1.l, t.l)};
#if defined(__CUDACC__)
#pragma unroll 1
#endif
    for (int q = 0; q < 3; ++q) e = add(scale(e, 2.0f), zmulu(e, e));
    Z2 p, w;
    split_newton(wb, z, e, s, p, w);
    return p;
}

// Continuation over a small s (|s| <= 1e-3) from a point whose W and r are
// known in two floats: W (exp(d) - 1), with t = s r and v = W r,
//   exp(d) - 1 = t + t^2 (1 - v) (1/2 + (1 - 3v) t/6),
// the first order in two floats, the rest in FP32.
GRT_HD Z2 split_continue(Z2 w, Z2 r, Z2 s)
{
    const Z2 t = zmulu(s, r);
    const float2 v = cmul(w.h, r.h);
    const float2 c = {ffma(-0.5f, v.x, 1.0f / 6.0f), -0.5f * v.y};
    const float2 m = cmul(float2{fsub(1.0f, v.x), -v.y}, cfma(c, t.h, float2{0.5f, 0.0f}));
    return zmulu(w, Z2{t.h, vadd(t.l, cmul(cmul(m, t.h), t.h))});
}

// One RK4 step from s into o (kappa = k h^2 fk).  The four evaluations run in
// a rolled loop -- a solve at the second and fourth stages, a continuation at
// the third and at the end -- so that the step's code stays in the instruction
// cache.
GRT_HD void split_step(const SplitState& s, F2 kappa, SplitState& o)
{
    const F2 sixth = {0x1.555556p-3f, -0x1.555556p-28f};
    const Z2 wb = hi2(s.w);
    const float2 v = cmul(wb.h, s.r);
    // the displacement of the next solve and of the continuation after it
    Z2 d = scale(hi2(s.q), 0.5f), e = scale(s.f, 0.25f);
    Z2 sum = s.f;                                // Phi1 + 2 Phi2 + 2 Phi3 (+ Phi4)
    Z2 dif = s.f;                                // Phi1 - 2 Phi2 + Phi3
    Z2 w, r, f, p, c;
#if defined(__CUDACC__)
#pragma unroll 1
#endif
    for (int j = 0; j < 4; ++j) {
        if ((j & 1) == 0) {
            split_solve(wb, v, s.r, d, p, w);
        } else {
            c = split_continue(w, r, e);
            w = fast_addu(w, c);
        }
        split_force(w, kappa, f, r);
        if (j < 3) {
            sum = addu(sum, scale(f, (j == 2) ? 1.0f : 2.0f));
            if (j == 0) {
                dif = addu(dif, scale(f, -2.0f));
                d = add(hi2(s.q), scale(f, 0.5f));                 // D4 = Q + Phi2/2
            }
            if (j == 1) e = mul(addu(dif, f), sixth);              // D = D4 + (Phi1 - 2 Phi2 + Phi3)/6
        }
    }
    o.w = acc(s.w, addu(p, c));
    o.t = acc(s.t, fast_addu(d, e));
    o.q = acc(s.q, mul(sum, sixth));
    o.f = f;
    o.r = r.h;
}

}  // namespace grt
