// Rounding of the grating cloak's RK4 and Dormand-Prince steps in two and three
// floats (rt_split.cuh, its host form) and of the same methods in double, against
// 113 bits.  Prints, for a method, kA and a step, the error of (x, y, p_x, p_y)
// at the end of each of n rays: "<double> <split>" a line.
//   split_accuracy rk4|dp45 kA kh rays steps [tol]    (kh 0: the range's edge;
// Dormand-Prince: the largest step, with steps chosen for tol, 1e-6 by default)
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "rt_split.cuh"

using namespace grt;
#if defined(__x86_64__)
typedef __float128 Q;
#else
typedef long double Q;                                    // 113 bits on aarch64
#endif
static const Q kPiQ = (Q)3.141592653589793 + (Q)1.2246467991473532e-16 + (Q)(-2.9947698097183397e-33);
static const Q kQ = 2 * kPiQ;
static const double kPi = 3.14159265358979323846;

template <class R> struct Cx { R r, i; };
template <class R> static Cx<R> mul(Cx<R> a, Cx<R> b) { return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r}; }
template <class R> static Cx<R> inv(Cx<R> a) { const R m = a.r * a.r + a.i * a.i; return {a.r / m, -a.i / m}; }

static Cx<double> cexp(Cx<double> z) { const double e = exp(z.r); return {e * cos(z.i), e * sin(z.i)}; }
static Cx<Q> cexp(Cx<Q> z)                                // Taylor series of z / 2^9, then squarings
{
    Cx<Q> w = {z.r / 512, z.i / 512}, s = {1, 0}, t = {1, 0};
    for (int n = 1; n < 30; ++n) {
        t = mul(t, w);
        t = {t.r / n, t.i / n};
        s = {s.r + t.r, s.i + t.i};
    }
    for (int n = 0; n < 9; ++n) s = mul(s, s);
    return s;
}

// W0 at (x, y) by Newton steps on W + kA exp(-W + i k z) = 0 from w
template <class R> static Cx<R> w0(R kA, R k, R x, R y, Cx<R> w, R tol)
{
    for (int it = 0; it < 60; ++it) {
        const Cx<R> e = cexp(Cx<R>{-(w.r + k * y), k * x - w.i});
        const Cx<R> d = mul(Cx<R>{w.r + kA * e.r, w.i + kA * e.i}, inv(Cx<R>{1 + w.r, w.i}));
        w = {w.r - d.r, w.i - d.i};
        if (d.r * d.r + d.i * d.i < tol * tol) break;
    }
    return w;
}
template <class R> static void force(R k, Cx<R> w, R& fx, R& fy)
{
    const Cx<R> r = inv(Cx<R>{1 + w.r, w.i}), g = mul(w, mul(r, r));
    const R n2 = r.r * r.r + r.i * r.i;
    fx = k * n2 * g.i;
    fy = k * n2 * g.r;
}

template <class R> struct Ray { R x, y, px, py; Cx<R> w; R fx, fy; };

template <class R> static Ray<R> rk4(R kA, R k, R tol, const Ray<R>& s, R h)
{
    const R h2 = h / 2;
    R f2x, f2y, f3x, f3y, f4x, f4y;
    Cx<R> w = w0(kA, k, s.x + h2 * s.px, s.y + h2 * s.py, s.w, tol);
    force(k, w, f2x, f2y);
    w = w0(kA, k, s.x + h2 * (s.px + h2 * s.fx), s.y + h2 * (s.py + h2 * s.fy), w, tol);
    force(k, w, f3x, f3y);
    w = w0(kA, k, s.x + h * (s.px + h2 * f2x), s.y + h * (s.py + h2 * f2y), w, tol);
    force(k, w, f4x, f4y);
    Ray<R> o;
    o.x = s.x + (h * s.px + h * h / 6 * (s.fx + f2x + f3x));
    o.y = s.y + (h * s.py + h * h / 6 * (s.fy + f2y + f3y));
    o.px = s.px + h / 6 * (s.fx + 2 * (f2x + f3x) + f4x);
    o.py = s.py + h / 6 * (s.fy + 2 * (f2y + f3y) + f4y);
    o.w = w0(kA, k, o.x, o.y, w, tol);
    force(k, o.w, o.fx, o.fy);
    return o;
}

// Dormand-Prince 5(4) on r'' = F(r); kWide carries the stages' W0 as dp45_step_wide does
static const double A[8][8] = {
    {0}, {0}, {0, 1.0 / 5}, {0, 3.0 / 40, 9.0 / 40}, {0, 44.0 / 45, -56.0 / 15, 32.0 / 9},
    {0, 19372.0 / 6561, -25360.0 / 2187, 64448.0 / 6561, -212.0 / 729},
    {0, 9017.0 / 3168, -355.0 / 33, 46732.0 / 5247, 49.0 / 176, -5103.0 / 18656},
    {0, 35.0 / 384, 0, 500.0 / 1113, 125.0 / 192, -2187.0 / 6784, 11.0 / 84}};
static const double E[8] = {0, 35.0 / 384 - 5179.0 / 57600, 0, 500.0 / 1113 - 7571.0 / 16695, 125.0 / 192 - 393.0 / 640,
                            -2187.0 / 6784 + 92097.0 / 339200, 11.0 / 84 - 187.0 / 2100, -1.0 / 40};
template <class R, bool kWide> static Ray<R> dp45(R kA, R k, R tol, const Ray<R>& s, R h, double* error)
{
    R fx[8], fy[8], dx = 0, dy = 0;
    fx[1] = s.fx;
    fy[1] = s.fy;
    Cx<R> w = s.w;
    const Z2 wb = split2((double)s.w.r, (double)s.w.i);
    const Cx<R> r0 = inv(Cx<R>{1 + s.w.r, s.w.i});
    float2 z = {0, 0}, dp = z, r = {(float)r0.r, (float)r0.i};
    for (int j = 2; j <= 7; ++j) {
        R ax = 0, ay = 0, c = 0;
        for (int l = 1; l < j; ++l) {
            R a = 0;
            for (int m = l + 1; m < j; ++m) a += (R)A[j][m] * (R)A[m][l];
            ax += a * fx[l];
            ay += a * fy[l];
            c += (R)A[j][l];
        }
        dx = c * h * s.px + h * h * ax;
        dy = c * h * s.py + h * h * ay;
        if (kWide) {
            const Z2 d = split2(-2 * kPi * (double)dy, 2 * kPi * (double)dx);
            z = cfma(vsub(d.h, dp), r, z);
            dp = d.h;
            const Z2 p = split_solve_wide(wb, d, z);
            w = {s.w.r + (R)join_x(p), s.w.i + (R)join_y(p)};
            const Cx<R> q = inv(Cx<R>{1 + w.r, w.i});
            r = {(float)q.r, (float)q.i};
        } else {
            w = w0(kA, k, s.x + dx, s.y + dy, w, tol);
        }
        force(k, w, fx[j], fy[j]);
    }
    Ray<R> o = s;
    o.x = s.x + dx;
    o.y = s.y + dy;
    for (int l = 1; l <= 6; ++l) {
        o.px += h * (R)A[7][l] * fx[l];
        o.py += h * (R)A[7][l] * fy[l];
    }
    double gx = 0, gy = 0;                                // the momentum's error estimate
    for (int l = 1; l <= 7; ++l) {
        gx += E[l] * (double)fx[l];
        gy += E[l] * (double)fy[l];
    }
    *error = (double)h * sqrt(gx * gx + gy * gy);
    o.w = w0(kA, k, o.x, o.y, w, tol);
    force(k, o.w, o.fx, o.fy);
    return o;
}

static F2 floats2(Q x) { const float h = (float)x; return {h, (float)(x - h)}; }
static F3 floats3(Q x) { const float h = (float)x, m = (float)(x - h); return {h, m, (float)(x - h - m)}; }
static Z3 pair3(Q x, Q y)
{
    const F3 a = floats3(x), b = floats3(y);
    return {{a.h, b.h}, {a.m, b.m}, {a.l, b.l}};
}
static Q qx(Z3 a) { return (Q)a.h.x + a.m.x + a.l.x; }
static Q qy(Z3 a) { return (Q)a.h.y + a.m.y + a.l.y; }

int main(int argc, char** argv)
{
    if (argc < 6) return 2;
    const bool rk = !strcmp(argv[1], "rk4");
    const double kA = atof(argv[2]);
    double kh = atof(argv[3]);
    const int rays = atoi(argv[4]), steps = atoi(argv[5]);
    const double tol = argc > 6 ? atof(argv[6]) : 1e-6;
    if (kh == 0.0) {                                      // the largest step that the range takes
        double lo = 1e-6, hi = 1.0;
        for (int it = 0; it < 100; ++it) {
            kh = 0.5 * (lo + hi);
            (split_in_range(rk, kA, kh) ? lo : hi) = kh;
        }
        kh = lo;
    }
    if (!split_in_range(rk, kA, kh)) return 3;
    const double h = kh / (2 * kPi), top = 1.96, tolD = 1e-17;
    const Q hq = h, tolQ = (Q)1e-31;
    srand(7);
    auto uniform = [] { return rand() / (double)RAND_MAX; };
    for (int n = 0; n < rays; ++n) {
        const double u = uniform() - 0.5, el = (10 + 50 * uniform()) * kPi / 180, az = 1.5 * uniform();
        const bool up = n & 1;                            // from a crest's height upwards, or from the top down
        const double y0 = up ? kA / (2 * kPi) + 0.01 : top - kA / (2 * kPi);
        Ray<Q> q = {};
        q.x = u;
        q.y = y0;
        q.w = w0<Q>(kA, kQ, q.x, q.y, {0, 0}, tolQ);
        const double nn = 1.0 / sqrt((double)((1 + q.w.r) * (1 + q.w.r) + q.w.i * q.w.i));
        const double px = nn * cos(el) * cos(az), py = (up ? 1 : -1) * nn * sin(el);
        q.px = px;
        q.py = py;
        force(kQ, q.w, q.fx, q.fy);
        Ray<double> d = {u, y0, px, py, {(double)q.w.r, (double)q.w.i}, 0, 0};
        force(2 * kPi, d.w, d.fx, d.fy);
        Ray<double> v = d;                                // Dormand-Prince with carried W0
        SplitState s = {};
        const F2 kappa = floats2(kQ * hq * kQ * hq);
        s.t = pair3(-kQ * q.y, kQ * q.x);
        s.q = pair3(-kQ * hq * q.py, kQ * hq * q.px);
        s.w = split3((double)q.w.r, (double)q.w.i);
        Z2 r;
        split_force(hi2(s.w), kappa, s.f, r);
        s.r = r.h;
        double hs = h;
        for (int it = 0; it < steps; ++it) {
            if (rk) {
                q = rk4<Q>(kA, kQ, tolQ, q, hq);
                d = rk4<double>(kA, 2 * kPi, tolD, d, h);
                SplitState o;
                split_step(s, kappa, o);
                s = o;
            } else {
                double e, ignored;
                const Ray<Q> o = dp45<Q, false>(kA, kQ, tolQ, q, (Q)hs, &e);
                e /= 2 * tol;
                const double grow = fmin(5.0, fmax(0.2, 0.9 * pow(e + 1e-30, -0.2)));
                if (e > 1) {
                    hs *= fmin(grow, 1.0);
                    continue;
                }
                q = o;
                d = dp45<double, false>(kA, 2 * kPi, tolD, d, hs, &ignored);
                v = dp45<double, true>(kA, 2 * kPi, tolD, v, hs, &ignored);
                hs = fmin(hs * grow, h);
            }
            if ((double)(q.y + q.w.r / kQ) < 0.0 || (double)q.y > top) break;
        }
        auto worst = [&](Q x, Q y, Q a, Q b) {
            return fmax(fmax(fabs((double)(x - q.x)), fabs((double)(y - q.y))),
                        fmax(fabs((double)(a - q.px)), fabs((double)(b - q.py))));
        };
        const double ed = worst(d.x, d.y, d.px, d.py);
        const double es = rk ? worst(qy(s.t) / kQ, -qx(s.t) / kQ, qy(s.q) / (kQ * hq), -qx(s.q) / (kQ * hq))
                             : worst(v.x, v.y, v.px, v.py);
        printf("%.3e %.3e\n", ed, es);
    }
    return 0;
}
