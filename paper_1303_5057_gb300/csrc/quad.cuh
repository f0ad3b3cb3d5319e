// quad.cuh -- one RK4 step of a photon on four lanes of a warp.
//
// A warp issues at most one FP64 instruction every 64 cycles on GB300, whatever
// its active lanes (measured: 64.05 cycles for 1 to 32 lanes and for 1 to 8
// independent chains; an SM takes one per 19 cycles from four or more warps).
// One ray per lane therefore pays 64 cycles for each of the ~600 double
// operations of its step, 19 us, and a small image or the last long rays of a
// large one are bound by that latency.  Here the four lanes of a quad hold one
// ray: lane m owns component m of position and momentum (t, r, theta, phi),
// and each FP64 instruction (a "slot" below) does up to four different
// operations of the step, one per lane, with operands selected by lane and
// results exchanged by shuffles.  A step takes ~220 slots (about 60 of them the
// library's sincos), 14 000 cycles of the FP64 pipe; the selects and shuffles
// between dependent slots bring it to 12.7 us (19.3 us with one lane per ray:
// 64^2 image 45 -> 29 ms).  Counters: 2800 warp instructions per step, 220 of
// them FP64; stalls "wait" 3.8 and "short scoreboard" 3.2 per instruction, so
// the exchange latency between slots, not the pipe, is what is left.
//
// Every value is formed by the same operations on the same operands as in
// step_once<double, false>, with every product-sum contraction written out on
// both sides (plain_add, mul_add and fma there), so a ray's result is the same
// bits in both whatever the compiler does.  A product alone is taken as
// fma(x, y, -0), which rounds and signs as x * y does.
//
// All lanes of the warp run every slot (idle quads on a harmless state), so
// the shuffles always have the full warp; the rare paths are entered by the
// warp together and their results selected per quad.
#pragma once

#include "kerr.cuh"

namespace gray {

constexpr unsigned QUAD_FULL = 0xffffffffu;

__device__ __forceinline__ double qget(double x, int src) { return __shfl_sync(QUAD_FULL, x, src, 4); }
__device__ __forceinline__ double qsel(int m, double a, double b, double c, double d)
{
    const double lo = (m & 1) ? b : a, hi = (m & 1) ? d : c;
    return (m & 2) ? hi : lo;
}
__device__ __forceinline__ double qmul(double x, double y) { return fma(x, y, -0.0); }

// |d| <= t for a positive t whose low word is 0, on the integer pipe.
__device__ __forceinline__ bool qabs_le(double d, int t_hi)
{
    const int hi = __double2hiint(d) & 0x7fffffff;
    return hi < t_hi || (hi == t_hi && __double2loint(d) == 0);
}

// The products of an acceleration that do not need the reciprocals of the
// geometry, each in the lane that uses it (see quad_finish).
struct QuadPre {
    double p0;  // t: X0 = k^t + V/2      r: M A            theta: r k^r k^th        phi: M a A
    double p1;  // t: P A                 r: Delta r (..)   theta: -2 k^ph           phi: -2M r^2
    double p2;  // t: r^2 V               r: a^2 r s^2      theta: (k^th)^2          phi: r k^ph
    double p3;  // t: 2 a^2 r s c         r: 2 a^2 s c      theta: s c               phi: 2 M a r
    double p4;  // r: k^r k^th            theta: P
    double kp2; // (k^ph)^2
};

// The last ten slots of an acceleration: lane m returns dk^m/dl (accel_geo's
// expressions).
__device__ __forceinline__ double quad_finish(const Hole<double> &H, const Geo<double> &g, const QuadPre &q, int m,
                                              double kr, double kh, double kp, double &fa, double &fb)
{
    // X = X0/Sigma, u = k^r/Delta, cot = c/s
    const double v1 = qmul(qsel(m, q.p0, kr, g.c, g.c), qsel(m, g.iS, g.iD, g.is, g.is));
    const double X = qget(v1, 0), u = qget(v1, 1);
    // k^th X, q = k^r u, a X - 2 k^ph, Z = 2 M a r X
    const double v2 = fma(qsel(m, kh, kr, H.a, q.p3), qsel(m, X, u, X, X), qsel(m, -0.0, -0.0, q.p1, -0.0));
    const double qq = qget(v2, 1), Z = qget(v2, 3);
    // ut = P A X + r^2 V, Delta X, (k^th)^2 - q, M a A X
    const double v3 = fma(qsel(m, q.p1, g.Delta, 1.0, q.p0), m == 2 ? q.p2 : X, qsel(m, q.p2, -0.0, -qq, -0.0));
    // xt, q - Delta X^2, a^2 ((k^th)^2 - q), M a A X - 2 M r^2 k^ph
    const double v4 = fma(qsel(m, -q.p3, -v3, H.a2, q.p1), qsel(m, v2, X, v3, kp), qsel(m, -0.0, qq, -0.0, v3));
    // u ut + xt, M A (..) + Delta r (..), P (k^ph)^2 + .., inner
    const double v5 = fma(qsel(m, u, q.p0, q.p4, g.iS), qsel(m, v3, v4, q.kp2, v4), qsel(m, v4, q.p1, v4, q.p2));
    // -2M/Sigma, .. - a^2 r s^2 q, h_th, k^ph - Z/Sigma
    const double v6 = fma(qsel(m, H.m2M, -q.p2, Z, -Z), qsel(m, g.iS, qq, v2, g.iS), qsel(m, -0.0, v5, v5, kp));
    // a^t, .. + 2 a^2 s c k^r k^th, s c h_th, cot k^th
    const double v7 = fma(qsel(m, v6, q.p3, q.p3, v1), qsel(m, v5, q.p4, v6, kh), qsel(m, -0.0, v6, -0.0, -0.0));
    // s c h_th - 2 r k^r k^th, cot k^th (k^ph - Z/Sigma)
    const double v8 = fma(m == 2 ? q.p0 : v7, m == 2 ? -2.0 : v6, m == 2 ? v7 : -0.0);
    const double v9 = fma(u, v5, v8); // u inner + ..
    fa = qsel(m, v6, g.iS, g.iS, -2.0);
    fb = qsel(m, v5, v7, v8, v9);
    return qmul(fa, fb);
}

// The geometry and the products of QuadPre at one point.  Without a full sine
// and cosine at hand (STAGE) lanes 0 and 1 form them from the step's start
// point (s0, c0) and the angle increment d, by small_sincos's two ranges and
// the angle addition, while lanes 2 and 3 form what needs r and k alone;
// `far` takes sf, cf instead.  Without STAGE sf, cf are the sine and cosine.
// The reciprocal of Sigma Delta sin is refined in lane 1 beside the products
// that do not need it.
template <bool STAGE>
__device__ __forceinline__ void quad_point(const Hole<double> &H, int m, double r, double d, double s0, double c0,
                                           bool tiny_all, bool far, double sf, double cf, double kt, double kr,
                                           double kh, double kp, Geo<double> &g, QuadPre &q)
{
    const bool co = m & 1;
    g.r = r;
    // d^2, d^2, r - r_+, r^2
    const double v0 = fma(m < 2 ? d : r, qsel(m, d, d, 1.0, r), m == 2 ? -H.rp : -0.0);
    const double r2 = qget(v0, 3);
    double p = co ? 2.48015873015873e-05 : -1.984126984126984e-04;
    if (STAGE && !tiny_all) { // two more terms for |d| in (1/64, 1/4]
        const double y = fma(v0, co ? 2.08767569878681e-09 : -2.505210838544172e-08,
                             co ? -2.755731922398589e-07 : 2.7557319223985893e-06);
        const double z = fma(y, v0, p);
        p = qabs_le(d, 0x3F900000) ? p : z;
    }
    // series, series, r - r_-, r^2 + a^2
    const double v1 = fma(m < 2 ? p : m == 2 ? r : r2, m < 2 ? v0 : 1.0,
                          qsel(m, 8.333333333333333e-03, -1.388888888888889e-03, -H.rm, H.a2));
    // series, series, Delta, -2M r^2
    const double v2 = fma(m == 3 ? H.m2M : v1, m == 3 ? r2 : v0,
                          qsel(m, -1.6666666666666666e-01, 4.1666666666666664e-02, H.dc, -0.0));
    // series, series, Delta r, r k^ph
    const double v3 = fma(m == 3 ? r : v2, m < 2 ? v0 : m == 2 ? r : kp, m == 1 ? -0.5 : -0.0);
    const double Delta = qget(v2, 2), P = qget(v1, 3);
    // sin d, cos d, (k^th)^2, k^r k^th
    const double v4 = fma(m < 2 ? v3 : kh, qsel(m, d, v0, kh, kr), qsel(m, d, 1.0, -0.0, -0.0));
    const double sd = qget(v4, 0), cd = qget(v4, 1), kh2 = qget(v4, 2), krkh = qget(v4, 3);
    // c0 sin d, s0 sin d, (k^ph)^2, 2 M a r
    const double v5 = qmul(qsel(m, c0, s0, kp, H.t2Ma), m < 2 ? sd : m == 2 ? kp : r);
    // sin, cos, r k^r k^th, a^2 r
    const double v6 = fma(qsel(m, s0, c0, r, H.a2), m < 2 ? cd : m == 2 ? krkh : r, m == 0 ? v5 : m == 1 ? -v5 : -0.0);
    if (STAGE) {
        const double s = qget(v6, 0), c = qget(v6, 1);
        g.s = far ? sf : s;
        g.c = far ? cf : c;
    } else {
        g.s = sf;
        g.c = cf;
    }
    g.Delta = Delta;
    q.kp2 = qget(v5, 2);
    const double a2r = qget(v6, 3);
    // s^2, c^2, s c, Delta s
    const double v7 = qmul(qsel(m, g.s, g.c, g.s, Delta), m == 0 || m == 3 ? g.s : g.c);
    const double s2 = qget(v7, 0), sc = qget(v7, 2);
    // 2 a s^2, Sigma, r s c, 2 a^2 s c
    const double v8 = fma(qsel(m, H.t2a, H.a2, r, H.t2a2), m < 2 ? v7 : sc, m == 1 ? r2 : -0.0);
    g.Sigma = qget(v8, 1);
    // V, Sigma Delta, A = 2 r^2 - Sigma, Sigma s
    const double v9 = fma(qsel(m, -v8, Delta, 2.0, g.s), qsel(m, kp, g.Sigma, r2, g.Sigma), m == 2 ? -g.Sigma : -0.0);
    const double A = qget(v9, 2), ds = qget(v7, 3), ss = qget(v9, 3);
    // X0, Sigma Delta s, M A, P A
    const double v10 = fma(qsel(m, 0.5, g.s, H.M, P), m == 3 ? A : v9, m == 0 ? kt : -0.0);
    // the reciprocal's Newton steps in lane 1 (recip's four operations) beside
    // r^2 V, -, 2 a^2 r s c, M a A;  -, -, s^2 (k^ph)^2 + (k^th)^2, a^2 r s^2;
    // -, -, Delta r (..), -;  -, -, -2 k^ph, -
    double inv;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(inv) : "d"(v10));
    const double v11 = fma(qsel(m, r2, -v10, H.t2a2, H.Ma), qsel(m, v9, inv, v8, A), m == 1 ? 1.0 : -0.0);
    const double v12 = fma(qsel(m, s2, inv, s2, a2r), qsel(m, q.kp2, v11, q.kp2, s2), m == 1 ? inv : m == 3 ? -0.0 : kh2);
    const double v13 = fma(m == 1 ? -v10 : v12, m == 2 ? v3 : v12, m == 1 ? 1.0 : -0.0);
    const double v14 = fma(m == 1 ? v12 : kp, m == 1 ? v13 : -2.0, m == 1 ? v12 : -0.0);
    // 1/Sigma, 1/sin, 1/Delta
    const double v15 = qmul(qget(v14, 1), m == 0 ? ds : m == 1 ? v9 : ss);
    g.iS = qget(v15, 0);
    g.is = qget(v15, 1);
    g.iD = qget(v15, 2);
    const double MA = qget(v10, 2), PA = qget(v10, 3), Dss = qget(v13, 2), a2rs2 = qget(v12, 3), sc2a2 = qget(v8, 3);
    const double rsc2a2 = qget(v11, 2);
    q.p0 = qsel(m, v10, MA, v6, v11);
    q.p1 = qsel(m, PA, Dss, v14, v2);
    q.p2 = qsel(m, v11, a2rs2, kh2, v3);
    q.p3 = qsel(m, rsc2a2, sc2a2, sc, v5);
    q.p4 = m == 1 ? krkh : P;
}

// Eq. 4 test at the new point (xi_fails): uniform over the quad.
__device__ __forceinline__ bool quad_xi_fails(const Hole<double> &H, const Geo<double> &g, int m, double kt, double kr,
                                              double kh, double kp, double eps)
{
    const double s2 = qmul(g.s, g.s);
    // a s2, r^2 + a^2, (k^th)^2, -2M r
    const double w1 = fma(qsel(m, H.a, g.r, kh, H.m2M), qsel(m, s2, g.r, kh, g.r), qsel(m, -0.0, H.a2, -0.0, -0.0));
    // w, a k^t, k^r/Delta, 1 - 2M r/Sigma
    const double w2 = fma(qsel(m, -w1, H.a, kr, w1), qsel(m, kp, kt, g.iD, g.iS), qsel(m, kt, -0.0, -0.0, 1.0));
    // Delta w, v, (k^r)^2/Delta + (k^th)^2, (k^t)^2
    const double w3 = fma(qsel(m, g.Delta, w1, w2, kt), qsel(m, w2, kp, kr, kt), qsel(m, -0.0, -w2, w1, -0.0));
    // (Delta w) w, s2 v, -, g_tt (k^t)^2
    const double w4 = qmul(qsel(m, w3, s2, s2, w2), qsel(m, w2, w3, w3, w3));
    const double dww = qget(w4, 0), q = qget(w3, 2);
    // E in lane 1, eps |g_tt (k^t)^2| in lane 3
    const double w5 = fma(m == 3 ? eps : w4, m == 3 ? fabs(w4) : w3, m == 3 ? -0.0 : -dww);
    const double w6 = qmul(w5, g.iS);
    const double norm = fma(g.Sigma, q, w6); // lane 1
    const double lim = qget(w5, 3);
    const bool ok = fabs(norm) <= lim;
    return !__shfl_sync(QUAD_FULL, (int)ok, 1, 4);
}

__device__ __forceinline__ bool qfinite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// Status codes of the ray and counters a step changes.
struct QuadStep {
    int status;   // as step_once
    bool redo;    // the step was redone as forward Euler (Eq. 4)
    bool remap;   // Eq. 3 was applied
};

// One step (step_once<double, false>) of the quad's ray: x and k are lane m's
// components, g and pre the geometry and products of the current point, fin
// the stop point (uniform, written when the ray stops).  `has`: the quad holds a ray.
// The statuses are those of gray.h, passed in so that this header stands alone.
template <int CAPTURED, int ESCAPED, int NONFINITE, int EQUATOR>
__device__ __forceinline__ QuadStep quad_step(const Hole<double> &H, const StepOpt<double> &O, int m, bool has,
                                              double &x, double &k, Geo<double> &g, QuadPre &pre, double *fin)
{
    QuadStep out{0, false, false};
    const double th0 = qget(x, 2);
    double h;
    {
        const double y[8] = {0.0, qget(x, 1), th0, 0.0, 0.0, qget(k, 1), qget(k, 2), qget(k, 3)};
        h = step_size(H, O, y);
    }
    const double hh = 0.5 * h;
    const double x0 = x, k0 = k;
    double a1, ks = k0, as, tk = 0.0, ta = 0.0, fa, fb;
    {
        const double kr = qget(k0, 1), kh = qget(k0, 2), kp = qget(k0, 3);
        a1 = quad_finish(H, g, pre, m, kr, kh, kp, fa, fb);
        as = a1;
    }
    // The three later stages in one rolled loop: a slot's 64 cycles hide the
    // shuffles and selects, and the shorter code stays in the instruction cache.
#pragma unroll 1
    for (int stage = 0; stage < 3; ++stage) {
        const double cs = stage < 2 ? hh : h;
        const double kh0 = qget(ks, 2);
        // -, r, theta, d = c_s h k^th of the stage before
        const double xs = fma(cs, m == 3 ? kh0 : ks, m == 3 ? -0.0 : x0);
        const double d = qget(xs, 3);
        ks = fma(cs, as, k0);
        const bool far = has && !qabs_le(d, 0x3FD00000); // |d| > 1/4 (or NaN): full sine and cosine
        const bool tiny_all = __all_sync(QUAD_FULL, !has || qabs_le(d, 0x3F900000));
        const double ths = qget(xs, 2);
        double sf = 0.0, cf = 1.0;
        if (__any_sync(QUAD_FULL, far))
            sincos(ths, &sf, &cf);
        const double kt = qget(ks, 0), kr = qget(ks, 1), kh = qget(ks, 2), kp = qget(ks, 3);
        Geo<double> gs;
        QuadPre qs;
        quad_point<true>(H, m, qget(xs, 1), d, g.s, g.c, tiny_all, far, sf, cf, kt, kr, kh, kp, gs, qs);
        as = quad_finish(H, gs, qs, m, kr, kh, kp, fa, fb);
        if (stage == 0) {
            tk = ks;
            ta = as;
        } else if (stage == 1) {
            tk += ks;
            ta = plain_add(ta, as);
        }
    }
    const double h6 = h * (1.0 / 6.0), h9 = h * (1.0 / 9.0);
    // t and phi take h v and the sum in two roundings.  -0 comes from the asm so
    // that the compiler cannot see a bare product here and contract it into the
    // sum (plain_add, which forbids that too, took 1.4 % longer here).
    const bool tp = m == 0 || m == 3;
    double nz = -0.0;
    asm("" : "+d"(nz));
    double x1 = fma(h6, fma(2.0, tk, k0) + ks, tp ? nz : x0);
    double k1 = fma(h6, fma(fa, fb, fma(2.0, ta, a1)), k0);
    if (tp)
        x1 += x0;

    // sin and cos of the new angle in lanes 0 and 1, and of the angle a
    // forward-Euler redo would end at in lanes 2 and 3: a ray that crawls on
    // redos needs both every step
    const double xe = fma(h9, k0, tp ? nz : x0);
    const double th_rk = qget(x1, 2), th_eu = qget(xe, 2);
    double sv, cv;
    sincos(m < 2 ? th_rk : th_eu, &sv, &cv);
    Geo<double> g1;
    bool redo;
    {
        const double kt = qget(k1, 0), kr = qget(k1, 1), kh = qget(k1, 2), kp = qget(k1, 3);
        quad_point<false>(H, m, qget(x1, 1), 0.0, 0.0, 1.0, true, false, qget(sv, 0), qget(cv, 0), kt, kr, kh, kp, g1,
                          pre);
        redo = quad_xi_fails(H, g1, m, kt, kr, kh, kp, O.eps_xi);
        redo = redo && has;
    }
    if (__any_sync(QUAD_FULL, redo)) {
        const double ke = fma(h9, a1, k0);
        Geo<double> ge;
        QuadPre qe;
        quad_point<false>(H, m, qget(xe, 1), 0.0, 0.0, 1.0, true, false, qget(sv, 2), qget(cv, 2), qget(ke, 0),
                          qget(ke, 1), qget(ke, 2), qget(ke, 3), ge, qe);
        if (redo) {
            h = h9;
            x1 = tp ? xe + x0 : xe;
            k1 = ke;
            g1 = ge;
            pre = qe;
        }
    }
    out.redo = redo;

    // the rare outcomes, as in step_once, behind one warp-uniform test
    const double r1 = qget(x1, 1), th1 = qget(x1, 2);
    const int quad = threadIdx.x & 28;
    const bool finite = ((__ballot_sync(QUAD_FULL, qfinite(x1) && qfinite(k1)) >> quad) & 15u) == 15u;
    const double half_pi = 0.5 * pi_v<double>();
    const bool equator = O.stop_equator && (th0 - half_pi) * (th1 - half_pi) < 0.0;
    // r <= r_cap, r_esc <= r, theta <= pi, 0 <= theta, one per lane
    const bool cmp = qsel(m, r1, H.r_esc, th1, 0.0) <= qsel(m, H.r_cap, r1, pi_v<double>(), th1);
    const unsigned bits = (__ballot_sync(QUAD_FULL, cmp) >> quad) & 15u;
    const bool rare = has && (!finite || equator || bits != 12u);
    if (__any_sync(QUAD_FULL, rare)) {
        double y0[8], y1[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            y0[j] = qget(x0, j);
            y0[4 + j] = qget(k0, j);
            y1[j] = qget(x1, j);
            y1[4 + j] = qget(k1, j);
        }
        if (rare) {
            if (!finite) {
                out.status = NONFINITE;
                for (int j = 0; j < 4; ++j)
                    fin[j] = y1[j];
            } else if (equator) {
                equator_crossing(y0, y1, h, fin);
                out.status = EQUATOR;
            } else if (r1 <= H.r_cap) {
                stop_surface(y0, y1, h, H.r_cap, fin);
                out.status = CAPTURED;
            } else if (r1 >= H.r_esc && h * y1[5] > 0.0) {
                stop_surface(y0, y1, h, H.r_esc, fin);
                out.status = ESCAPED;
            }
            if (out.status != NONFINITE && (th1 > pi_v<double>() || th1 < 0.0)) { // Eq. 3
                const bool over = th1 > pi_v<double>();
                if (m == 2) {
                    x1 = over ? 2.0 * pi_v<double>() - x1 : -x1;
                    k1 = -k1;
                }
                if (m == 3)
                    x1 = over ? x1 + pi_v<double>() : x1 - pi_v<double>();
                out.remap = true;
            }
        }
        if (__any_sync(QUAD_FULL, out.remap)) {
            double s, c;
            sincos(qget(x1, 2), &s, &c);
            Geo<double> gr;
            QuadPre qr;
            quad_point<false>(H, m, qget(x1, 1), 0.0, 0.0, 1.0, true, false, s, c, qget(k1, 0), qget(k1, 1),
                              qget(k1, 2), qget(k1, 3), gr, qr);
            if (out.remap) {
                g1 = gr;
                pre = qr;
            }
        }
    }
    x = x1;
    k = k1;
    g = g1;
    return out;
}

} // namespace gray
