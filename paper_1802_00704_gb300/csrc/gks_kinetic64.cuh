// Device arithmetic of the third-order BGK flux at one Gauss point (Sec. II.B)
// in FP64.  (The mixed flux forms its FP32 slope-carrying terms by
// gks_kinetic.cuh.)
//
// Everything is formed in the peculiar velocities of each state: with U, V its
// mean velocity (face frame, U along the normal) and h = p / rho the variance
// of a velocity component, x = (u - U) / sqrt(h), y = (v - V) / sqrt(h) and
// z = xi.xi / h are two standard normals and a chi-square of K degrees of
// freedom.  In the basis phi = (1, x, y, q), q = (x^2 + y^2 + z - N) / 2 with
// N = K + 2, the moment matrix <phi phi^T> is diag(1, 1, 1, N/2), so a slope
// (Eq. (12)) needs no matrix inverse, and every full-space moment is a number.
// Lengths are scaled by sqrt(h) as well (a slope along n or t is multiplied by
// it), which leaves the time of Eqs. (8)-(15) as it is.
//
// Notation of a state's slopes: al, be the slopes along n and t (coefficients
// in phi); T = A + (U al + V be) / sqrt(h) the slope along the mean motion; the
// second derivatives are products plus a linear part, d2g/dn2 / g = al al + nn,
// al be + nt, be be + tt, and along the mean motion T al + Tn, T be + Tt,
// T T + TT.  The compatibility conditions <phi Dg/Dt> = 0 and their derivatives
// along n, t and the mean motion read
//   <phi (T + x al + y be)> = 0,   <phi (T al + Tn + x (al al + nn) + y (al be + nt))> = 0, ...
// The FP64 flux kernels are bound by the FP64 pipe (91 % busy), so this form is
// there for its operation count: about 480 multiply-adds per state, a third of
// the sums over monomials in (u, v, e) that it replaced.  Measured on GB300 at
// 399,424 triangles (1.2 M Gauss points): 8,392 -> 4,262 FP64 operations per
// point, 10.3 -> 5.75 ms per launch; 100,003 state pairs 935 -> 488 us.  Projections
// subtracted in place, the full-space moments in closed form and the reconstruction
// straight into the face frame: 2,690 -> 2,511 instructions, 5.75 -> 5.32 ms, 488 -> 471 us.
#pragma once

#include <cuda_runtime.h>

namespace gks {
namespace kin64 {

// Moments that depend on the number of degrees of freedom N = K + 2 alone;
// g = (y^2 + z - M) / 2 is the part of q without x, M = N - 1 its degrees.
template <typename R>
struct Gas {
    R N, hN, iN2;     // N, N / 2 = <q^2>, 2 / N
    R c33;            // <x^2 q^2> = 2 + N / 2
    R M, G2;          // M = <g^3>, M / 2 = <g^2>
    R g22, yg3;       // <y^2 g^2> = 2 + M / 2, <y^2 g^3> = 6 + 5 M / 2
};

template <typename R>
__device__ __forceinline__ Gas<R> gas(R K)
{
    Gas<R> c;
    c.N = K + R(2);
    c.hN = R(0.5) * c.N;
    c.iN2 = R(2) / c.N;
    c.c33 = R(2) + c.hN;
    c.M = K + R(1);
    c.G2 = R(0.5) * c.M;
    c.g22 = R(2) + c.G2;
    c.yg3 = R(6) + R(2.5) * c.M;
    return c;
}

template <typename R>
struct State {
    R rho, U, V, p, h;     // h = p / rho = 1 / (2 lambda), Eq. (3)
    R ir, sg, isg;         // 1 / rho, sqrt(h), 1 / sqrt(h)
    R a, b;                // U / sqrt(h), V / sqrt(h)
};

// Primitive variables of a state (rho, rho U, rho V, E); false unless rho > 0 and p > 0,
// and for a SIDE of the face unless four times its internal energy is in range (the
// sums over both sides would overflow; tested on the exponent, off the FP64 pipe).
template <bool SIDE = false, typename R>
__device__ __forceinline__ bool prim(const R *w, R gamma, State<R> &s)
{
    s.rho = w[0];
    s.ir = R(1) / w[0];
    s.U = w[1] * s.ir;
    s.V = w[2] * s.ir;
    const R eint = w[3] - R(0.5) * (w[1] * s.U + w[2] * s.V);
    s.p = (gamma - R(1)) * eint;
    s.h = s.p * s.ir;
    s.isg = rsqrt(s.h);
    s.sg = s.h * s.isg;
    s.a = s.U * s.isg;
    s.b = s.V * s.isg;
    const bool fits = !SIDE || (__double2hiint(eint) & 0x7ff00000) < 0x7fd00000;     // |eint| < 2^1022
    return s.rho > R(0) && s.p > R(0) && fits;
}

// Moments <x^k>, k < 10, over u > 0 (sign = +1: x > -a) or u < 0 (sign = -1),
// from m0 = <1> and the density pdf = exp(-a^2/2) / sqrt(2 pi) at the edge x = -a.
template <typename R>
__device__ __forceinline__ void half_edge(R a, R sign, R &m0, R &pdf)
{
    m0 = R(0.5) * erfc(-sign * R(0.70710678118654752440) * a);
    pdf = R(0.39894228040143267794) * exp(R(-0.5) * a * a);
}

template <typename R>
__device__ __forceinline__ void half_moments(R a, R sign, R m0, R pdf, R *m)
{
    R e = sign * pdf;                      // sign (-a)^k pdf
    m[0] = m0;
    m[1] = e;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        e *= -a;
        m[k + 2] = R(k + 1) * m[k] + e;
    }
}

// Conservative moments <psi f>, psi = (1, u, v, e), from M = <phi f>.
template <typename R>
__device__ __forceinline__ void to_psi(const State<R> &s, const Gas<R> &c, const R *M, R *o)
{
    const R ke = R(0.5) * (s.U * s.U + s.V * s.V) + c.hN * s.h;
    o[0] = M[0];
    o[1] = s.U * M[0] + s.sg * M[1];
    o[2] = s.V * M[0] + s.sg * M[2];
    o[3] = ke * M[0] + s.sg * (s.U * M[1] + s.V * M[2]) + s.h * M[3];
}

// ---- slopes

template <typename R>
struct Slopes {
    R al[4], be[4], nn[4], nt[4], tt[4];     // from the derivative rows
    R T[4], Tn[4], Tt[4], TT[4];             // from the compatibility conditions
};

// o -= <phi s t>, the q entry over N / 2 (the coefficients of the projection of s t)
template <typename R>
__device__ __forceinline__ void sub_proj(const Gas<R> &c, const R *s, const R *t, R *o)
{
    const R s03 = s[0] + s[3], t03 = t[0] + t[3];
    o[0] -= s[0] * t[0];
    o[0] -= s[1] * t[1];
    o[0] -= s[2] * t[2];
    o[0] -= c.hN * s[3] * t[3];
    o[1] -= s03 * t[1];
    o[1] -= s[1] * t03;
    o[2] -= s03 * t[2];
    o[2] -= s[2] * t03;
    o[3] -= s[3] * t03;
    o[3] -= s03 * t[3];
    o[3] -= c.iN2 * (s[1] * t[1] + s[2] * t[2]);
}

// entries 1 (D = 1) or 2 (D = 2), 3 - D and 3 of <phi d s t>, d = x (D = 1) or y (D = 2), taken off o
template <int D, typename R>
__device__ __forceinline__ void sub_proj_dir(const Gas<R> &c, const R *s, const R *t, R *o)
{
    constexpr int E = 3 - D;
    const R t03 = t[0] + t[3], t033 = t[0] + c.c33 * t[3], s033 = s[0] + c.c33 * s[3];
    o[D] -= s[0] * t03;
    o[D] -= s[3] * t033;
    o[D] -= R(3) * s[D] * t[D];
    o[D] -= s[E] * t[E];
    o[E] -= s[1] * t[2];
    o[E] -= s[2] * t[1];
    o[3] -= c.iN2 * (t[D] * s033 + s[D] * t033);
}

// The linear part l of the derivative of a slope along the mean motion (or of
// the slope Tn, Tt themselves): l = -( proj(T, s) + <phi [x (pn + ln) + y (pt + lt)]> ) with the
// products pn = s al, pt = s be; r0 = <x (pn + ln)> + <y (pt + lt)>, entry 0 of that.
template <typename R>
__device__ __forceinline__ void along(const Gas<R> &c, const R *T, const R *s, const R *al, const R *be, const R *ln,
                                      const R *lt, R r0, R *l)
{
    l[0] = -r0;
    l[1] = -(ln[0] + ln[3]);
    l[2] = -(lt[0] + lt[3]);
    l[3] = -c.iN2 * (ln[1] + lt[2]);
    sub_proj(c, T, s, l);
    sub_proj_dir<1>(c, s, al, l);
    sub_proj_dir<2>(c, s, be, l);
}

// Slopes of a state from the conservative derivative rows [5][4] (d/dn, d/dt,
// d2/dn2, d2/dndt, d2/dt2), times f.  TIME: also TT (the equilibrium state's).
template <bool TIME, typename R>
__device__ __forceinline__ void slopes(const State<R> &s, const Gas<R> &c, const R *rows, Slopes<R> &o, R f = R(1))
{
    const R ke = R(0.5) * (s.U * s.U + s.V * s.V);
    // rows to phi: d(rho), d(rho u) - U d(rho), ..., scaled by sqrt(h) (first) and h (second derivatives)
    const R ir = f * s.ir;
    const R f0[2] = {s.sg * ir, s.h * ir}, f1[2] = {ir, f0[0]}, f3[2] = {c.iN2 * ir * s.isg, c.iN2 * ir};
    R *const dst[5] = {o.al, o.be, o.nn, o.nt, o.tt};
#pragma unroll
    for (int r = 0; r < 5; ++r) {
        const R *d = rows + 4 * r;
        const int k = r >= 2;
        const R m1 = d[1] - s.U * d[0], m2 = d[2] - s.V * d[0];
        const R en = d[3] - s.U * d[1] - s.V * d[2] + ke * d[0];
        dst[r][0] = f0[k] * d[0];
        dst[r][1] = f1[k] * m1;
        dst[r][2] = f1[k] * m2;
        dst[r][3] = f3[k] * en - dst[r][0];
    }
    // <x (al al + nn)> etc. are entry 1 (2) of the rows themselves
    const R nn1 = o.nn[1], nt1 = o.nt[1], nt2 = o.nt[2], tt2 = o.tt[2];
    sub_proj(c, o.al, o.al, o.nn);
    sub_proj(c, o.al, o.be, o.nt);
    sub_proj(c, o.be, o.be, o.tt);
    const R div = o.al[1] + o.be[2];
    o.T[0] = -div;
    o.T[1] = -(o.al[0] + o.al[3]);
    o.T[2] = -(o.be[0] + o.be[3]);
    o.T[3] = -c.iN2 * div;
    along(c, o.T, o.al, o.al, o.be, o.nn, o.nt, nn1 + nt2, o.Tn);
    along(c, o.T, o.be, o.al, o.be, o.nt, o.tt, nt1 + tt2, o.Tt);
    if (TIME) {
        // <x (T al + Tn)> and <y (T be + Tt)>
        const R x = (o.T[0] + o.T[3]) * o.al[1] + o.T[1] * (o.al[0] + o.al[3]) + o.Tn[1];
        const R y = (o.T[0] + o.T[3]) * o.be[2] + o.T[2] * (o.be[0] + o.be[3]) + o.Tt[2];
        along(c, o.T, o.T, o.al, o.be, o.Tn, o.Tt, x + y, o.TT);
    }
}

// ---- moments of the distribution's expansion
//
// A slope s with coefficients in phi is S(x) + s2 y + s3 g, S(x) = (s0 - s3/2) +
// s1 x + (s3/2) x^2.  The expansion Q (polynomial in x, y, g) is reduced to its
// means over y and z at given x: E0 = <Q>, Eg = <g Q>, Ey = <y Q>, polynomials
// in x; the half-space or full-space moments in x close the integrals.

template <typename R>
struct Cond {
    R e[7], g[5], y[6];    // E0, Eg, Ey
};

// S(x) with y and g parts that may depend on x: p[NP], two[ND], three[ND]
template <typename R, int NP, int ND>
struct Lin {
    R p[NP], two[ND], thr[ND];
};

template <typename R>
__device__ __forceinline__ Lin<R, 3, 1> lin(const R *s)
{
    Lin<R, 3, 1> o;
    const R h3 = R(0.5) * s[3];
    o.p[0] = s[0] - h3;
    o.p[1] = s[1];
    o.p[2] = h3;
    o.two[0] = s[2];
    o.thr[0] = s[3];
    return o;
}

// (s + f x t) of two slopes: one degree more in x
template <typename R>
__device__ __forceinline__ Lin<R, 4, 2> lin_x(const R *s, R f, const R *t)
{
    Lin<R, 4, 2> o;
    const R h3 = R(0.5) * s[3], k1 = f * t[1], k2 = f * t[2], k3 = f * t[3], h = R(0.5) * k3;
    o.p[0] = s[0] - h3;
    o.p[1] = s[1] + f * t[0] - h;
    o.p[2] = h3 + k1;
    o.p[3] = h;
    o.two[0] = s[2];
    o.two[1] = k2;
    o.thr[0] = s[3];
    o.thr[1] = k3;
    return o;
}

// out[off + i + j] += f_i g_j
template <int OFF, typename R, int NF, int NG>
__device__ __forceinline__ void mac(R *out, const R (&f)[NF], const R (&g)[NG])
{
#pragma unroll
    for (int i = 0; i < NF; ++i)
#pragma unroll
        for (int j = 0; j < NG; ++j) out[OFF + i + j] += f[i] * g[j];
}

template <int OFF, typename R, int NF>
__device__ __forceinline__ void axpy(R *out, R f, const R (&g)[NF])
{
#pragma unroll
    for (int i = 0; i < NF; ++i) out[OFF + i] += f * g[i];
}

// Q += x^OFF s t
template <int OFF, typename R, int NP, int ND>
__device__ __forceinline__ void add0(const Gas<R> &c, Cond<R> &Q, const Lin<R, 3, 1> &s, const Lin<R, NP, ND> &t)
{
    const R s2 = s.two[0], s3 = s.thr[0], k3 = c.G2 * s3;
    mac<OFF>(Q.e, s.p, t.p);                      // <s t> = S T + s2 t2 + <g^2> s3 t3
    axpy<OFF>(Q.e, s2, t.two);
    axpy<OFF>(Q.e, k3, t.thr);
    axpy<OFF>(Q.g, k3, t.p);                      // <g s t> = <g^2> (s3 T + t3 S) + s2 t2 + <g^3> s3 t3
    axpy<OFF>(Q.g, s2, t.two);
    axpy<OFF>(Q.g, c.M * s3, t.thr);
    R t3[ND];
#pragma unroll
    for (int i = 0; i < ND; ++i) t3[i] = c.G2 * t.thr[i];
    mac<OFF>(Q.g, s.p, t3);
    axpy<OFF>(Q.y, s2, t.p);                      // <y s t> = s2 T + t2 S + s2 t3 + s3 t2
    axpy<OFF>(Q.y, s2, t.thr);
    axpy<OFF>(Q.y, s3, t.two);
    mac<OFF>(Q.y, s.p, t.two);
}

// Q += y s t
template <typename R, int NP, int ND>
__device__ __forceinline__ void add1(const Gas<R> &c, Cond<R> &Q, const Lin<R, 3, 1> &s, const Lin<R, NP, ND> &t)
{
    const R s2 = s.two[0], s3 = s.thr[0];
    R c2[NP] = {}, c2s[ND] = {};                  // s2 T + t2 S; s2 t3 + s3 t2
    axpy<0>(c2, s2, t.p);
    mac<0>(c2, s.p, t.two);
    axpy<0>(c2s, s2, t.thr);
    axpy<0>(c2s, s3, t.two);
    axpy<0>(Q.e, R(1), c2);
    axpy<0>(Q.e, R(1), c2s);
    axpy<0>(Q.g, R(1), c2);                       // <y g s t>
    axpy<0>(Q.g, c.g22, c2s);
    mac<0>(Q.y, s.p, t.p);                        // <y^2 s t> = S T + 3 s2 t2 + s3 T + t3 S + <y^2 g^2> s3 t3
    axpy<0>(Q.y, R(3) * s2, t.two);
    axpy<0>(Q.y, s3, t.p);
    mac<0>(Q.y, s.p, t.thr);
    axpy<0>(Q.y, c.g22 * s3, t.thr);
}

// Q += f y^2 s s
template <typename R>
__device__ __forceinline__ void add2(const Gas<R> &c, Cond<R> &Q, R f, const Lin<R, 3, 1> &s)
{
    const R s2 = s.two[0], s3 = s.thr[0];
    R ss[5] = {}, fs[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) fs[i] = f * s.p[i];
    mac<0>(ss, s.p, fs);
    const R f22 = f * s2 * s2, f33 = f * s3 * s3, f3 = R(2) * s3, f2 = R(6) * s2;
    axpy<0>(Q.e, R(1), ss);                       // <y^2 s s>
    axpy<0>(Q.e, f3, fs);
    Q.e[0] += R(3) * f22 + c.g22 * f33;
    axpy<0>(Q.g, R(1), ss);                       // <y^2 g s s>
    axpy<0>(Q.g, c.g22 * f3, fs);
    Q.g[0] += R(6) * f22 + c.yg3 * f33;
    axpy<0>(Q.y, f2, fs);                         // <y^3 s s> = 6 s2 S + 12 s2 s3
    Q.y[0] += R(2) * f2 * (f * s3);
}

// Time coefficients of the expansion (Eqs. (11), (15)): 1, the slope in time, the slopes along the
// particle path, their squares, the mixed and the second time slopes.
template <typename R>
struct QCoef {
    R k1, kA, kL, kS, kAL, kAA;
};

// Q = k1 + kA A + kL (al u + be v) + kS [(al al + nn) u^2 + 2 (al be + nt) u v + (be be + tt) v^2]
//     + kAL [(A al + An) u + (A be + At) v] + kAA (A A + Att),
// written in the mean motion's slopes with D = a al + b be: the products sum to
// D (kappa D + mu T) + kAA T T + l E + kS l l, l = x al + y be,
// E = (2 kS - kAL) D + kAL T, kappa = kS - kAL + kAA, mu = kAL - 2 kAA.
template <bool EQ, typename R>
__device__ __forceinline__ void expand(const State<R> &s, const Gas<R> &c, const Slopes<R> &o, const QCoef<R> &k,
                                       Cond<R> &Q)
{
    const R kAA = EQ ? k.kAA : R(0);
    const R kap = k.kS - k.kAL + kAA, mu = k.kAL - R(2) * kAA, nu = R(2) * k.kS - k.kAL;
    R D[4], E[4], E1[4], L0[4], Lx[4], Ly[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        D[q] = s.a * o.al[q] + s.b * o.be[q];
        E[q] = nu * D[q] + k.kAL * o.T[q];
        E1[q] = kap * D[q] + mu * o.T[q];
        const R ln = s.a * o.nn[q] + s.b * o.nt[q], lt = s.a * o.nt[q] + s.b * o.tt[q];
        L0[q] = (k.kL - k.kA) * D[q] + k.kA * o.T[q] + kap * (s.a * ln + s.b * lt) +
                mu * (s.a * o.Tn[q] + s.b * o.Tt[q]);
        if (EQ) L0[q] += kAA * o.TT[q];
        Lx[q] = k.kL * o.al[q] + nu * ln + k.kAL * o.Tn[q];
        Ly[q] = k.kL * o.be[q] + nu * lt + k.kAL * o.Tt[q];
    }
    const R k2 = R(2) * k.kS;
    // the linear part: L0 + x Lx + kS x^2 nn + y (Ly + 2 kS x nt) + kS y^2 tt
    {
        const Lin<R, 3, 1> v0 = lin(L0), vx = lin(Lx), vxx = lin(o.nn), vy = lin(Ly), vxy = lin(o.nt), vyy = lin(o.tt);
        const R t3 = k.kS * vyy.thr[0];
        Q.e[0] = k.k1 + v0.p[0] + vy.two[0] + k.kS * vyy.p[0] + t3;
        Q.e[1] = v0.p[1] + vx.p[0] + k2 * vxy.two[0] + k.kS * vyy.p[1];
        Q.e[2] = v0.p[2] + vx.p[1] + k.kS * (vxx.p[0] + vyy.p[2]);
        Q.e[3] = vx.p[2] + k.kS * vxx.p[1];
        Q.e[4] = k.kS * vxx.p[2];
        Q.e[5] = Q.e[6] = R(0);
        Q.g[0] = c.G2 * v0.thr[0] + vy.two[0] + k.kS * vyy.p[0] + c.g22 * t3;
        Q.g[1] = c.G2 * vx.thr[0] + k2 * vxy.two[0] + k.kS * vyy.p[1];
        Q.g[2] = k.kS * (c.G2 * vxx.thr[0] + vyy.p[2]);
        Q.g[3] = Q.g[4] = R(0);
        Q.y[0] = v0.two[0] + vy.p[0] + vy.thr[0] + R(3) * k.kS * vyy.two[0];
        Q.y[1] = vx.two[0] + vy.p[1] + k2 * (vxy.p[0] + vxy.thr[0]);
        Q.y[2] = k.kS * vxx.two[0] + vy.p[2] + k2 * vxy.p[1];
        Q.y[3] = k2 * vxy.p[2];
        Q.y[4] = Q.y[5] = R(0);
    }
    const Lin<R, 3, 1> al = lin(o.al), be = lin(o.be);
    add0<0>(c, Q, lin(D), lin(E1));
    if (EQ) {
        R kT[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) kT[q] = kAA * o.T[q];
        add0<0>(c, Q, lin(o.T), lin(kT));
    }
    add0<1>(c, Q, al, lin_x(E, k.kS, o.al));      // x al (E + kS x al)
    add1(c, Q, be, lin_x(E, k2, o.al));           // y be (E + 2 kS x al)
    add2(c, Q, k.kS, be);                         // kS y^2 be be
}

// M = <phi Q> from the conditional means and the moments m of x
template <typename R>
__device__ __forceinline__ void close(const Cond<R> &Q, const R *m, R *M)
{
    R s0 = R(0), s1 = R(0), s2 = R(0), sg = R(0), sy = R(0);
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        s0 += Q.e[i] * m[i];
        s1 += Q.e[i] * m[i + 1];
        s2 += Q.e[i] * m[i + 2];
    }
#pragma unroll
    for (int i = 0; i < 5; ++i) sg += Q.g[i] * m[i];
#pragma unroll
    for (int i = 0; i < 6; ++i) sy += Q.y[i] * m[i];
    M[0] = s0;
    M[1] = s1;
    M[2] = sy;
    M[3] = R(0.5) * (s2 - s0) + sg;
}

// Over the whole line, <x^k> = 1, 0, 1, 0, 3, 0, 15, 0, 105: M = <phi Q> / sqrt(h) u and m = <phi Q>
template <typename R>
__device__ __forceinline__ void close_full(const Cond<R> &Q, R a, R *M, R *m)
{
    const R A = Q.e[0] + Q.e[2] + R(3) * Q.e[4] + R(15) * Q.e[6], B = Q.e[1] + R(3) * Q.e[3] + R(15) * Q.e[5];
    const R C = Q.e[0] + R(3) * Q.e[2] + R(15) * Q.e[4] + R(105) * Q.e[6];
    const R D = R(3) * Q.e[1] + R(15) * Q.e[3] + R(105) * Q.e[5];
    const R g = Q.g[0] + Q.g[2] + R(3) * Q.g[4], y = Q.y[0] + Q.y[2] + R(3) * Q.y[4];
    m[0] = A;
    m[1] = B;
    m[2] = y;
    m[3] = R(0.5) * (C - A) + g;
    const R s0 = a * A + B;
    M[0] = s0;
    M[1] = a * B + C;
    M[2] = a * y + (Q.y[1] + R(3) * Q.y[3] + R(15) * Q.y[5]);
    M[3] = R(0.5) * (a * C + D - s0) + (a * g + (Q.g[1] + R(3) * Q.g[3]));
}

// rho <u psi Q> (added to f) and, HEAT, rho <psi Q> (added to d); m: the moments of
// x over a half space, NULL: over the whole line
template <bool HEAT, typename R>
__device__ __forceinline__ void add_flux(const State<R> &s, const Gas<R> &c, const Cond<R> &Q, const R *m, R *f, R *d)
{
    R n[9], M[4], H[4], o[4];
    if (m) {
#pragma unroll
        for (int i = 0; i < 9; ++i) n[i] = s.a * m[i] + m[i + 1];     // <u x^i> / sqrt(h)
        close(Q, n, M);
        if (HEAT) close(Q, m, H);
    } else {
        close_full(Q, s.a, M, H);
    }
    to_psi(s, c, M, o);
    const R k = s.rho * s.sg;
#pragma unroll
    for (int q = 0; q < 4; ++q) f[q] += k * o[q];
    if (HEAT) {
        to_psi(s, c, H, o);
#pragma unroll
        for (int q = 0; q < 4; ++q) d[q] += s.rho * o[q];
    }
}

// Time integrals over [0, dt] of c1..c8 of Eq. (13) and of t^2 c7, with
// x = dt / tau: closed forms for x >= 1/2, power series where they cancel.
template <typename R>
__device__ __forceinline__ void time_integrals(R dt, R tau, int tau2_exact, R *C)
{
    const R x = dt / tau;
    R t0, t1, t2, c1, c2, c3;   // t_n = int_0^x s^n e^{-s} ds; c* the scaled C1, C2, C3
    if (x >= R(0.5)) {
        const R e = exp(-x);
        t0 = R(1) - e;                         // no cancellation: e <= 0.61
        t1 = t0 - x * e;
        t2 = R(2) * t1 - x * x * e;
        c1 = x - t0;
        c2 = t1 + t0 - x;
        c3 = R(0.5) * x * x - x + t0;
    } else {
        // t_n = sum_k (-1)^k x^{n+k+1} / (k! (n+k+1)); c1 = sum_{p>=2} (-1)^p x^p / p!;
        // c2 = sum_{p>=3} (-1)^p (p-2) x^p / p!;  c3 = sum_{p>=3} (-1)^{p+1} x^p / p!
        t0 = t1 = t2 = c1 = c2 = c3 = R(0);
        R xp = x;                              // x^{k+1} / k!
        R sg = R(1);
#pragma unroll
        for (int k = 0; k < 18; ++k) {         // term k: (-1)^k x^{k+1} / k!
            const R base = sg * xp;            // (-1)^k x^{k+1} / k!
            t0 += base * R(1.0 / (k + 1));
            t1 += base * x * R(1.0 / (k + 2));
            t2 += base * x * x * R(1.0 / (k + 3));
            xp *= x * R(1.0 / (k + 1));
            sg = -sg;
        }
        R pw = x * x * R(0.5);                   // x^p / p! starting at p = 2
        R s2 = R(1);                           // (-1)^p at p = 2
#pragma unroll
        for (int p = 2; p < 20; ++p) {
            c1 += s2 * pw;
            if (p >= 3) {
                c2 += s2 * R(p - 2) * pw;
                c3 -= s2 * pw;
            }
            pw *= x * R(1.0 / (p + 1));
            s2 = -s2;
        }
    }
    const R tau2 = tau * tau, tau3 = tau2 * tau;
    C[0] = tau * c1;                                   // int c1
    C[1] = tau2 * c2;                                  // int c2
    C[2] = tau2 * c3;                                  // int c3
    C[3] = -tau3 * (t2 + R(2) * t1);                   // int c4 (as printed)
    C[4] = tau3 * (x * x * x * R(1.0 / 3.0) - x * x);          // int c5 (as printed)
    C[5] = -tau3 * (R(0.5) * x * x + t1);              // int c6 (as printed)
    C[6] = tau * t0;                                   // int c7
    C[7] = -tau2 * t1;                                 // int c8
    C[8] = tau3 * t2;                                  // int t^2 c7
    if (tau2_exact) {
        const R k = R(2) * tau3 * c1;                  // 2 tau^2 int (1 - e^{-t/tau}) dt
        C[3] += k;
        C[4] += k;
        C[5] += k;
    }
}

// Interface data of one Gauss point: primitive left/right states with their
// half-space edge values, the interface equilibrium W0 = rho_l <psi>_{u>0} +
// rho_r <psi>_{u<0} with the sum of the left/right derivatives (of which it takes half), its primitive
// state, the collision time (Eqs. (39)-(40), pressure-jump term scaled by dt)
// and the time integrals.
template <typename R>
struct Iface {
    State<R> L, Rs, Z;
    R m0[2], pdf[2];       // <1> and the edge density of the two half spaces
    R w0[24];
    R tau;
    R C[9];
};

template <typename R>
__device__ __forceinline__ bool interface_state(const R *wl, const R *wr, R dt, R gamma, R mu, const Gas<R> &c,
                                                int tau2_exact, Iface<R> &I)
{
    if (!(prim<true>(wl, gamma, I.L) & prim<true>(wr, gamma, I.Rs))) return false;
#pragma unroll
    for (int q = 0; q < 4; ++q) I.w0[q] = R(0);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const State<R> &s = side ? I.Rs : I.L;
        const R sg = side ? R(-1) : R(1);
        half_edge(s.a, sg, I.m0[side], I.pdf[side]);
        // <phi> over the half space: <x> = +-pdf, <x^2> - <1> = -a <x>
        const R e = sg * I.pdf[side];
        const R M[4] = {I.m0[side], e, R(0), R(-0.5) * s.a * e};
        R o[4];
        to_psi(s, c, M, o);
#pragma unroll
        for (int q = 0; q < 4; ++q) I.w0[q] += s.rho * o[q];
    }
#pragma unroll
    for (int q = 4; q < 24; ++q) I.w0[q] = wl[q] + wr[q];
    if (!prim(I.w0, gamma, I.Z)) return false;
    const R jump = fabs(I.L.p - I.Rs.p) / fabs(I.L.p + I.Rs.p);
    I.tau = mu > R(0) ? mu / I.Z.p + dt * jump : R(0.01) * dt + dt * jump;
    time_integrals(dt, I.tau, tau2_exact, I.C);
    return true;
}

// Kinetic weighting of the interface derivatives (slope0_mode 1): the
// derivative rows of W0 become the half-space moments of the derivatives of
// the left and right distributions, rho_k <psi g_k'/g_k>_k (u > 0 left, u < 0
// right) with g_n/g = al, g_t/g = be, g_nn/g = al al + nn, g_nt/g = al be + nt,
// g_tt/g = be be + tt (scaled back by sqrt(h)): the derivatives of the value
// rho_l <psi>_{u>0} + rho_r <psi>_{u<0} when the two states vary as their
// reconstructions do.
template <typename R>
__device__ __forceinline__ void kinetic_w0(Iface<R> &I, const Gas<R> &c, const Slopes<R> &o, int side)
{
    const State<R> &s = side ? I.Rs : I.L;
    R m[10];
    half_moments(s.a, side ? R(-1) : R(1), I.m0[side], I.pdf[side], m);
    const R *const l[5] = {o.al, o.be, o.nn, o.nt, o.tt}, *const pa[5] = {nullptr, nullptr, o.al, o.al, o.be};
    const R *const pb[5] = {nullptr, nullptr, o.al, o.be, o.be};
#pragma unroll
    for (int r = 0; r < 5; ++r) {
        Cond<R> Q = {};
        const Lin<R, 3, 1> v = lin(l[r]);
        axpy<0>(Q.e, R(1), v.p);
        Q.g[0] = c.G2 * v.thr[0];
        Q.y[0] = v.two[0];
        if (r >= 2) add0<0>(c, Q, lin(pa[r]), lin(pb[r]));
        R M[4], w[4];
        close(Q, m, M);
        to_psi(s, c, M, w);
        const R f = s.rho * (r >= 2 ? s.isg * s.isg : s.isg);
#pragma unroll
        for (int q = 0; q < 4; ++q) I.w0[4 + 4 * r + q] += f * w[q];
    }
}

// Flux terms of Eqs. (11) and (15) at y = 0, from the slopes of the three
// states.  with_const = false leaves out the zeroth-order terms C1 g0 and
// C7 g_k.
//
// HEAT: also d_alpha = <psi_alpha f> (the time-integrated moments without the
// factor u), for the heat flux of the Prandtl correction.
// KIN: interface derivatives by kinetic weighting (kinetic_w0) instead of the
// mean of the left and right rows held in I.w0.
template <typename R, bool HEAT = false, bool KIN = false>
__device__ __forceinline__ void body_flux(const R *wl, const R *wr, Iface<R> &I, const Gas<R> &c, bool with_const,
                                          R *f, R *d = nullptr)
{
    const R tau = I.tau;
    const R *C = I.C;
    R m[10];
    Cond<R> Q;
#pragma unroll
    for (int q = 0; q < 4; ++q) f[q] = R(0);
    if (HEAT)
#pragma unroll
        for (int q = 0; q < 4; ++q) d[q] = R(0);
    if (KIN) {
        // the left and right slopes first: the interface derivatives are built from them
#pragma unroll
        for (int q = 4; q < 24; ++q) I.w0[q] = R(0);
        Slopes<R> o;
        slopes<false>(I.L, c, wl + 4, o);
        kinetic_w0(I, c, o, 0);
        slopes<false>(I.Rs, c, wr + 4, o);
        kinetic_w0(I, c, o, 1);
    }
    // equilibrium part, Eq. (15)
    {
        Slopes<R> o;
        slopes<true>(I.Z, c, I.w0 + 4, o, R(KIN ? 1.0 : 0.5));
        const QCoef<R> k = {with_const ? C[0] : R(0), C[2], C[1], R(0.5) * C[3], C[5], R(0.5) * C[4]};
        expand<true>(I.Z, c, o, k, Q);
        add_flux<HEAT>(I.Z, c, Q, (const R *)nullptr, f, d);
    }
    // non-equilibrium part, Eq. (11), left (u > 0) and right (u < 0): one copy
    // of the code for both sides (the flux kernels are long enough for
    // instruction fetch to stall them), the side's state and rows copied in
    const QCoef<R> k = {with_const ? C[6] : R(0), -tau * C[6], C[7] - tau * C[6], R(0.5) * C[8] - tau * C[7],
                        -tau * C[7], R(0)};
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        const State<R> st = side ? I.Rs : I.L;
        R rows[20];
#pragma unroll
        for (int q = 0; q < 20; ++q) rows[q] = side ? wr[4 + q] : wl[4 + q];
        Slopes<R> o;
        slopes<false>(st, c, rows, o);
        expand<false>(st, c, o, k, Q);
        half_moments(st.a, side ? R(-1) : R(1), side ? I.m0[1] : I.m0[0], side ? I.pdf[1] : I.pdf[0], m);
        add_flux<HEAT>(st, c, Q, m, f, d);
    }
}

// Heat flux relative to the velocity (U, V) from the flux moments F = <u psi f>
// and the moments D = <psi f>: <(1/2)(u - U)|c|^2 f>, c = (u - U, v - V, xi),
// expanded in the moments u e, u^2, u v, u, e, v, 1.
template <typename R>
__device__ __forceinline__ R heat_flux(const R *F, const R *D, R U, R V)
{
    const R q2 = U * U + V * V;
    return F[3] - U * F[1] - V * F[2] + (R(0.5) * q2 + U * U) * F[0] - U * D[3] + U * V * D[2] -
           R(0.5) * U * q2 * D[0];
}

// Time-integrated flux through a unit-length face at one Gauss point, all in
// precision R.  wl, wr: [6][4] face-frame rows (value, d/dn, d/dt, d2/dn2,
// d2/dndt, d2/dt2).  Returns false if a state is not physical (f is zero).
// HEAT: Prandtl correction F_E += (1/Pr - 1) q, q the heat flux relative to the
// interface equilibrium velocity (not in the paper; the BGK model has Pr = 1;
// the correction of the BGK-NS scheme, K. Xu, J. Comput. Phys. 171 (2001)).
template <typename R, bool HEAT = false, bool KIN = false>
__device__ __forceinline__ bool gp_flux(const R *wl, const R *wr, R dt, R gamma, R mu, int tau2_exact, R *f,
                                        R prandtl = R(1))
{
    Iface<R> I;
    const Gas<R> c = gas(R(2) / (gamma - R(1)) - R(2));
    if (!interface_state(wl, wr, dt, gamma, mu, c, tau2_exact, I)) {
#pragma unroll
        for (int q = 0; q < 4; ++q) f[q] = R(0);
        return false;
    }
    R d[4];
    body_flux<R, HEAT, KIN>(wl, wr, I, c, true, f, d);
    if (HEAT) f[3] += (R(1) / prandtl - R(1)) * heat_flux(f, d, I.Z.U, I.Z.V);
    return true;
}

}  // namespace kin64
}  // namespace gks
