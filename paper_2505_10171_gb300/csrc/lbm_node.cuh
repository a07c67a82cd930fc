// Per-node arithmetic of the collision (Sec. IV of arXiv 2505.10171): velocity
// and force, MRT with Guo forcing in its two-relaxation-time form, recolouring.
// The gathered form is one template: V is double, float (16-bit storage), or
// F2, two floats that an instruction handles at once (a node pair of 16-bit
// storage).  FP32 storage relaxes direction by direction (BY_DIRECTION).
#pragma once

#include <type_traits>
#include "lbm_internal.cuh"

namespace lbmg {

// two floats in one register pair (sm_100 and later: add, mul and fma.f32x2 do
// both halves in one issue slot, each rounded as the scalar instruction)
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float a, float b)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack(F2 a, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}

template <class V>
__device__ __forceinline__ V cst(double x) { return (V)x; }
template <>
__device__ __forceinline__ F2 cst<F2>(double x) { return f2((float)x, (float)x); }

template <class V>
__device__ __forceinline__ V add(V a, V b) { return a + b; }
template <class V>
__device__ __forceinline__ V sub(V a, V b) { return a - b; }
template <class V>
__device__ __forceinline__ V mul(V a, V b) { return a * b; }
__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ F2 mad(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
template <>
__device__ __forceinline__ F2 add<F2>(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
template <>
__device__ __forceinline__ F2 sub<F2>(F2 a, F2 b)
{
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
template <>
__device__ __forceinline__ F2 mul<F2>(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

// reciprocals of three values: FP64 by one division, whose instruction sequence
// weighs more than the five products
__device__ __forceinline__ void rcp3(float a, float b, float c, float &ra, float &rb, float &rc)
{
    ra = frcp(a); rb = frcp(b); rc = frcp(c);
}
__device__ __forceinline__ void rcp3(double a, double b, double c, double &ra, double &rb, double &rc)
{
    const double ab = a * b, r = 1.0 / (ab * c), rab = r * c;
    ra = rab * b;
    rb = rab * a;
    rc = r * ab;
}
__device__ __forceinline__ void rcp3(F2 a, F2 b, F2 c, F2 &ra, F2 &rb, F2 &rc)
{
    float x, y;
    unpack(a, x, y); ra = f2(frcp(x), frcp(y));
    unpack(b, x, y); rb = f2(frcp(x), frcp(y));
    unpack(c, x, y); rc = f2(frcp(x), frcp(y));
}
__device__ __forceinline__ F2 frsqrt(F2 a)
{
    float x, y;
    unpack(a, x, y);
    return f2(frsqrt(x), frsqrt(y));
}

// What a node's collision does to its directions.  With the sum s = F_i + F_ib
// and difference d = F_i - F_ib of an opposite pair (i, i + 9), the paper's S
// relaxes every even non-conserved moment with omega and every odd one with
// omega', i.e. the MRT operator is exactly the two-relaxation-time operator on
// the pair's even and odd parts:
//   E = a s + K0 + (c.u)(A1 (c.u) + A2 (c.F)),   a = (1 - omega)/2,
//   O = b d + B1 (c.u) + B2 (c.F),               b = (1 - omega')/2,
//   F*_i = E + O,  F*_ib = E - O,  F*_0 = 2 a F_0 + K0,
// the equilibrium's and Guo's terms gathered by their power of c.u:
//   K0 = omega (sF - 3/2 rr u.u) - 3 (1 - omega/2) u.F/rho0,  A1 = 9/2 omega rr,
//   A2 = 9 (1 - omega/2)/rho0,  B1 = 3 omega' rr,  B2 = 3 (1 - omega'/2)/rho0.
// With x = rho/eta the harmonic-mean viscosity's tau = 3/x + 1/2 gives
// omega = 2 x/(6 + x) and omega' = 8 (2 - omega)/(8 - omega) = 16/(8 + x).
template <class V>
struct Collision {
    V rr, bq;          // rho/rho0; b = beta/2 rr (1 - phi^2)
    V u[3], f[3];      // velocity, force density
    V a, b, K0, A1, A2, B1, B2;
};

// fluid parameters as the collision takes them, from those of an instance
template <class V>
struct CollidePar {
    V csf, m0[3], m1[3], rho0, h0, h1, ir0, bh;
    template <class R>
    __device__ __forceinline__ explicit CollidePar(const FluidPar<R> &P)
    {
        csf = bc(R(-0.5) * P.sigma);
        for (int k = 0; k < 3; k++) {
            m0[k] = bc(R(0.5) * (P.ba[k] + P.bb[k]));  // phase-weighted body force m0 + phi m1
            m1[k] = bc(R(0.5) * (P.ba[k] - P.bb[k]));
        }
        rho0 = bc(P.rho0);
        h0 = bc(P.h_ia + P.h_ib);                      // 1/eta = h0 + phi h1
        h1 = bc(P.h_ia - P.h_ib);
        ir0 = bc(P.ir0);
        bh = bc(R(0.5) * P.beta);
    }
    template <class R>
    static __device__ __forceinline__ V bc(R x)
    {
        if constexpr (std::is_same_v<V, F2>) return f2(x, x);
        else return x;
    }
};

// F: streamed total offsets; on return F[i] and F[i + 9] of every pair hold its
// sum and difference.  phi: the order parameter after streaming; g: corrected
// grad(phi); kap: curvature.
template <class V>
__device__ __forceinline__ Collision<V> collide_setup(const CollidePar<V> &P, V (&F)[Q], V phi, const V (&g)[3], V kap)
{
    Collision<V> c;
#pragma unroll
    for (int i = 1; i <= 9; i++) {
        const V s = add(F[i], F[i + 9]), d = sub(F[i], F[i + 9]);
        F[i] = s;
        F[i + 9] = d;
    }
    const V w1 = cst<V>(1.0 / 18.0), w2 = cst<V>(1.0 / 36.0), half = cst<V>(0.5), one = cst<V>(1.0);
    // moments: pairs 1..3 are the axes, 4..9 the diagonals (1,1,0), (1,-1,0),
    // (1,0,1), (1,0,-1), (0,1,1), (0,1,-1)
    const V sa = add(add(F[1], F[2]), F[3]);
    const V sd = add(add(add(F[4], F[5]), add(F[6], F[7])), add(F[8], F[9]));
    const V sF = mad(cst<V>(1.0 / 3.0), F[0], mad(w1, sa, mul(w2, sd)));
    const V *d = F + 9;
    const V j[3] = {mad(w1, d[1], mul(w2, add(add(d[4], d[5]), add(d[6], d[7])))),
                    mad(w1, d[2], mul(w2, add(sub(d[4], d[5]), add(d[8], d[9])))),
                    mad(w1, d[3], mul(w2, add(sub(d[6], d[7]), sub(d[8], d[9]))))};
    c.rr = add(one, sF);
    // force density: CSF -1/2 sigma kappa grad(phi) plus the body forces
    const V hs = mul(P.csf, kap);
#pragma unroll
    for (int k = 0; k < 3; k++) c.f[k] = mad(hs, g[k], mad(phi, P.m1[k], P.m0[k]));
    const V rho = mul(P.rho0, c.rr);
    const V x = mul(mad(phi, P.h1, P.h0), rho);
    V irho, r6, r8;
    rcp3(rho, add(cst<V>(6.0), x), add(cst<V>(8.0), x), irho, r6, r8);
    // velocity: rho u = sum c f + F/2
#pragma unroll
    for (int k = 0; k < 3; k++) c.u[k] = mul(mad(half, c.f[k], mul(P.rho0, j[k])), irho);
    const V om = mul(add(x, x), r6), op = mul(cst<V>(16.0), r8);
    const V uu = mad(c.u[0], c.u[0], mad(c.u[1], c.u[1], mul(c.u[2], c.u[2])));
    const V uf = mad(c.u[0], c.f[0], mad(c.u[1], c.f[1], mul(c.u[2], c.f[2])));
    const V mh = cst<V>(-0.5);
    const V ge = mul(mad(mh, om, one), P.ir0), go = mul(mad(mh, op, one), P.ir0);
    const V omr = mul(om, c.rr);
    // omega (sF - 3/2 rr u.u) - 3 ge u.F
    c.K0 = mad(om, sF, mul(cst<V>(-1.5), mad(omr, uu, mul(cst<V>(2.0), mul(ge, uf)))));
    c.A1 = mul(cst<V>(4.5), omr);
    c.A2 = mul(cst<V>(9.0), ge);
    c.B1 = mul(cst<V>(3.0), mul(op, c.rr));
    c.B2 = mul(cst<V>(3.0), go);
    c.a = mad(mh, om, half);
    c.b = mad(mh, op, half);
    c.bq = mul(mul(P.bh, c.rr), mad(mul(cst<V>(-1.0), phi), phi, one));
    return c;
}

// post-collision rest population
template <class V>
__device__ __forceinline__ V collide_rest(const Collision<V> &c, V F0)
{
    return mad(add(c.a, c.a), F0, c.K0);
}

// c_i . v
template <int i, class V>
__device__ __forceinline__ V along(const V (&v)[3])
{
    if constexpr (i <= 3) return v[i - 1];
    else if constexpr (cx(i)) return cy(i) ? (cy(i) > 0 ? add(v[0], v[1]) : sub(v[0], v[1]))
                                           : (cz(i) > 0 ? add(v[0], v[2]) : sub(v[0], v[2]));
    else return cz(i) > 0 ? add(v[1], v[2]) : sub(v[1], v[2]);
}

// opposite pair (i, i + 9), i in 1..9, of sum s and difference d
template <int i, class V>
__device__ __forceinline__ void collide_pair(const Collision<V> &c, V s, V d, V &Fi, V &Fib)
{
    const V cu = along<i>(c.u), cf = along<i>(c.f);
    const V E = mad(c.a, s, mad(cu, mad(c.A1, cu, mul(c.A2, cf)), c.K0));
    const V O = mad(c.b, d, mad(c.B1, cu, mul(c.B2, cf)));
    Fi = add(E, O);
    Fib = sub(E, O);
}

template <class R, int i = 1>
struct PairLoop {
    template <class Fn>
    __device__ __forceinline__ static void run(Fn &&f)
    {
        f(std::integral_constant<int, i>());
        PairLoop<R, i + 1>::run(f);
    }
};
template <class R>
struct PairLoop<R, 10> {
    template <class Fn>
    __device__ __forceinline__ static void run(Fn &&) {}
};

// colour record (phi, b n) of the node, n = g/sqrt(|g|^2 + eps^2) its
// regularised normal, formed here again from the gradient: seven instructions,
// and the record of the gradient pass is one 16-byte load
template <class R>
__device__ __forceinline__ ColRec<R> colour_record(R bq, R eps2, R phi, R g0, R g1, R g2)
{
    const R b = bq * frsqrt(g0 * g0 + g1 * g1 + g2 * g2 + eps2);
    return ColRec<R>{phi, b * g0, b * g1, b * g2};
}

// The form of FP32 storage: moments summed and pairs relaxed direction by
// direction.  The collision is bound by memory there (119 us per 256x128x128
// launch either way), so the gathered form has nothing to give, and it rounds
// otherwise (see BY_DIRECTION).
template <class R>
struct DirCollision {
    R sF, rr, u[3], f[3], om, omp, uu, uF, cpe, cpo, bq;
};

// g, kap: corrected grad(phi) and curvature
template <class R>
__device__ __forceinline__ DirCollision<R> dir_setup(const FluidPar<R> &P, const R (&F)[Q], R phi, const R (&g)[3], R kap)
{
    DirCollision<R> c;
    R sF = 0, jx = 0, jy = 0, jz = 0;
#pragma unroll
    for (int i = 0; i < Q; i++) {
        const R w = wgt<R>(i);
        sF += w * F[i];
        if (cx(i)) jx += w * cx(i) * F[i];
        if (cy(i)) jy += w * cy(i) * F[i];
        if (cz(i)) jz += w * cz(i) * F[i];
    }
    c.sF = sF;
    c.rr = R(1) + sF;  // rho / rho0
    // force density: CSF -1/2 sigma kappa grad(phi) plus phase-weighted body forces
    const R hs = R(-0.5) * P.sigma * kap;
    const R pa = R(0.5) * (R(1) + phi), pb = R(0.5) * (R(1) - phi);
    // (which product is rounded by itself is part of the results: it differs in x)
    c.f[0] = fma_rn(pb, P.bb[0], fma_rn(pa, P.ba[0], mul_rn(hs, g[0])));
    c.f[1] = fma_rn(pb, P.bb[1], fma_rn(hs, g[1], mul_rn(pa, P.ba[1])));
    c.f[2] = fma_rn(pb, P.bb[2], fma_rn(hs, g[2], mul_rn(pa, P.ba[2])));
    // velocity: rho u = sum c f + F/2
    const R rho = P.rho0 * c.rr;
    const R irho = frcp(rho);
    c.u[0] = (P.rho0 * jx + R(0.5) * c.f[0]) * irho;
    c.u[1] = (P.rho0 * jy + R(0.5) * c.f[1]) * irho;
    c.u[2] = (P.rho0 * jz + R(0.5) * c.f[2]) * irho;
    // relaxation rates: harmonic-mean viscosity, tau = eta/(rho cs2) + 1/2
    const R inv_eta = (R(1) + phi) * P.h_ia + (R(1) - phi) * P.h_ib;
    const R tau = R(3) * frcp(inv_eta * rho) + R(0.5);
    c.om = frcp(tau);
    c.omp = R(8) * (R(2) - c.om) * frcp(R(8) - c.om);
    c.uu = c.u[0] * c.u[0] + c.u[1] * c.u[1] + c.u[2] * c.u[2];
    c.uF = c.u[0] * c.f[0] + c.u[1] * c.f[1] + c.u[2] * c.f[2];
    c.cpe = R(1) - R(0.5) * c.om;
    c.cpo = R(1) - R(0.5) * c.omp;
    c.bq = R(0.5) * P.beta * c.rr * (R(1) - phi * phi);
    return c;
}

template <class R>
__device__ __forceinline__ R dir_rest(const FluidPar<R> &P, const DirCollision<R> &c, R F0)
{
    const R feq0 = c.sF + c.rr * (R(-1.5) * c.uu);
    const R fb0 = R(-3) * c.uF * P.ir0;
    return F0 - c.om * (F0 - feq0) + c.cpe * fb0;
}

// opposite pair (i, i + 9), relaxed in its even and odd parts
template <int i, class R>
__device__ __forceinline__ void dir_pair(const FluidPar<R> &P, const DirCollision<R> &c, R Fi_in, R Fib_in, R &Fi, R &Fib)
{
    const R cu = cx(i) * c.u[0] + cy(i) * c.u[1] + cz(i) * c.u[2];
    const R cF = cx(i) * c.f[0] + cy(i) * c.f[1] + cz(i) * c.f[2];
    const R eqp = c.sF + c.rr * (R(4.5) * cu * cu - R(1.5) * c.uu);
    const R eqm = c.rr * R(3) * cu;
    const R fbp = (R(9) * cu * cF - R(3) * c.uF) * P.ir0;
    const R fbm = R(3) * cF * P.ir0;
    const R fp = R(0.5) * (Fi_in + Fib_in);
    const R fm = R(0.5) * (Fi_in - Fib_in);
    const R dp = -c.om * (fp - eqp) + c.cpe * fbp;
    const R dm = -c.omp * (fm - eqm) + c.cpo * fbm;
    Fi = Fi_in + dp + dm;
    Fib = Fib_in + dp - dm;
}

// force, velocity, MRT with Guo forcing, recolouring and the write of node n.
// The recolouring of Sec. IV gives G*_i = phi (1 + F*_i) + b (c_i . n)/|c_i|
// with b = beta/2 (rho/rho0)(1 - phi^2): the state is complete with F* and
// the colour record (phi, b n), which are written (C).  F is consumed.
template <class S>
__device__ __forceinline__ void collide_store_phi(const FluidPar<typename Store<S>::real> &P,
                                                  typename Store<S>::real (&F)[Q], typename Store<S>::real phi,
                                                  const GradRec<typename Store<S>::real> &gr, const Pop<S> &out, int n,
                                                  const ColSlotOf<S> &C, typename Store<S>::real *U,
                                                  long long Ustride, unsigned *status)
{
    using R = typename Store<S>::real;
    using FT = typename Pop<S>::FT;
    const int N = out.N;
    FT *const of = out.f + n;  // F_0 of this node; F_i at of + i N
    const R g[3] = {gr.g0, gr.g1, gr.g2};
    auto store_moments = [&](R rr, const R *u) {
        if (status && (!(rr > R(0)) || !(phi == phi))) atomicOr(status, ST_UNSTABLE);
        if (U) { U[n] = u[0]; U[Ustride + n] = u[1]; U[2 * Ustride + n] = u[2]; }
    };
    if constexpr (BY_DIRECTION<S>) {
        // the gradient as the product of its norm and normal, as it was formed
        R nn[3];
        const R m = dir_normal(g, P.eps2, nn);
        const R gm[3] = {nn[0] * m, nn[1] * m, nn[2] * m};
        const DirCollision<R> c = dir_setup(P, F, phi, gm, gr.k);
        store_moments(c.rr, c.u);
        C.set(ColRec<R>{phi, c.bq * nn[0], c.bq * nn[1], c.bq * nn[2]});
        Store<FT>::st(of, dir_rest(P, c, F[0]));
        PairLoop<R>::run([&](auto ic) {
            constexpr int i = decltype(ic)::value, ib = i + 9;
            R Fi, Fib;
            dir_pair<i>(P, c, F[i], F[ib], Fi, Fib);
            Store<FT>::st(of + i * N, Fi);
            Store<FT>::st(of + ib * N, Fib);
        });
    } else {
        const Collision<R> c = collide_setup(CollidePar<R>(P), F, phi, g, gr.k);
        store_moments(c.rr, c.u);
        C.set(colour_record(c.bq, P.eps2, phi, g[0], g[1], g[2]));
        Store<FT>::st(of, collide_rest(c, F[0]));
        PairLoop<R>::run([&](auto ic) {
            constexpr int i = decltype(ic)::value, ib = i + 9;
            R Fi, Fib;
            collide_pair<i>(c, F[i], F[ib], Fi, Fib);
            Store<FT>::st(of + i * N, Fi);
            Store<FT>::st(of + ib * N, Fib);
        });
    }
}

}  // namespace lbmg
