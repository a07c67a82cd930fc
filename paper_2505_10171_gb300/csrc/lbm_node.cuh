// Per-node device functions of the fluid update (Sec. IV, V E of arXiv
// 2505.10171), shared by the kernels so that all run the same arithmetic:
// collision + recolouring + write, colour record.
#pragma once

#include <type_traits>
#include "lbm_internal.cuh"

namespace lbmg {

// ---------------------------------------------------------------------------
// per-node device functions
// ---------------------------------------------------------------------------

// the node's state before the per-direction updates of the collision
template <class R>
struct CollideState {
    R sF, rr, ux, uy, uz, Fx, Fy, Fz, om, omp, uu, uF, cpe, cpo, bq;
};

template <class R>
__device__ __forceinline__ CollideState<R> collide_state(const FluidPar<R> &P, const R *F, R phi, const GradRec<R> &g)
{
    CollideState<R> c;
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
    const R hs = R(-0.5) * P.sigma * g.k;
    const R pa = R(0.5) * (R(1) + phi), pb = R(0.5) * (R(1) - phi);
    c.Fx = hs * g.g0 + pa * P.ba[0] + pb * P.bb[0];
    c.Fy = hs * g.g1 + pa * P.ba[1] + pb * P.bb[1];
    c.Fz = hs * g.g2 + pa * P.ba[2] + pb * P.bb[2];
    // velocity: rho u = sum c f + F/2
    const R rho = P.rho0 * c.rr;
    const R irho = frcp(rho);
    c.ux = (P.rho0 * jx + R(0.5) * c.Fx) * irho;
    c.uy = (P.rho0 * jy + R(0.5) * c.Fy) * irho;
    c.uz = (P.rho0 * jz + R(0.5) * c.Fz) * irho;
    // relaxation rates: harmonic-mean viscosity, tau = eta/(rho cs2) + 1/2
    const R inv_eta = (R(1) + phi) * P.h_ia + (R(1) - phi) * P.h_ib;
    const R tau = R(3) * frcp(inv_eta * rho) + R(0.5);
    c.om = frcp(tau);
    c.omp = R(8) * (R(2) - c.om) * frcp(R(8) - c.om);
    c.uu = c.ux * c.ux + c.uy * c.uy + c.uz * c.uz;
    c.uF = c.ux * c.Fx + c.uy * c.Fy + c.uz * c.Fz;
    c.cpe = R(1) - R(0.5) * c.om;
    c.cpo = R(1) - R(0.5) * c.omp;
    c.bq = R(0.5) * P.beta * c.rr * (R(1) - phi * phi);
    return c;
}

// colour record (phi, b n) of the node, n = g/sqrt(|g|^2 + eps^2) its
// regularised normal, formed here again from the gradient: seven instructions,
// and the record of the gradient pass is one 16-byte load
template <class R>
__device__ __forceinline__ ColRec<R> colour_record(const FluidPar<R> &P, const CollideState<R> &c, R phi,
                                                   const GradRec<R> &g)
{
    const R b = c.bq * frsqrt(g.g0 * g.g0 + g.g1 * g.g1 + g.g2 * g.g2 + P.eps2);
    return ColRec<R>{phi, b * g.g0, b * g.g1, b * g.g2};
}

// post-collision rest population
template <class R>
__device__ __forceinline__ R collide_rest(const FluidPar<R> &P, const CollideState<R> &c, R F0)
{
    const R feq0 = c.sF + c.rr * (R(-1.5) * c.uu);
    const R fb0 = R(-3) * c.uF * P.ir0;
    return F0 - c.om * (F0 - feq0) + c.cpe * fb0;
}

// opposite pair (i, i+9): the paper's S relaxes every even non-conserved
// moment with omega and every odd one with omega', i.e. the MRT operator is
// exactly the two-relaxation-time operator on the pair's even/odd parts.
// Returns F*_i and F*_ib.
template <class R, int i>
__device__ __forceinline__ void collide_pair(const FluidPar<R> &P, const CollideState<R> &c, R Fi_in, R Fib_in,
                                             R &Fi, R &Fib)
{
    const R cu = cx(i) * c.ux + cy(i) * c.uy + cz(i) * c.uz;
    const R cF = cx(i) * c.Fx + cy(i) * c.Fy + cz(i) * c.Fz;
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

// force, velocity, MRT (two-relaxation-time form) with Guo forcing (Sec. IV),
// recolouring and the write of node n.  F: streamed total offsets; phi: the
// order parameter after streaming (stored by the order-parameter pass); g:
// corrected grad(phi) of the node and its curvature.
// The recolouring of Sec. IV gives G*_i = phi (1 + F*_i) + b (c_i . n)/|c_i|
// with b = beta/2 (rho/rho0)(1 - phi^2): the state is complete with F* and
// the colour record (phi, b n), which are written (C).
template <class S>
__device__ __forceinline__ void collide_store_phi(const FluidPar<typename Store<S>::real> &P,
                                                  const typename Store<S>::real *F, typename Store<S>::real phi,
                                                  const GradRec<typename Store<S>::real> &g, const Pop<S> &out, int n,
                                                  const ColSlotOf<S> &C, typename Store<S>::real *U,
                                                  long long Ustride, unsigned *status)
{
    using R = typename Store<S>::real;
    using FT = typename Pop<S>::FT;
    const int N = out.N;
    FT *const of = out.f + n;  // F_0 of this node; F_i at of + i N
    const CollideState<R> c = collide_state(P, F, phi, g);
    if (status && (!(c.rr > R(0)) || !(phi == phi))) atomicOr(status, ST_UNSTABLE);
    if (U) { U[n] = c.ux; U[Ustride + n] = c.uy; U[2 * Ustride + n] = c.uz; }
    C.set(colour_record(P, c, phi, g));
    Store<FT>::st(of, collide_rest(P, c, F[0]));
    PairLoop<R>::run([&](auto ic) {
        constexpr int i = decltype(ic)::value, ib = i + 9;
        R Fi, Fib;
        collide_pair<R, i>(P, c, F[i], F[ib], Fi, Fib);
        Store<FT>::st(of + i * N, Fi);
        Store<FT>::st(of + ib * N, Fib);
    });
}

}  // namespace lbmg
