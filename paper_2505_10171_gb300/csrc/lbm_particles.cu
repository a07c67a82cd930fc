// Particle kernels of one coupled time step (Sec. III and V of arXiv 2505.10171):
//   k_contacts     velocity-Verlet prediction and contact forces (normal
//                  spring-dashpot, Luding sliding and rolling friction, Sec. III):
//                  they need the previous step's forces only, so they run early
//   k_mem          momentum-exchange force and torque per particle (Sec. V B)
//   k_capillary    capillary force and torque from the Lagrangian surface points
//                  (Sec. V F)
//   k_dem          fixed-order sums of the per-block partials of both, the
//                  velocity-Verlet correction (Sec. III) and the step's record:
//                  one warp per particle
//   k_geom_owner, k_geom_surface, k_refill
//                  solid map update with the next step's boundary lists, and
//                  refilling of uncovered nodes (Sec. V C)
// Per-link and per-point arithmetic runs in the storage precision's arithmetic
// type (double for FP64 storage, float otherwise); positions, velocities and
// every sum over links, points or contacts are FP64 with a fixed order (warp
// exchange, then blocks), so results are reproducible run to run.  An FP64
// warp instruction holds its SM's FP64 pipe for about 16 cycles, so these
// kernels count them: sums of K values over a warp exchange halves (K + 4
// additions, not 5 K), and the work is spread over SMs in small CTAs.
#include "lbm_internal.cuh"

namespace lbmg {

// Sums of K values (a power of two, 2 to 16) over the 32 lanes by exchanging
// halves: at each of the first log2 K steps a lane keeps half of its values and
// adds its partner's copies of them, so that K - 1 additions (and one per step
// left) do the work of 5 K.  The sum of value a is left in v[0] of lane
// a 32/K (and of the lanes above it up to the next one's).
template <int K, class T>
__device__ __forceinline__ void warp_sums(T *v)
{
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int h = K / 2; h >= 1; h >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int a = 0; a < h; a++) {
            const T keep = up ? v[a + h] : v[a], give = up ? v[a] : v[a + h];
            v[a] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
        o >>= 1;
    }
    for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
}

// sums of K values over a CTA of NT threads, warps in order; thread a < n
// writes sum a to out
template <int K, int NT, class T>
__device__ __forceinline__ void block_sums(T *v, int n, double *out)
{
    __shared__ T sm[NT / 32][K];
    warp_sums<K>(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane % (32 / K) == 0) sm[wid][lane / (32 / K)] = v[0];
    __syncthreads();
    if ((int)threadIdx.x < n) {
        T s = sm[0][threadIdx.x];
#pragma unroll
        for (int w = 1; w < NT / 32; w++) s += sm[w][threadIdx.x];
        out[threadIdx.x] = (double)s;
    }
}

// particle centre in the arithmetic type R (single-precision copy for float)
__device__ __forceinline__ void centre(const PartDev &P, double *c) { c[0] = P.x[0]; c[1] = P.x[1]; c[2] = P.x[2]; }
__device__ __forceinline__ void centre(const PartDev &P, float *c) { c[0] = P.xf[0]; c[1] = P.xf[1]; c[2] = P.xf[2]; }

// Sec. V B momentum exchange (Wen 2014, Galilean invariant): per link from a
// fluid node x into particle p, force on p = (c_out - u_w) f_out - (c_in - u_w) f_in
// with f_out = f*_ibar(x) leaving towards the solid and f_in = f_i(x) bounced
// back; torque lever from the centre to the link midpoint.
//
// With f_out = w rho0 (1 + F), f_in = w rho0 (1 + F + 6 rr c.u_w) the link
// term is -2 w rho0 c (the rest part, order 0.1, cancelling over the closed
// surface) plus w rho0 (-c (2F + 6 rr c.u_w) + u_w 6 rr c.u_w) (order 1e-4).
// Rounding the sum in single precision would swamp the offsets, and FP64
// arithmetic per link is slow on this GPU, so the rest part is kept exactly in
// integers: with k = 36 w in {1, 2} and the lever d - delta, d the half-integer
// offset of the link midpoint from the integer point xr = floor(x_p), delta =
// x_p - xr, its force is -(rho0/18) K and its torque -(rho0/18) (M - delta x K)
// with K = sum k c and M = sum k d x c. The block partials hold the small
// part's force and torque, K and 2M; the DEM kernel assembles them in FP64.
//
// A node's flags and populations are loaded together, whatever its links.
template <class S>
__global__ void __launch_bounds__(MEM_THREADS) k_mem(Lattice L, int cur, FastDiv fd)
{
    using R = typename Store<S>::real;
    const int p = blockIdx.y;
    const PartDev &P = L.parts[p];
    const InstDev &I = L.inst[P.inst];
    Region reg;
    reg.init(P.xf, (int)fd.d, I.nx, I.ny, I.nz);
    R acc[6] = {0, 0, 0, 0, 0, 0};
    int kin[6] = {0, 0, 0, 0, 0, 0};  // K, then 2M
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    bool links = false;
    int x = 0, y = 0, z = 0, n = 0;
    const uint8_t *fli = L.flags + I.node_off;
    if (t < reg.count()) {
        reg.coord(t, fd, I.nx, I.ny, I.nz, &x, &y, &z);
        n = (z * I.ny + y) * I.nx + x;
        const uint8_t fl = fli[n];
        links = (fl & OWNER_MASK) == OWN_FLUID && (fl & BOUND_BIT);
    }
    if (links) {
        const Pop<S> in(L.pop[cur], I);
        Nbr nb;
        nb.init(x, y, z, I.nx, I.ny, I.nz);
        const int mine = 2 + P.local;
        int own[Q];
        R F[Q];
#pragma unroll
        for (int i = 0; i < Q; i++) {
            own[i] = fli[nb.at(-cx(i), -cy(i), -cz(i))];
            F[i] = in.F(i, n);
        }
        R c[3], v[3], w[3];
        centre(P, c);
        for (int a = 0; a < 3; a++) { v[a] = (R)P.v[a]; w[a] = (R)P.w[a]; }
        // twice the node's offset from xr, minimum image (|.| < n)
        const int per[3] = {I.nx, I.ny, I.nz};
        const int pos[3] = {x, y, z};
        int D0[3];
        for (int a = 0; a < 3; a++) {
            int d = 2 * (pos[a] - (int)floor(P.x[a]));
            d += d >= per[a] ? -2 * per[a] : (d < -per[a] ? 2 * per[a] : 0);
            D0[a] = d;
        }
        const R r0 = sizeof(R) == 8 ? (R)I.rho0 : (R)I.f_rho0;
        R sF = 0;  // the offsets' sum first: added to 1 one by one, each would be rounded at 1
#pragma unroll
        for (int i = 0; i < Q; i++) sF += wgt<R>(i) * F[i];
        const R r6 = R(6) * (R(1) + sF);
        // lever and wall velocity of a link, and c.u_w
        auto link = [&](int i, const R *lev, const R *uw, R cu) {
            const R wt = wgt<R>(i) * r0;
            const R e = r6 * cu;
            const R q = R(2) * F[opp(i)] + e;
            const R dp[3] = {wt * (uw[0] * e - cx(i) * q), wt * (uw[1] * e - cy(i) * q), wt * (uw[2] * e - cz(i) * q)};
            acc[0] += dp[0];
            acc[1] += dp[1];
            acc[2] += dp[2];
            acc[3] += lev[1] * dp[2] - lev[2] * dp[1];
            acc[4] += lev[2] * dp[0] - lev[0] * dp[2];
            acc[5] += lev[0] * dp[1] - lev[1] * dp[0];
            // rest part: k c and k (2d) x c, 2d = D0 - c
            const int k = csq(i) == 1 ? 2 : 1;
            const int E[3] = {D0[0] - cx(i), D0[1] - cy(i), D0[2] - cz(i)};
            kin[0] += k * cx(i);
            kin[1] += k * cy(i);
            kin[2] += k * cz(i);
            kin[3] += k * (E[1] * cz(i) - E[2] * cy(i));
            kin[4] += k * (E[2] * cx(i) - E[0] * cz(i));
            kin[5] += k * (E[0] * cy(i) - E[1] * cx(i));
        };
        R d[3];
        if (sizeof(R) == 8 && node_lever<R>(I, x, y, z, c, d)) {
            // the node's velocity u and lever d for all links: u_w = u - (w x c_i)/2,
            // c_i.u_w = c_i.u (FP64, R = 4: 27 -> 15 us)
            const R u[3] = {v[0] + (w[1] * d[2] - w[2] * d[1]), v[1] + (w[2] * d[0] - w[0] * d[2]),
                            v[2] + (w[0] * d[1] - w[1] * d[0])};
            const R hw[3] = {R(0.5) * w[0], R(0.5) * w[1], R(0.5) * w[2]};
#pragma unroll
            for (int i = 1; i < Q; i++) {
                if ((own[i] & OWNER_MASK) != mine) continue;
                R lev[3] = {d[0], d[1], d[2]}, uw[3] = {u[0], u[1], u[2]}, cu = 0;
                if (cx(i)) {
                    lev[0] -= R(0.5) * cx(i);
                    uw[1] -= cx(i) * hw[2];
                    uw[2] += cx(i) * hw[1];
                    cu += cx(i) * u[0];
                }
                if (cy(i)) {
                    lev[1] -= R(0.5) * cy(i);
                    uw[0] += cy(i) * hw[2];
                    uw[2] -= cy(i) * hw[0];
                    cu += cy(i) * u[1];
                }
                if (cz(i)) {
                    lev[2] -= R(0.5) * cz(i);
                    uw[0] -= cz(i) * hw[1];
                    uw[1] += cz(i) * hw[0];
                    cu += cz(i) * u[2];
                }
                link(i, lev, uw, cu);
            }
        } else {
#pragma unroll
            for (int i = 1; i < Q; i++) {
                if ((own[i] & OWNER_MASK) != mine) continue;
                const R lev[3] = {min_image_r<R>((x - R(0.5) * cx(i)) - c[0], I.nx),
                                  min_image_r<R>((y - R(0.5) * cy(i)) - c[1], I.ny),
                                  min_image_r<R>((z - R(0.5) * cz(i)) - c[2], I.nz)};
                const R uw[3] = {v[0] + (w[1] * lev[2] - w[2] * lev[1]), v[1] + (w[2] * lev[0] - w[0] * lev[2]),
                                 v[2] + (w[0] * lev[1] - w[1] * lev[0])};
                link(i, lev, uw, cx(i) * uw[0] + cy(i) * uw[1] + cz(i) * uw[2]);
            }
        }
    }
    double *out = L.mem_part + ((long long)p * L.mem_blocks + blockIdx.x) * MEM_PART;
    if (!__syncthreads_or(links)) {  // most blocks of the cube: nothing to add
        if (threadIdx.x < MEM_PART) out[threadIdx.x] = 0.0;
        return;
    }
    double accd[8];
    for (int a = 0; a < 8; a++) accd[a] = a < 6 ? (double)acc[a] : 0.0;
    block_sums<8, MEM_THREADS>(accd, 6, out);
    int kin8[8];
    for (int a = 0; a < 8; a++) kin8[a] = a < 6 ? kin[a] : 0;
    block_sums<8, MEM_THREADS>(kin8, 6, out + 6);
}

// Sec. V F: dF = C sigma (1 - phi^2) dA (n x n_s) x n at the points
// alpha_j = (j + 1/2) 2 deg, varphi_k = k 2 deg on r = R_p, n the regularised
// normal of the trilinearly interpolated grad(phi) (fluid corners only);
// torque R_p n_s x dF.  With BUOY also the phase-a share of the surface for
// the buoyancy (reading c28): s = (1 + phi)/2 clipped to [0, 1] and dA, summed
// over the points with a fluid corner.
//
// The eight corners' flags, phi and gradients are loaded together, solid or not.
__device__ __forceinline__ void surface_point(const Lattice &L, int pt, float *t)
{
    const float4 v = reinterpret_cast<const float4 *>(L.cap_pts_f)[pt];
    t[0] = v.x; t[1] = v.y; t[2] = v.z; t[3] = v.w;
}
__device__ __forceinline__ void surface_point(const Lattice &L, int pt, double *t)
{
    for (int a = 0; a < 4; a++) t[a] = L.cap_pts[4 * pt + a];
}

template <class S, bool BUOY>
__global__ void __launch_bounds__(CAP_THREADS) k_capillary(Lattice L)
{
    using R = typename Store<S>::real;
    const int p = blockIdx.y;
    const PartDev &P = L.parts[p];
    const InstDev &I = L.inst[P.inst];
    R acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const int pt = blockIdx.x * blockDim.x + threadIdx.x;
    if (pt < CAP_POINTS) {
        R tp[4];
        surface_point(L, pt, tp);
        const R ns[3] = {tp[0], tp[1], tp[2]};
        const R sa = tp[3];
        const R da = R(2.0 * M_PI / 180.0);
        R c[3];
        centre(P, c);
        const R Rp = sizeof(R) == 8 ? (R)P.R : (R)P.Rf;
        const R xi[3] = {c[0] + Rp * ns[0], c[1] + Rp * ns[1], c[2] + Rp * ns[2]};
        const R dA = Rp * Rp * sa * da * da;
        int lo[3], hi[3];
        R fr[3];
        const int n3[3] = {I.nx, I.ny, I.nz};
        for (int a = 0; a < 3; a++) {
            const R fl = floor(xi[a]);
            fr[a] = xi[a] - fl;
            const int b = (int)fl;
            lo[a] = b < 0 ? b + n3[a] : (b >= n3[a] ? b - n3[a] : b);
            hi[a] = b + 1 < 0 ? b + 1 + n3[a] : (b + 1 >= n3[a] ? b + 1 - n3[a] : b + 1);
        }
        const uint8_t *fli = L.flags + I.node_off;
        const R *ph = (const R *)L.phi + I.node_off;
        const GradRec<R> *Gr = (const GradRec<R> *)L.grad + I.node_off;
        uint8_t fl[8];
        R pc[8];
        GradRec<R> gc[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const int X = k & 1 ? hi[0] : lo[0], Y = k & 2 ? hi[1] : lo[1], Z = k & 4 ? hi[2] : lo[2];
            const int m = (Z * I.ny + Y) * I.nx + X;
            fl[k] = fli[m];
            pc[k] = ph[m];
            gc[k] = Gr[m];
        }
        R ws = 0, phs = 0, gs[3] = {0, 0, 0};
#pragma unroll
        for (int k = 0; k < 8; k++) {
            if ((fl[k] & OWNER_MASK) != OWN_FLUID) continue;
            const R wgt_ = (k & 1 ? fr[0] : R(1) - fr[0]) * (k & 2 ? fr[1] : R(1) - fr[1]) * (k & 4 ? fr[2] : R(1) - fr[2]);
            R g[3] = {gc[k].g0, gc[k].g1, gc[k].g2};
            if constexpr (BY_DIRECTION<S>) {  // as the collision takes it
                R nn[3];
                const R m = dir_normal(g, I.f_eps2, nn);
                for (int a = 0; a < 3; a++) g[a] = mul_rn(nn[a], m);
            }
            ws += wgt_;
            phs += wgt_ * pc[k];
            for (int a = 0; a < 3; a++) gs[a] += wgt_ * g[a];
        }
        if (ws > R(0)) {
            const R phv = phs / ws;
            if (BUOY) {
                acc[6] = fmin(fmax(R(0.5) * (R(1) + phv), R(0)), R(1)) * dA;
                acc[7] = dA;
            }
            const R g0 = gs[0] / ws, g1 = gs[1] / ws, g2 = gs[2] / ws;
            if (fabs(phv) < R(1)) {
                const R eps2 = sizeof(R) == 8 ? (R)(I.grad_eps * I.grad_eps) : (R)I.f_eps2;
                const R gr = sqrt(g0 * g0 + g1 * g1 + g2 * g2 + eps2);
                const R nn[3] = {g0 / gr, g1 / gr, g2 / gr};
                const R c0 = nn[1] * ns[2] - nn[2] * ns[1], c1 = nn[2] * ns[0] - nn[0] * ns[2],
                        c2 = nn[0] * ns[1] - nn[1] * ns[0];
                const R mv[3] = {c1 * nn[2] - c2 * nn[1], c2 * nn[0] - c0 * nn[2], c0 * nn[1] - c1 * nn[0]};
                const R coef = (sizeof(R) == 8 ? (R)(I.cap_norm * I.sigma) : (R)I.f_cap) * (R(1) - phv * phv) * dA;
                R dF[3];
                for (int a = 0; a < 3; a++) dF[a] = coef * mv[a];
                const R r[3] = {Rp * ns[0], Rp * ns[1], Rp * ns[2]};
                acc[0] = dF[0];
                acc[1] = dF[1];
                acc[2] = dF[2];
                acc[3] = r[1] * dF[2] - r[2] * dF[1];
                acc[4] = r[2] * dF[0] - r[0] * dF[2];
                acc[5] = r[0] * dF[1] - r[1] * dF[0];
            }
        }
    }
    double accd[8];
    for (int a = 0; a < 8; a++) accd[a] = a < (BUOY ? 8 : 6) ? (double)acc[a] : 0.0;
    block_sums<8, CAP_THREADS>(accd, BUOY ? 8 : 6, L.cap_part + ((long long)p * CAP_BLOCKS + blockIdx.x) * CAP_PART);
}


// ---------------------------------------------------------------------------
// DEM (Sec. III).  Positions, velocities, spring histories and the Verlet
// sums are FP64; the contact arithmetic runs in T: double in the FP64 mode,
// float otherwise (FP64 issues at a small fraction of the FP32 rate here and
// the DEM is one serial chain of dependent operations).
// ---------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ T dot3(const T *a, const T *b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }
template <class T>
__device__ __forceinline__ void cross3(const T *a, const T *b, T *r)
{
    T t0 = a[1] * b[2] - a[2] * b[1], t1 = a[2] * b[0] - a[0] * b[2], t2 = a[0] * b[1] - a[1] * b[0];
    r[0] = t0; r[1] = t1; r[2] = t2;
}

// Luding spring: project on the tangent plane, trial force, Coulomb cap,
// spring update (static: xi += v dt; sliding: xi = -(F + gamma v)/k).
template <class T>
__device__ void dem_spring(T *xi, const T *n, const T *v, T k, T gam, T FC, T *F)
{
    T xn = dot3(xi, n);
    for (int a = 0; a < 3; a++) xi[a] -= xn * n[a];
    T F0[3];
    for (int a = 0; a < 3; a++) F0[a] = -k * xi[a] - gam * v[a];
    T m = sqrt(dot3(F0, F0));
    if (m <= FC) {
        for (int a = 0; a < 3; a++) { F[a] = F0[a]; xi[a] += v[a]; }
    } else {
        for (int a = 0; a < 3; a++) F[a] = FC * F0[a] / m;
        for (int a = 0; a < 3; a++) xi[a] = k > T(0) ? -(F[a] + gam * v[a]) / k : T(0);
    }
}

// contact of particle i with partner j (j < 0: substrate); n from partner to
// i, delta > 0 the overlap.  Contact point X_i - (R_c,i - delta/2) n;
// F_n = [k_n delta - g_n v_rel.n] n; rolling velocity -a'(w_i - w_j) x n with
// torque -a' n x F_r on i (+a' n x F_r on j).  rec receives the force and
// torque on i, then on j.
template <class T>
__device__ void dem_contact(const InstDev &I, const PartDev *P, int i, int j, const T *vp, const T *wp, const T *n,
                            T delta, T *xi, T *xir, T *rec)
{
    const T Rci = (T)P[i].Rc;
    T bi[3], bj[3] = {0, 0, 0}, t[3], vi[3], vj[3];
    for (int a = 0; a < 3; a++) bi[a] = -(Rci - T(0.5) * delta) * n[a];
    cross3(wp + 3 * i, bi, t);
    for (int a = 0; a < 3; a++) vi[a] = vp[3 * i + a] + t[a];
    T ap;
    if (j >= 0) {
        const T Rcj = (T)P[j].Rc;
        for (int a = 0; a < 3; a++) bj[a] = (Rcj - T(0.5) * delta) * n[a];
        cross3(wp + 3 * j, bj, t);
        for (int a = 0; a < 3; a++) vj[a] = vp[3 * j + a] + t[a];
        ap = Rci * Rcj / (Rci + Rcj);
    } else {
        for (int a = 0; a < 3; a++) vj[a] = (T)I.wall_u[a];
        ap = Rci;
    }
    T vr[3];
    for (int a = 0; a < 3; a++) vr[a] = vi[a] - vj[a];
    const T vn = dot3(vr, n);
    const T Fnm = (T)I.kn * delta - (T)I.gn * vn;
    T vt[3];
    for (int a = 0; a < 3; a++) vt[a] = vr[a] - vn * n[a];
    T Ft[3];
    dem_spring(xi, n, vt, (T)I.kt, (T)I.gt, (T)I.mu_s * fabs(Fnm), Ft);
    T wrel[3], vrl[3];
    for (int a = 0; a < 3; a++) wrel[a] = wp[3 * i + a] - (j >= 0 ? wp[3 * j + a] : T(0));
    cross3(wrel, n, vrl);
    for (int a = 0; a < 3; a++) vrl[a] *= -ap;
    T Fr[3];
    dem_spring(xir, n, vrl, (T)I.kr, (T)I.gr, (T)I.mu_r * fabs(Fnm), Fr);
    T Tt[3], Tr[3];
    cross3(bi, Ft, Tt);
    cross3(n, Fr, Tr);
    T mFt[3] = {-Ft[0], -Ft[1], -Ft[2]}, Ttj[3];
    cross3(bj, mFt, Ttj);
    for (int a = 0; a < 3; a++) {
        rec[a] = Fnm * n[a] + Ft[a];
        rec[3 + a] = Tt[a] - ap * Tr[a];
        rec[6 + a] = -(Fnm * n[a] + Ft[a]);
        rec[9 + a] = Ttj[a] + ap * Tr[a];
    }
}

// orientation: exact rotation by |w| about w (unit quaternion, FP64 storage)
template <class T>
__device__ void quat_rotate(double *q, const T *w)
{
    T wm = sqrt(dot3(w, w));
    if (wm == T(0)) return;
    T h = T(0.5) * wm, s = sin(h) / wm;
    T d0 = cos(h), d1 = s * w[0], d2 = s * w[1], d3 = s * w[2];
    T q0 = (T)q[0], q1 = (T)q[1], q2 = (T)q[2], q3 = (T)q[3];
    T r0 = d0 * q0 - d1 * q1 - d2 * q2 - d3 * q3;
    T r1 = d0 * q1 + d1 * q0 + d2 * q3 - d3 * q2;
    T r2 = d0 * q2 - d1 * q3 + d2 * q0 + d3 * q1;
    T r3 = d0 * q3 + d1 * q2 - d2 * q1 + d3 * q0;
    T l = sqrt(r0 * r0 + r1 * r1 + r2 * r2 + r3 * r3);
    q[0] = r0 / l; q[1] = r1 / l; q[2] = r2 / l; q[3] = r3 / l;
}

// pair index c in [0, np(np-1)/2) -> (i, j), i < j, lexicographic
__device__ __forceinline__ void pair_of(int c, int np, int *i, int *j)
{
    int a = 0;
    while (c >= np - 1 - a) {
        c -= np - 1 - a;
        a++;
    }
    *i = a;
    *j = a + 1 + c;
}

__device__ __forceinline__ int pair_index(int i, int j, int np) { return i * np - i * (i + 1) / 2 + (j - i - 1); }

// Velocity-Verlet prediction per particle (kept in its xn) and contact forces,
// one thread per contact (substrate contacts, then pairs), kept per contact; one
// block per instance.  All of it follows from the particles' state and the
// previous step's forces, so it runs early in the step, beside the fluid
// kernels.  Block 0 counts the step for the record ring.
constexpr int CONTACT_THREADS = 128;
template <class T>
__global__ void __launch_bounds__(CONTACT_THREADS) k_contacts(Lattice L)
{
    const InstDev &I = L.inst[blockIdx.x];
    const int np = I.np;
    const int tid = threadIdx.x;
    if (L.ring_ctr && blockIdx.x == 0 && tid == 0) *L.ring_ctr += 1;
    if (np == 0) return;
    PartDev *P = L.parts + I.part_off;
    double *hist = L.hist + (long long)I.hist_off * 6;
    double *rec = L.crec + (long long)I.crec_off * 12;
    __shared__ double xn[3 * MAX_PART];
    __shared__ T vp[3 * MAX_PART], wp[3 * MAX_PART];
    for (int k = tid; k < 3 * np; k += blockDim.x) {
        const int p = k / 3, a = k - 3 * p;
        const PartDev &q = P[p];
        const double acc = q.kin ? 0.0 : q.Fp[a] * q.inv_m, alp = q.kin ? 0.0 : q.Tp[a] * q.inv_I;
        xn[k] = q.x[a] + q.v[a] + 0.5 * acc;
        vp[k] = (T)(q.v[a] + acc);
        wp[k] = (T)(q.w[a] + alp);
        P[p].xn[a] = xn[k];
    }
    __syncthreads();
    const int npair = np * (np - 1) / 2;
    for (int c = tid; c < np + npair; c += blockDim.x) {
        double *r = rec + 12 * c;
        T rt[12];
        for (int a = 0; a < 12; a++) rt[a] = T(0);
        double *hs;
        T xi[6];
        bool touch = false;
        if (c < np) {
            // particle-substrate contact, delta = R_c - (z_p - 0.5); history record c
            const int p = c;
            hs = hist + 6 * p;
            for (int a = 0; a < 6; a++) xi[a] = (T)hs[a];
            const double delta = P[p].Rc - (xn[3 * p + 2] - 0.5);
            if (I.wall_z0 && delta > 0.0) {
                const T n[3] = {T(0), T(0), T(1)};
                dem_contact<T>(I, P, p, -1, vp, wp, n, (T)delta, xi, xi + 3, rt);
                touch = true;
            }
        } else {
            // particle pair, delta_ij = R_c,i + R_c,j - |X_i - X_j|; history record np + i*np + j
            int i, j;
            pair_of(c - np, np, &i, &j);
            hs = hist + 6 * (np + i * np + j);
            for (int a = 0; a < 6; a++) xi[a] = (T)hs[a];
            const double d[3] = {min_image(xn[3 * i] - xn[3 * j], I.nx), min_image(xn[3 * i + 1] - xn[3 * j + 1], I.ny),
                                 min_image(xn[3 * i + 2] - xn[3 * j + 2], I.nz)};
            const double dl = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
            const double delta = P[i].Rc + P[j].Rc - dl;
            if (delta > 0.0 && dl > 0.0) {
                const T n[3] = {(T)(d[0] / dl), (T)(d[1] / dl), (T)(d[2] / dl)};
                dem_contact<T>(I, P, i, j, vp, wp, n, (T)delta, xi, xi + 3, rt);
                touch = true;
            }
        }
        for (int a = 0; a < 6; a++) hs[a] = touch ? (double)xi[a] : 0.0;
        for (int a = 0; a < 12; a++) r[a] = (double)rt[a];
    }
}

// The step of a particle, by one warp: the fluid forces from the block partials
// of the momentum-exchange and capillary kernels (lanes over a fixed block
// stride, then warp_sums, WARPS of them for the momentum exchange's and their
// sums in order; sum_fluid 0: the surrogate has set them), contacts
// added in a fixed order (substrate, then partners in increasing index), the
// velocity-Verlet correction with lane a and 3 + a on axis a, and the record
// in the record ring.  It also empties the boundary and refill lists that the
// geometry kernels after it fill.  One warp a CTA: the particles' FP64 chains
// run on as many SMs (a CTA of 8 warps per instance, contacts included, took
// 28 us for 8 particles and 17 for one; now 14, and 6 for the contacts).  A large
// sphere has a partial for each 64 nodes of its cube (R = 8: 145, 16: 792, 60:
// 30518), a round trip for every 32 that a warp takes: the kernel took 14, 31 and
// 843 us with one warp, 14, 17 and 126 with eight (sixteen 15, 18 and 120).
constexpr int DEM_WARPS = 8;
constexpr int DEM_ONE_WARP = 96;  // partials that one warp takes
template <class T, bool BUOY, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_dem(Lattice L, int sum_fluid)
{
    const int pg = blockIdx.x, lane = threadIdx.x;
    PartDev &P = L.parts[pg];
    __shared__ double wide[WARPS > 1 ? WARPS : 1][MEM_PART];
    if constexpr (WARPS > 1) {
        if (sum_fluid) {
            double m[16];
            for (int a = 0; a < 16; a++) m[a] = 0.0;
            for (int b = threadIdx.x; b < L.mem_blocks; b += 32 * WARPS)
                for (int a = 0; a < MEM_PART; a++) m[a] += L.mem_part[((long long)pg * L.mem_blocks + b) * MEM_PART + a];
            warp_sums<16>(m);
            const int l = threadIdx.x & 31;
            if (l % 2 == 0 && l / 2 < MEM_PART) wide[threadIdx.x >> 5][l / 2] = m[0];
            __syncthreads();
        }
        if (threadIdx.x >= 32) return;  // the first warp goes on
    }
    if (pg == 0 && lane < 4) L.list_n[lane] = 0;
    const InstDev &I = L.inst[P.inst];
    const int np = I.np, p = P.local;
    const double *rec = L.crec + (long long)I.crec_off * 12;
    __shared__ double s[20], now[6];
    if (sum_fluid) {
        double m[16], c[8];
        for (int a = 0; a < 16; a++) m[a] = 0.0;
        for (int a = 0; a < 8; a++) c[a] = 0.0;
        constexpr int NC = BUOY ? 8 : 6;  // capillary partials used
        for (int b = lane; b < CAP_BLOCKS; b += 32)
            for (int a = 0; a < NC; a++) c[a] += L.cap_part[((long long)pg * CAP_BLOCKS + b) * CAP_PART + a];
        if constexpr (WARPS > 1) {
            if (lane < MEM_PART) {
                double t = wide[0][lane];
                for (int w = 1; w < WARPS; w++) t += wide[w][lane];
                s[lane] = t;
            }
        } else {
            for (int b = lane; b < L.mem_blocks; b += 32)
                for (int a = 0; a < MEM_PART; a++) m[a] += L.mem_part[((long long)pg * L.mem_blocks + b) * MEM_PART + a];
            warp_sums<16>(m);
            if (lane % 2 == 0 && lane / 2 < MEM_PART) s[lane / 2] = m[0];
        }
        warp_sums<8>(c);
        if (lane % 4 == 0) s[12 + lane / 4] = c[0];
        __syncwarp();
        if (lane < 3) {
            // momentum exchange: small part plus the exact rest part
            // -(rho0/18) K, -(rho0/18) (M - delta x K), M = (2M)/2
            const double g = -I.rho0 / 18.0;
            const int a1 = lane == 2 ? 0 : lane + 1, a2 = lane == 0 ? 2 : lane - 1;
            const double d1 = P.x[a1] - floor(P.x[a1]), d2 = P.x[a2] - floor(P.x[a2]);
            P.Feta[lane] = s[lane] + g * s[6 + lane];
            P.Teta[lane] = s[3 + lane] + g * (0.5 * s[9 + lane] - (d1 * s[6 + a2] - d2 * s[6 + a1]));
            P.Fsig[lane] = s[12 + lane];
            P.Tsig[lane] = s[15 + lane];
            // buoyancy (reading c28): a flat interface at height h = (2a - 1) R
            // above the centre leaves the volume fraction (1 + t)^2 (2 - t)/4,
            // t = h/R, of the sphere below it (a spherical zone's area is
            // proportional to its height)
            if constexpr (BUOY) {
                double sub = 0.0;
                if (s[19] > 0.0) {
                    const double t = 2.0 * (s[18] / s[19]) - 1.0;
                    sub = (1.0 + t) * (1.0 + t) * (2.0 - t) / 4.0;
                }
                if (lane == 0) P.sub = sub;
                P.Fb[lane] = 4.0 / 3.0 * M_PI * P.R * P.R * P.R * sub * I.buoy[lane];
            }
        }
        __syncwarp();
    }
    // contacts: lanes 0..2 the force, 3..5 the torque
    double contact = 0.0, total = 0.0, wold = 0.0;
    if (lane < 6) {
        contact = rec[12 * p + lane];
#pragma unroll 4
        for (int q = 0; q < np; q++) {
            if (q == p) continue;
            // p is the second member of (q, p), q < p
            contact += rec[12 * (np + (q < p ? pair_index(q, p, np) : pair_index(p, q, np))) + (q < p ? 6 : 0) + lane];
        }
        if (lane < 3) {
            P.Fc[lane] = contact;
            total = contact + I.g_part[lane] + P.Feta[lane] + P.Fsig[lane] + P.Fb[lane];
            if (!P.kin) P.v[lane] += 0.5 * (P.Fp[lane] + total) * P.inv_m;
            P.Fp[lane] = total;
        } else {
            const int a = lane - 3;
            P.Tc[a] = contact;
            total = contact + P.Teta[a] + P.Tsig[a];
            wold = P.w[a];
            if (!P.kin) P.w[a] += 0.5 * (P.Tp[a] + total) * P.inv_I;
            P.Tp[a] = total;
            now[a] = 0.5 * (wold + P.w[a]);
        }
    }
    // the geometry kernels assume a move below the margin: a larger or
    // non-finite one sets the status and leaves the particle where it was
    // (the run is reported unstable), so that nothing indexes with it
    const bool near = lane >= 3 || fabs(P.xn[lane] - P.x[lane]) < GEOM_MARGIN - 1;
    const bool ok = __all_sync(0xffffffffu, near);
    if (lane < 3) {
        const int per = lane == 0 ? I.nx : (lane == 1 ? I.ny : I.nz);
        const double x0 = P.x[lane], xn = P.xn[lane];
        P.x_old[lane] = x0;
        P.xfo[lane] = P.xf[lane];
        // periodic domain: positions kept in [0, n) (the move is below a period)
        const double x1 = !ok ? x0 : (xn < 0.0 ? xn + per : (xn >= per ? xn - per : xn));
        P.x[lane] = x1;
        P.xf[lane] = (float)x1;
    }
    __syncwarp();
    if (lane == 0) {
        if (!ok) atomicOr(L.status, ST_DISPLACEMENT);
        const T wm[3] = {(T)now[0], (T)now[1], (T)now[2]};
        quat_rotate<T>(P.q, wm);
    }
    __syncwarp();
    if (L.ring) {
        double *slot = L.ring + ((size_t)((*L.ring_ctr - 1) % L.ring_slots) * L.n_parts + pg) * RECORD;
        for (int a = lane; a < RECORD; a += 32) slot[a] = record_entry(P, a);
    }
}

// ---------------------------------------------------------------------------
// Geometry update and refilling (Sec. V C)
// ---------------------------------------------------------------------------
// owner of node (x,y,z) for the particle positions `which` (0: current, 1:
// previous): |x - x_p|^2 < R_p^2, decided in single precision when clear of
// the sphere surface by a margin and in double precision otherwise
__device__ __forceinline__ int particle_owner(const InstDev &I, const PartDev *parts, int x, int y, int z, int which)
{
    for (int p = 0; p < I.np; p++) {
        const PartDev &P = parts[I.part_off + p];
        const float *cf = which ? P.xfo : P.xf;
        const float e0 = min_image_r<float>((float)x - cf[0], I.nx);
        const float e1 = min_image_r<float>((float)y - cf[1], I.ny);
        const float e2 = min_image_r<float>((float)z - cf[2], I.nz);
        const float d2 = e0 * e0 + e1 * e1 + e2 * e2;
        if (d2 > P.R2hi) continue;
        if (d2 < P.R2lo) return 2 + p;
        const double *c = which ? P.x_old : P.x;
        const double d0 = min_image(x - c[0], I.nx), d1 = min_image(y - c[1], I.ny), dd = min_image(z - c[2], I.nz);
        if (d0 * d0 + d1 * d1 + dd * dd < P.R * P.R) return 2 + p;
    }
    return OWN_FLUID;
}

// is node (x, y, z) inside particle P at its current (which 0) or previous position
__device__ __forceinline__ bool inside_particle(const InstDev &I, const PartDev &P, int x, int y, int z, int which)
{
    const float *cf = which ? P.xfo : P.xf;
    const float e0 = min_image_r<float>((float)x - cf[0], I.nx);
    const float e1 = min_image_r<float>((float)y - cf[1], I.ny);
    const float e2 = min_image_r<float>((float)z - cf[2], I.nz);
    const float d2 = e0 * e0 + e1 * e1 + e2 * e2;
    if (d2 > P.R2hi) return false;
    if (d2 < P.R2lo) return true;
    const double *c = which ? P.x_old : P.x;
    const double d0 = min_image(x - c[0], I.nx), d1 = min_image(y - c[1], I.ny), dd = min_image(z - c[2], I.nz);
    return d0 * d0 + d1 * d1 + dd * dd < P.R * P.R;
}

// New owner and fresh bit inside a particle's region (a pure function of the
// particle positions, so overlapping regions write identical bytes).  Only a
// node inside the region's own particle, now or before, or left fresh by the
// step before can change here: the others cost two distances (with all
// particles' distances taken for every node, 512 spheres R = 3 took 126 us,
// now 44).  Uncovered and newly covered nodes are listed once, for the refill.
__global__ void __launch_bounds__(PART_THREADS) k_geom_owner(Lattice L, FastDiv fd)
{
    const PartDev &P = L.parts[blockIdx.y];
    const InstDev &I = L.inst[P.inst];
    Region reg;
    reg.init(P.xf, (int)fd.d, I.nx, I.ny, I.nz);
    const int mine = 2 + P.local;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < reg.count();
         t += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        reg.coord(t, fd, I.nx, I.ny, I.nz, &x, &y, &z);
        const int n = (z * I.ny + y) * I.nx + x;
        uint8_t *fl = L.flags + I.node_off + n;
        const uint8_t old = *fl;
        if (own_static(old & OWNER_MASK)) continue;
        if (!(old & FRESH_BIT) && !inside_particle(I, P, x, y, z, 0) && !inside_particle(I, P, x, y, z, 1)) continue;
        const int own = particle_owner(I, L.parts, x, y, z, 0);
        const int prev = particle_owner(I, L.parts, x, y, z, 1);
        uint8_t f = (uint8_t)own;
        if (own == OWN_FLUID && prev != OWN_FLUID) {
            f |= FRESH_BIT;
            if (prev == mine) L.fresh[atomicAdd(L.list_n + LIST_FRESH, 1ull)] = list_entry(P.inst, n);
        }
        if (own == mine && prev == OWN_FLUID) L.covered[atomicAdd(L.list_n + LIST_COVERED, 1ull)] = list_entry(P.inst, n);
        *fl = (uint8_t)(f | (old & BOUND_BIT));
    }
}

// boundary bit: fluid with a solid neighbour, or solid with a fluid neighbour.
// *mine: some neighbour is owned by `owner`; returns the flags.
__device__ __forceinline__ uint8_t set_boundary(const Lattice &L, const InstDev &I, int x, int y, int z, int owner,
                                                bool *mine)
{
    const uint8_t *fli = L.flags + I.node_off;
    const int n = (z * I.ny + y) * I.nx + x;
    Nbr nb;
    nb.init(x, y, z, I.nx, I.ny, I.nz);
    uint8_t o[Q];
    o[0] = fli[n];
#pragma unroll
    for (int i = 1; i < Q; i++) o[i] = fli[nb.at(cx(i), cy(i), cz(i))];
    const bool fluid = (o[0] & OWNER_MASK) == OWN_FLUID;
    bool b = false, m = false;
#pragma unroll
    for (int i = 1; i < Q; i++) {
        const int ow = o[i] & OWNER_MASK;
        b |= (ow == OWN_FLUID) != fluid;
        m |= ow == owner;
    }
    const uint8_t f = (uint8_t)((o[0] & ~BOUND_BIT) | (b ? BOUND_BIT : 0));
    if (f != o[0]) L.flags[I.node_off + n] = f;
    *mine = m;
    return f;
}

// Boundary bits around the particles, and the next step's lists: the fluid
// nodes next to a particle (L.pbl, for the boundary passes) and the particles'
// solid nodes next to fluid (L.psl, for the solid-phi fill), appended with one
// atomic per warp; order within a list does not matter, a node next to two
// particles is listed twice and written twice with the same value.  A bit can
// change only within one link of a node whose owner changed, i.e. within
// the particle's last displacement and one link of its surface: the other
// nodes of the cube cost a distance (all: the bits of every node and no lists,
// when particles are added); the cube is cut to what the surface reaches (23 -> 11
// nodes a side there; its nodes are found by integer division, no slower than
// by a precomputed one).  512 spheres R = 3: 80 us with 18 flags read for every
// node, 43 with the whole cube's distances, now 22.
__global__ void __launch_bounds__(PART_THREADS) k_geom_surface(Lattice L, FastDiv fd, int all)
{
    const PartDev &P = L.parts[blockIdx.y];
    const InstDev &I = L.inst[P.inst];
    const int mine = 2 + P.local;
    const float m0 = min_image_r<float>(P.xf[0] - P.xfo[0], I.nx), m1 = min_image_r<float>(P.xf[1] - P.xfo[1], I.ny),
                m2 = min_image_r<float>(P.xf[2] - P.xfo[2], I.nz);
    // one link is at most sqrt 2; 0.1 covers the single-precision distance
    const float reach = sqrtf(m0 * m0 + m1 * m1 + m2 * m2) + 1.52f;
    const float lo = fmaxf(P.Rf - reach, 0.0f), hi = P.Rf + reach, lo2 = P.Rf > reach ? lo * lo : -1.0f, hi2 = hi * hi;
    // nodes within hi of the centre lie floor(hi) below to floor(hi) + 1 above its floor
    Region reg;
    reg.init(P.xf, all ? (int)fd.d : min((int)fd.d, 2 * (int)hi + 3), I.nx, I.ny, I.nz);
    const long long count = reg.count();
    const int lane = threadIdx.x & 31;
    auto append = [&](bool take, long long e, long long *list, unsigned long long *n) {
        const unsigned m = __ballot_sync(0xffffffffu, take);
        if (!m) return;
        const int leader = __ffs(m) - 1;
        unsigned long long base = 0;
        if (lane == leader) base = atomicAdd(n, (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (take) list[base + __popc(m & ((1u << lane) - 1u))] = e;
    };
    // warp-uniform trip count: every lane takes part in the ballots
    for (long long t0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); t0 < count;
         t0 += (long long)gridDim.x * blockDim.x) {
        const long long t = t0 + lane;
        bool fluid = false, solid = false;
        long long e = 0;
        if (t < count) {
            int x, y, z;
            reg.coord(t, fd, I.nx, I.ny, I.nz, &x, &y, &z);
            const float e0 = min_image_r<float>((float)x - P.xf[0], I.nx), e1 = min_image_r<float>((float)y - P.xf[1], I.ny),
                        e2 = min_image_r<float>((float)z - P.xf[2], I.nz);
            const float d2 = e0 * e0 + e1 * e1 + e2 * e2;
            if (all || (d2 >= lo2 && d2 <= hi2)) {
                bool next;
                const uint8_t f = set_boundary(L, I, x, y, z, mine, &next);
                const int own = f & OWNER_MASK;
                fluid = own == OWN_FLUID && next;
                solid = own == mine && (f & BOUND_BIT);
                e = list_entry(P.inst, (z * I.ny + y) * I.nx + x);
            }
        }
        if (all) continue;
        append(fluid, e, L.pbl, L.list_n + LIST_FLUID);
        append(solid, e, L.psl, L.list_n + LIST_SOLID);
    }
}

__global__ void k_boundary_full(Lattice L, int inst)
{
    const InstDev &I = L.inst[inst];
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < I.N;
         n += (long long)gridDim.x * blockDim.x) {
        int x = (int)(n % I.nx), y = (int)((n / I.nx) % I.ny), z = (int)(n / ((long long)I.nx * I.ny));
        bool next;
        set_boundary(L, I, x, y, z, -1, &next);
    }
}

// Sec. V C refilling (Caiazzo 2008): a node uncovered this step gets
// f^{a,b} = feq(rho^{a,b}, u_p + w_p x (x - x_p)), rho^{a,b} the mean over the
// 18 moving-direction neighbours that are fluid and not fresh (two hops out if
// none; ambient (0, rho0) if still none).
//
// In the stored form (F* and the colour record (phi, b n) per node) the
// refilled state is F_i = (rho/rho0) e_i - 1 with the record
// (phi = (rho^a - rho^b)/rho, 0): its colour offsets (rho^a - rho^b)/rho0 e_i
// are phi (1 + F_i) exactly.  A neighbour's rho^a - rho^b is phi rho (its
// colour offsets sum to phi (1 + sum w F)).
//
// Few nodes are uncovered per step (about the swept surface area): one warp
// works on each listed one, lane i-1 takes neighbour i and issues its 19
// population loads at once, the sums meet in a shuffle reduction and lane i
// writes direction i.  The nodes newly covered get their solid mark.
template <class R>
__device__ __forceinline__ R warp_sum(R v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <class S>
__device__ void refill_node(const InstDev &I, const PartDev *parts, const Pop<S> &pop,
                            typename Store<S>::real *ph, ColSlotOf<S> col, const uint8_t *fli,
                            int x, int y, int z, int lane)
{
    using R = typename Store<S>::real;
    R sF = 0, sG = 0;
    int nf = 0;
    for (int hop = 1; hop <= 2 && nf == 0; hop++) {
        R aF = 0, aG = 0;
        int ok = 0;
        if (lane < Q - 1) {
            const int i = lane + 1;
            const int X = ((x + hop * cx(i)) % I.nx + I.nx) % I.nx;
            const int Y = ((y + hop * cy(i)) % I.ny + I.ny) % I.ny;
            const int Z = ((z + hop * cz(i)) % I.nz + I.nz) % I.nz;
            const int m = (Z * I.ny + Y) * I.nx + X;
            const uint8_t fm = fli[m];
            if ((fm & OWNER_MASK) == OWN_FLUID && !(fm & FRESH_BIT)) {
                ok = 1;
#pragma unroll
                for (int j = 0; j < Q; j++) aF += wgt<R>(j) * (R(1) + pop.F(j, m));
                aG = col.phi(m) * aF;
            }
        }
        sF = warp_sum(aF);
        sG = warp_sum(aG);
        nf = __reduce_add_sync(0xffffffffu, ok);
    }
    // mean rho/rho0 and (rho^a - rho^b)/rho0 of the neighbours
    R rr, rd;
    if (nf > 0) { rr = sF / nf; rd = sG / nf; }
    else { rr = R(1); rd = R(-1); }
    if (lane >= Q) return;
    const int prev = particle_owner(I, parts, x, y, z, 1);
    const PartDev &P = parts[I.part_off + (prev >= 2 ? prev - 2 : 0)];
    R c[3];
    centre(P, c);
    const R d0 = min_image_r<R>(x - c[0], I.nx), d1 = min_image_r<R>(y - c[1], I.ny),
            d2 = min_image_r<R>(z - c[2], I.nz);
    const R w[3] = {(R)P.w[0], (R)P.w[1], (R)P.w[2]};
    const R u[3] = {(R)P.v[0] + w[1] * d2 - w[2] * d1, (R)P.v[1] + w[2] * d0 - w[0] * d2,
                    (R)P.v[2] + w[0] * d1 - w[1] * d0};
    const R uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const int i = lane;
    const int n = (z * I.ny + y) * I.nx + x;
    const R cu = cx(i) * u[0] + cy(i) * u[1] + cz(i) * u[2];
    const R e = R(1) + R(3) * cu + R(4.5) * cu * cu - R(1.5) * uu;
    pop.setF(i, n, rr * e - R(1));
    if (lane == 0) {
        ph[n] = rd / rr;
        col.shifted(n).set(ColRec<R>{rd / rr, R(0), R(0), R(0)});
    }
}

constexpr int REFILL_THREADS = 128, REFILL_CTAS = 64;
template <class S>
__global__ void __launch_bounds__(REFILL_THREADS) k_refill(Lattice L, int nxt)
{
    using R = typename Store<S>::real;
    const long long nf = (long long)L.list_n[LIST_FRESH], nc = (long long)L.list_n[LIST_COVERED];
    const int lane = threadIdx.x & 31;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    for (long long k = warp; k < nf; k += (long long)gridDim.x * (REFILL_THREADS / 32)) {
        const long long e = L.fresh[k];
        const InstDev &I = L.inst[e >> 32];
        const int n = (int)(unsigned)e, row = n / I.nx, z = row / I.ny;
        refill_node<S>(I, L.parts, Pop<S>(L.pop[nxt], I), (R *)L.phi + I.node_off, col_slot<S>(L, I.node_off),
                       L.flags + I.node_off, n - row * I.nx, row - z * I.ny, z, lane);
    }
    if (sizeof(S) >= 4)
        for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < nc;
             k += (long long)gridDim.x * blockDim.x) {
            const long long e = L.covered[k];
            set_solid_mark(((GradRec<R> *)L.grad)[L.inst[e >> 32].node_off + (unsigned)e]);
        }
}

// initial particle marking: owner at the current positions, no fresh nodes
__global__ void __launch_bounds__(PART_THREADS) k_mark(Lattice L, FastDiv fd)
{
    const PartDev &P = L.parts[blockIdx.y];
    const InstDev &I = L.inst[P.inst];
    Region reg;
    reg.init(P.xf, (int)fd.d, I.nx, I.ny, I.nz);
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < reg.count();
         t += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        reg.coord(t, fd, I.nx, I.ny, I.nz, &x, &y, &z);
        const long long g = I.node_off + ((long long)z * I.ny + y) * I.nx + x;
        const uint8_t old = L.flags[g];
        if (own_static(old & OWNER_MASK)) continue;
        L.flags[g] = (uint8_t)(particle_owner(I, L.parts, x, y, z, 0) | (old & BOUND_BIT));
    }
}

// ---------------------------------------------------------------------------
static FastDiv divide_by(int side)
{
    FastDiv fd;
    fd.set((unsigned)side);
    return fd;
}

template <class S>
void launch_momentum_exchange(const Lattice &L, int cur, cudaStream_t st, long long *launches, const Marker &mk)
{
    if (L.n_parts == 0) return;
    mk(STAGE_MEM, 0);
    k_mem<S><<<dim3(L.mem_blocks, L.n_parts), MEM_THREADS, 0, st>>>(L, cur, divide_by(L.mem_side));
    mk(STAGE_MEM, 1);
    *launches += 1;
}

template <class S>
void launch_capillary(const Lattice &L, cudaStream_t st, long long *launches, const Marker &mk)
{
    if (L.n_parts == 0) return;
    mk(STAGE_CAPILLARY, 0);
    if (L.buoyancy)
        k_capillary<S, true><<<dim3(CAP_BLOCKS, L.n_parts), CAP_THREADS, 0, st>>>(L);
    else
        k_capillary<S, false><<<dim3(CAP_BLOCKS, L.n_parts), CAP_THREADS, 0, st>>>(L);
    mk(STAGE_CAPILLARY, 1);
    *launches += 1;
}

template <class S>
void launch_contacts(const Lattice &L, cudaStream_t st, long long *launches, const Marker &mk)
{
    if (L.n_parts == 0) return;
    mk(STAGE_CONTACTS, 0);
    k_contacts<typename Store<S>::real><<<L.n_inst, CONTACT_THREADS, 0, st>>>(L);
    mk(STAGE_CONTACTS, 1);
    *launches += 1;
}

template <class S>
void launch_dem(const Lattice &L, cudaStream_t st, long long *launches, const Marker &mk, bool sum_fluid)
{
    using R = typename Store<S>::real;
    if (L.n_parts == 0) return;
    mk(STAGE_DEM, 0);
    const bool wide = sum_fluid && L.mem_blocks > DEM_ONE_WARP;
    auto kernel = L.buoyancy ? (wide ? k_dem<R, true, DEM_WARPS> : k_dem<R, true, 1>)
                             : (wide ? k_dem<R, false, DEM_WARPS> : k_dem<R, false, 1>);
    kernel<<<L.n_parts, wide ? 32 * DEM_WARPS : 32, 0, st>>>(L, sum_fluid ? 1 : 0);
    mk(STAGE_DEM, 1);
    *launches += 1;
}

void launch_geom_owner(const Lattice &L, cudaStream_t st, long long *launches, const Marker &mk)
{
    if (L.n_parts == 0) return;
    // region sides: the owner update covers the solid of the last two positions,
    // the surface pass one more node around
    mk(STAGE_GEOM_OWNER, 0);
    k_geom_owner<<<dim3(L.geom_blocks, L.n_parts), PART_THREADS, 0, st>>>(L, divide_by(L.geom_side));
    mk(STAGE_GEOM_OWNER, 1);
    *launches += 1;
}

void launch_geom_surface(const Lattice &L, cudaStream_t st, long long *launches, const Marker &mk)
{
    if (L.n_parts == 0) return;
    mk(STAGE_GEOM_BOUND, 0);
    k_geom_surface<<<dim3(L.geom_blocks, L.n_parts), PART_THREADS, 0, st>>>(L, divide_by(L.geom_side + 2), 0);
    mk(STAGE_GEOM_BOUND, 1);
    *launches += 1;
}

template <class S>
void launch_refill(const Lattice &L, int nxt, cudaStream_t st, long long *launches, const Marker &mk)
{
    if (L.n_parts == 0) return;
    mk(STAGE_REFILL, 0);
    k_refill<S><<<REFILL_CTAS, REFILL_THREADS, 0, st>>>(L, nxt);
    mk(STAGE_REFILL, 1);
    *launches += 1;
}

void launch_mark_particles(const Lattice &L, cudaStream_t st)
{
    if (L.n_parts == 0) return;
    k_mark<<<dim3(L.geom_blocks, L.n_parts), PART_THREADS, 0, st>>>(L, divide_by(L.geom_side));
    k_geom_surface<<<dim3(L.geom_blocks, L.n_parts), PART_THREADS, 0, st>>>(L, divide_by(L.geom_side + 2), 1);
}

void launch_first_lists(const Lattice &L, cudaStream_t st)
{
    if (L.n_parts == 0) return;
    cudaMemsetAsync(L.list_n, 0, 4 * sizeof(unsigned long long), st);
    k_geom_surface<<<dim3(L.geom_blocks, L.n_parts), PART_THREADS, 0, st>>>(L, divide_by(L.geom_side + 2), 0);
}

void launch_boundary_full(const Lattice &L, int inst, long long N, cudaStream_t st)
{
    long long blocks = (N + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    k_boundary_full<<<(unsigned)blocks, 256, 0, st>>>(L, inst);
}

#define INST(S)                                                                                             \
    template void launch_momentum_exchange<S>(const Lattice &, int, cudaStream_t, long long *, const Marker &); \
    template void launch_capillary<S>(const Lattice &, cudaStream_t, long long *, const Marker &);           \
    template void launch_contacts<S>(const Lattice &, cudaStream_t, long long *, const Marker &);            \
    template void launch_dem<S>(const Lattice &, cudaStream_t, long long *, const Marker &, bool);       \
    template void launch_refill<S>(const Lattice &, int, cudaStream_t, long long *, const Marker &);
INST(double)
INST(float)
INST(__half)
INST(__nv_bfloat16)
#undef INST

}  // namespace lbmg
