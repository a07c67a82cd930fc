// Internal device-side definitions of the sm_103a LBM-DEM library.
//
// Lattice: D3Q19 (Sec. IV of arXiv 2505.10171).  The device order is
// i = 0 rest, i = 1..9 the positive half-set h_k below, i = 10..18 their
// opposites, so that the opposite of i is i +- 9; the C ABI order (LBM_C in
// include/lbm.h) is mapped on the way in and out.
//
// Populations are stored as total offsets F_i = f_i/(w_i rho0) - 1, structure
// of arrays pop[i*N + n].  The colour offsets G_i = (f^a_i - f^b_i)/(w_i rho0)
// are not stored: the recolouring step (Sec. IV) leaves every node with
//   G*_i = phi (1 + F*_i) + b (c_i . n)/|c_i|,   b = beta/2 (rho/rho0)(1 - phi^2),
// phi and n the order parameter and interface normal its collision used, so a
// state is F* plus one record (phi, a = b n) per node, and G is rebuilt where
// it is needed: G*_i = phi (1 + F*_i) + (c_i . a)/|c_i|.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <type_traits>
#include <vector>

namespace lbmg {

constexpr int Q = 19;
constexpr int NPOP = 38;

// positive half-set of D3Q19: +x, +y, +z, then the face diagonals
__host__ __device__ constexpr int hx(int k) { return (k == 0 || k == 3 || k == 4 || k == 5 || k == 6) ? 1 : 0; }
__host__ __device__ constexpr int hy(int k) { return (k == 1 || k == 3 || k == 7 || k == 8) ? 1 : (k == 4 ? -1 : 0); }
__host__ __device__ constexpr int hz(int k) { return (k == 2 || k == 5 || k == 7) ? 1 : ((k == 6 || k == 8) ? -1 : 0); }
__host__ __device__ constexpr int cx(int i) { return i == 0 ? 0 : (i <= 9 ? hx(i - 1) : -hx(i - 10)); }
__host__ __device__ constexpr int cy(int i) { return i == 0 ? 0 : (i <= 9 ? hy(i - 1) : -hy(i - 10)); }
__host__ __device__ constexpr int cz(int i) { return i == 0 ? 0 : (i <= 9 ? hz(i - 1) : -hz(i - 10)); }
__host__ __device__ constexpr int opp(int i) { return i == 0 ? 0 : (i <= 9 ? i + 9 : i - 9); }
// the direction with c = (x, y, z)
__host__ __device__ constexpr int dir_of(int x, int y, int z)
{
    for (int i = 0; i < Q; i++)
        if (cx(i) == x && cy(i) == y && cz(i) == z) return i;
    return -1;
}
__host__ __device__ constexpr int csq(int i) { return cx(i) * cx(i) + cy(i) * cy(i) + cz(i) * cz(i); }
template <class T>
__host__ __device__ constexpr T wgt(int i)
{
    return csq(i) == 0 ? T(1) / T(3) : (csq(i) == 1 ? T(1) / T(18) : T(1) / T(36));
}

// node flags: owner in the low 6 bits (0 fluid, 1 static solid, 2+p particle p
// of the instance), bit 6 = refilled this step, bit 7 = next to the other kind
constexpr uint8_t OWNER_MASK = 0x3f;
constexpr uint8_t FRESH_BIT = 0x40;
constexpr uint8_t BOUND_BIT = 0x80;
constexpr uint8_t OWN_FLUID = 0;
constexpr uint8_t OWN_WALL = 1;
// outside of an inlet / outlet face of the Sec. V D pressure boundary (the
// node planes z = 0 and z = nz - 1); particles own 2 .. 62
constexpr uint8_t OWN_PRESS = 63;
__host__ __device__ __forceinline__ bool own_static(int o) { return o == OWN_WALL || o == OWN_PRESS; }

// sticky status bits
constexpr unsigned ST_UNSTABLE = 1u;
constexpr unsigned ST_DISPLACEMENT = 2u;
constexpr unsigned ST_TIMEOUT = 4u;  // a bounded wait for an asynchronous copy gave up

constexpr int MAX_PART = 61;  // particles of an instance (LBM_MAX_PARTICLES)
constexpr int CAP_POINTS = 90 * 180;  // Sec. V F: 2 deg x 2 deg Lagrangian points
constexpr int CAP_THREADS = 256;
constexpr int CAP_BLOCKS = (CAP_POINTS + CAP_THREADS - 1) / CAP_THREADS;
constexpr int CAP_PART = 8;  // per block: F_sig, T_sig, sum s dA, sum dA
constexpr int PART_THREADS = 256;
// the momentum exchange in small CTAs: its links are arithmetic-heavy (FP64
// storage: FP64-bound) and few, so they are spread over the SMs
constexpr int MEM_THREADS = 64;
constexpr int RECORD = 36;  // doubles of a particle record (LBM_PARTICLE_RECORD)
// lists rebuilt each step and their counters
enum ListId { LIST_FLUID = 0, LIST_SOLID, LIST_FRESH, LIST_COVERED };
// doubles per block partial of the momentum exchange: force and torque of the
// small part, then the integer sums K and 2M of the rest part
constexpr int MEM_PART = 12;
constexpr int GEOM_MARGIN = 3;  // lattice units a particle may move per step, < this

// division by an integer fixed when the work items are planned (Granlund and
// Montgomery, "Division by invariant integers using multiplication", 1994):
// q = (mulhi(n, m) + n) >> l with l = ceil(log2 d), m = floor(2^32 (2^l - d)/d) + 1,
// exact for 0 <= n < 2^31 and 1 <= d < 2^31 (n + mulhi stays below 2^32); a
// handful of instructions instead of the runtime divide sequence
struct FastDiv {
    unsigned d, m;
    int l;
    void set(unsigned d_)
    {
        d = d_ ? d_ : 1;
        l = 0;
        while ((1ull << l) < d) l++;
        m = (unsigned)((((unsigned long long)1 << 32) * ((1ull << l) - d)) / d + 1);
    }
    __device__ __forceinline__ int div(int n) const { return (int)((__umulhi((unsigned)n, m) + (unsigned)n) >> l); }
};

struct InstDev {
    int nx, ny, nz, np;
    long long N;         // nodes of the instance
    long long node_off;  // first node in the per-node arrays
    long long pop_off;   // byte offset of the instance's population block
    int pstride;         // population stride (N)
    int part_off;        // first particle of the instance
    int hist_off;        // first pair-history record of the instance
    int crec_off;        // first DEM contact record of the instance
    int wall_z0, store_u;
    int press;                 // pressure faces at z = 0.5 and z = nz - 1.5 (Sec. V D)
    double rin, rout;          // their densities over rho0
    float f_rin, f_rout;
    double rho0, sigma, beta, cap_norm, eta_a, eta_b;
    double body_a[3], body_b[3], wall_u[3];
    double cos_tw, sin_tw;
    double grad_eps, wet_max;
    double kn, kt, kr, gn, gt, gr, mu_s, mu_r, dR;
    double g_part[3];
    double buoy[3];      // force per unit particle volume immersed in phase a (reading c28)
    // single-precision copies of the fluid parameters (no FP64 conversions in
    // the FP32 and 16-bit kernels)
    float f_rho0, f_sigma, f_beta, f_eta_a, f_eta_b, f_eps2, f_wet_max;
    float f_body_a[3], f_body_b[3];
    float f_ir0, f_h_ia, f_h_ib;
    float f_wall_u[3];
    float f_cap;  // cap_norm sigma
    // work items of the collision: consecutive nodes
    long long item_start;
    FastDiv fd_nx, fd_ny;
    // surrogate inputs: shell gap, velocity and radius scales
    double sh_gap, sh_uref, sh_rref, sh_box;
    // gradient + curvature work items: gc_tiles_x * gc_tiles_y column tiles x
    // gc_nchunks z-chunks of gc_zc planes
    long long gc_item_start;
    int gc_tiles_x, gc_tiles_y, gc_nchunks, gc_zc;
    FastDiv fd_nchunks, fd_tiles_x;  // gc_nchunks, gc_tiles_x
    // order-parameter work items: ph_tiles_x column tiles along x, ph_nchunks
    // z-chunks of ph_zc planes
    long long ph_item_start;
    int ph_tiles_x, ph_nchunks, ph_zc;
    FastDiv fd_ph_nchunks, fd_ph_tiles_x;
    long long pn_item_start;  // the same of the instances that it takes a node per thread
    // drop-speed control (body force on phase a): component mask, interval,
    // target velocity, PI gains, base force
    int sp_mask, sp_interval;
    double sp_target[3], sp_kp, sp_ki, sp_f0[3];
};

// fluid parameters in the arithmetic precision R
template <class R>
struct FluidPar {
    R rho0, sigma, beta, eta_a, eta_b, eps2, wet_max, ba[3], bb[3];
    R ir0, h_ia, h_ib;  // 1/rho0, 1/(2 eta_a), 1/(2 eta_b)
};
__device__ __forceinline__ void load_par(const InstDev &I, FluidPar<double> &p)
{
    p.rho0 = I.rho0; p.sigma = I.sigma; p.beta = I.beta; p.eta_a = I.eta_a; p.eta_b = I.eta_b;
    p.eps2 = I.grad_eps * I.grad_eps; p.wet_max = I.wet_max;
    for (int a = 0; a < 3; a++) { p.ba[a] = I.body_a[a]; p.bb[a] = I.body_b[a]; }
    p.ir0 = 1.0 / I.rho0; p.h_ia = 0.5 / I.eta_a; p.h_ib = 0.5 / I.eta_b;
}
__device__ __forceinline__ void load_par(const InstDev &I, FluidPar<float> &p)
{
    p.rho0 = I.f_rho0; p.sigma = I.f_sigma; p.beta = I.f_beta; p.eta_a = I.f_eta_a; p.eta_b = I.f_eta_b;
    p.eps2 = I.f_eps2; p.wet_max = I.f_wet_max;
    for (int a = 0; a < 3; a++) { p.ba[a] = I.f_body_a[a]; p.bb[a] = I.f_body_b[a]; }
    p.ir0 = I.f_ir0; p.h_ia = I.f_h_ia; p.h_ib = I.f_h_ib;
}

struct PartDev {
    double x[3], v[3], w[3], q[4];
    double x_old[3];
    double R, Rc, m, I, cos_t, sin_t;
    double inv_m, inv_I;  // 1/m, 1/I
    double Fp[3], Tp[3];
    double Feta[3], Teta[3], Fsig[3], Tsig[3], Fc[3], Tc[3];
    double sub, Fb[3];    // immersed volume fraction in phase a, buoyancy
    double xn[3];         // predicted position of the step
    float xf[3], xfo[3];  // single-precision copies of x and x_old
    float R2lo, R2hi;     // |x - x_p|^2 below / above these is inside / outside for sure
    float Rf;             // R in single precision
    int kin, inst, local;
};

struct Lattice {
    const InstDev *inst;
    int n_inst;
    int buoyancy;        // some instance has a nonzero buoyancy_a: the immersed fractions are summed
    // boundary lists: entries of list_entry, the static ones in node order
    const long long *static_list;  // static solid nodes next to non-static ones
    long long n_static;
    const long long *static_bfl;   // non-static nodes next to static solid ones
    long long n_static_bfl;
    uint8_t *flags;
    int mark;            // bytes of a real where solid nodes' gradient records are marked, 0: 16-bit storage
    void *pop[2];
    void *phi;           // [Ntot] real: the order parameter of the step (outside a step: of the last one)
    void *col;           // [Ntot] ColRec<real>: colour record (phi, b n) of the stored state
    void *grad;          // [Ntot] GradRec<real>: corrected grad(phi) and curvature of fluid nodes
    void *nrm;           // [3][Ntot] real: the normals between the gradient and curvature kernels (null: one marching pass)
    void *u;             // [3][Ntot] real (store_velocity)
    long long Ntot;
    PartDev *parts;
    int n_parts;
    int mem_blocks;      // blocks per particle of the momentum-exchange kernel
    int mem_side;        // side of the cube it covers
    int geom_blocks;     // blocks per particle of the geometry kernels
    int geom_side;       // side of the cube the geometry kernels cover
    // lists of list_entry that the geometry kernels of the step before (for the
    // first step launch_first_lists) have filled, and their lengths by ListId: fluid
    // nodes next to a particle, particle nodes next to fluid, uncovered and
    // covered nodes
    long long *pbl, *psl, *fresh, *covered;
    unsigned long long *list_n;
    int bound_ctas;              // CTAs of the grid-stride boundary passes
    double *mem_part;    // [n_parts][mem_blocks][MEM_PART]
    double *cap_part;    // [n_parts][CAP_BLOCKS][CAP_PART]
    const double *cap_pts;  // [CAP_POINTS][4]: unit normal (3) and sin(alpha) of each surface point
    const float *cap_pts_f; // the same in single precision
    // record ring (null: none): every step's records go to slot (*ring_ctr - 1) mod
    // ring_slots, ring_ctr counting the steps begun
    double *ring;
    int ring_slots;
    long long *ring_ctr;
    double *hist;        // contact springs: per instance np*(np+1) records of 6
    double *crec;        // DEM contact forces: per instance np + np(np-1)/2 records of 12
    unsigned *status;
};

// materialise a value here: the loads it depends on must be issued before
// any branch that follows, so the compiler cannot sink them into the one path
// that uses them (which would put the node's flag load and the population
// loads in series: two dependent DRAM round trips instead of one)
__device__ __forceinline__ void keep(float &v) { asm volatile("" : "+f"(v)); }
__device__ __forceinline__ void keep(double &v) { asm volatile("" : "+d"(v)); }

// programmatic dependent launch: a kernel launched with programmatic stream
// serialisation may start while its predecessor in the stream drains; it must
// wait here before touching anything the predecessor writes or reads.  A
// predecessor signals early that its dependent may be scheduled (all of its
// CTAs have started by then, so the dependent cannot take their places).
// Both are no-ops for a kernel launched without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// streamed populations are read through the read-only path (measured on this
// GPU: as fast as plain loads, faster than evict-first streaming loads)
template <class T>
__device__ __forceinline__ T pop_load(const T *p)
{
    return __ldg(p);
}

// The boundary pass of the order parameter keeps bounced offsets in slots of solid
// nodes (FP32 and FP64 storage); its own threads and the bulk pass beside it load
// such a slot while it may be written, for a node that drops the value.  Those
// loads are plain ones: the read-only path is for memory that nothing writes
// while a kernel runs.  (Same time either way.)
template <class S>
constexpr bool BOUNCE_IN_SLOTS = sizeof(S) >= 4;
template <class T>
__device__ __forceinline__ T pop_load_beside_writes(const T *p)
{
    return BOUNCE_IN_SLOTS<T> ? *p : pop_load(p);
}

template <class S>
struct Store;
template <>
struct Store<double> {
    using real = double;
    static __device__ __forceinline__ double ld(const double *p) { return pop_load(p); }
    static __device__ __forceinline__ double cvt(double v) { return v; }
    static __device__ __forceinline__ void st(double *p, double v) { *p = v; }
};
template <>
struct Store<float> {
    using real = float;
    static __device__ __forceinline__ float ld(const float *p) { return pop_load(p); }
    static __device__ __forceinline__ float cvt(float v) { return v; }
    static __device__ __forceinline__ void st(float *p, float v) { *p = v; }
};
template <>
struct Store<__half> {
    using real = float;
    static __device__ __forceinline__ float ld(const __half *p) { return __half2float(pop_load(p)); }
    static __device__ __forceinline__ float cvt(__half v) { return __half2float(v); }
    static __device__ __forceinline__ void st(__half *p, float v) { *p = __float2half_rn(v); }
};
template <>
struct Store<__nv_bfloat16> {
    using real = float;
    static __device__ __forceinline__ float ld(const __nv_bfloat16 *p) { return __bfloat162float(pop_load(p)); }
    static __device__ __forceinline__ float cvt(__nv_bfloat16 v) { return __bfloat162float(v); }
    static __device__ __forceinline__ void st(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
};

// populations of one instance: F_i (i-major, stride pstride = N) at the
// instance block's byte offset; instance blocks follow one another in node order
template <class S>
struct Pop {
    using FT = S;
    using R = typename Store<S>::real;
    static constexpr size_t node_bytes = Q * sizeof(S);
    FT *f;
    int N;  // stride between directions (the instance's pstride)
    __host__ __device__ __forceinline__ Pop(const void *base, const InstDev &I)
        : f((FT *)((char *)base + I.pop_off)), N(I.pstride)
    {
    }
    __device__ __forceinline__ R F(int i, int m) const { return Store<FT>::ld(f + i * N + m); }
    __device__ __forceinline__ R F_beside_writes(int i, int m) const
    {
        return Store<FT>::cvt(pop_load_beside_writes(f + i * N + m));
    }
    __device__ __forceinline__ void setF(int i, int m, R v) const { Store<FT>::st(f + i * N + m, v); }
};

// two consecutive 16-bit values of a node pair (x even) as one 32-bit access,
// and the pair store of two reals
__device__ __forceinline__ void ld_pair(const __half *p, float &a, float &b)
{
    const __half2 v = __ldg(reinterpret_cast<const __half2 *>(p));
    a = __low2float(v);
    b = __high2float(v);
}
__device__ __forceinline__ void ld_pair(const __nv_bfloat16 *p, float &a, float &b)
{
    const __nv_bfloat162 v = __ldg(reinterpret_cast<const __nv_bfloat162 *>(p));
    a = __low2float(v);
    b = __high2float(v);
}
__device__ __forceinline__ void st_pair(__half *p, float a, float b)
{
    *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(a, b);
}
__device__ __forceinline__ void st_pair(__nv_bfloat16 *p, float a, float b)
{
    *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(a, b);
}

// minimum-image displacement on a periodic axis of n nodes (|d| < 3n/2): the
// same value as d - n floor(d/n + 1/2) without a double-precision division
__host__ __device__ __forceinline__ double min_image(double d, int n)
{
    const double h = 0.5 * n;
    return d >= h ? d - n : (d < -h ? d + n : d);
}

// the same in single precision (|d| < 3n/2)
__device__ __forceinline__ float min_image_f(float d, int n)
{
    const float h = 0.5f * n;
    return d >= h ? d - n : (d < -h ? d + n : d);
}

template <class R>
__device__ __forceinline__ R min_image_r(R d, int n)
{
    const R h = R(0.5) * n;
    return d >= h ? d - n : (d < -h ? d + n : d);
}

// offset d of a node from a particle's centre c, minimum image; whether the
// midpoints of all the node's links (half a node away at most) have that
// image too, so that theirs is d - c_i/2
template <class R>
__device__ __forceinline__ bool node_lever(const InstDev &I, int x, int y, int z, const R *c, R *d)
{
    d[0] = min_image_r<R>((R)x - c[0], I.nx);
    d[1] = min_image_r<R>((R)y - c[1], I.ny);
    d[2] = min_image_r<R>((R)z - c[2], I.nz);
    return fabs(d[0]) < R(0.5) * I.nx - R(0.75) && fabs(d[1]) < R(0.5) * I.ny - R(0.75) &&
           fabs(d[2]) < R(0.5) * I.nz - R(0.75);
}

// periodic neighbourhood of one node: x coordinates and row/plane offsets of
// x-1..x+1, y-1..y+1, z-1..z+1 (instance-local 32-bit node indices; every
// instance has fewer than 2^31/38 nodes)
struct Nbr {
    int X[3], YO[3], ZO[3];
    __device__ __forceinline__ void init(int x, int y, int z, int nx_, int ny_, int nz_)
    {
        const int nxy = nx_ * ny_;
        X[0] = x == 0 ? nx_ - 1 : x - 1; X[1] = x; X[2] = x == nx_ - 1 ? 0 : x + 1;
        YO[0] = (y == 0 ? ny_ - 1 : y - 1) * nx_; YO[1] = y * nx_; YO[2] = (y == ny_ - 1 ? 0 : y + 1) * nx_;
        ZO[0] = (z == 0 ? nz_ - 1 : z - 1) * nxy; ZO[1] = z * nxy; ZO[2] = (z == nz_ - 1 ? 0 : z + 1) * nxy;
    }
    __device__ __forceinline__ int at(int dx, int dy, int dz) const { return ZO[dz + 1] + YO[dy + 1] + X[dx + 1]; }
    __device__ __forceinline__ int idx(int dx, int dy, int dz) const { return at(dx, dy, dz); }
};

// reciprocal and inverse square root: IEEE for double, the fast single-precision
// forms otherwise (the FP32 and 16-bit paths are held to 1e-4 / 2e-3)
__device__ __forceinline__ double frcp(double x) { return 1.0 / x; }
__device__ __forceinline__ float frcp(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ double frsqrt(double x) { return 1.0 / sqrt(x); }
__device__ __forceinline__ float frsqrt(float x) { return rsqrtf(x); }

// cube of side `side` (clamped to the domain) centred on a particle's node
struct Region {
    int lo[3], sz[3];
    // (from the single-precision centre, which may round up to the next node: the
    // sides leave room for that, and FP64 here would bind the kernels that run
    // one thread per node of the cube)
    __device__ __forceinline__ void init(const float *xc, int side, int nx, int ny, int nz)
    {
        const int n[3] = {nx, ny, nz};
        for (int a = 0; a < 3; a++) {
            int s = side < n[a] ? side : n[a];
            sz[a] = s;
            int lo_ = (int)floorf(xc[a]) - (s - 1) / 2;
            lo[a] = s == n[a] ? 0 : lo_;
        }
    }
    __device__ __forceinline__ long long count() const { return (long long)sz[0] * sz[1] * sz[2]; }
    // node t of the cube (t < count < 2^31); lo + i lies in (-n, 2n), so one
    // conditional wrap per axis suffices
    // (fd divides by the side asked for, the size of every axis that it fits)
    __device__ __forceinline__ void coord(long long t, const FastDiv &fd, int nx, int ny, int nz, int *x, int *y,
                                          int *z) const
    {
        const int tt = (int)t;
        const int ij = sz[0] == (int)fd.d ? fd.div(tt) : tt / sz[0];
        const int i = tt - ij * sz[0];
        const int k = sz[1] == (int)fd.d ? fd.div(ij) : ij / sz[1];
        const int j = ij - k * sz[1];
        int a = lo[0] + i, b = lo[1] + j, c = lo[2] + k;
        a += a < 0 ? nx : (a >= nx ? -nx : 0);
        b += b < 0 ? ny : (b >= ny ? -ny : 0);
        c += c < 0 ? nz : (c >= nz ? -nz : 0);
        *x = a;
        *y = b;
        *z = c;
    }
};

// FP32 storage sums the order parameter, the gradient, the curvature and the
// moments of the collision direction by direction, in the order of the
// directions; the other types gather terms (fewer instructions or FP64 operations).
// A regrouped FP32 sum moves phi by some 1e-7, and the wetting rotation
// applies where |phi| < wet_max: a node whose phi lies that close to the cut
// falls on its other side, turns its normal (by 60 degrees at a wall of 150) and
// moves phi by up to 8e-4 from there on.  A run in FP32 follows one order of
// summation for good, so that its results stay the same from one version of
// these kernels to the next.  (In 16-bit storage the offsets' own rounding is
// coarser than any regrouping; in FP64 no node comes that close.)
template <class S>
constexpr bool BY_DIRECTION = std::is_same_v<S, float>;

// Operations rounded as written.  Several copies of the gradient's arithmetic
// (a tile's own nodes, those around it, the form without tiles) must give a
// node the same bits, and the compiler would be free to contract each into
// different multiply-adds (with the copies contracted apart, a symmetric drop
// took up a sideways drift of 1e-4 of its speed).
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// regularised interface normal n = g/sqrt(|g|^2 + eps^2) of FP32 storage;
// returns the norm
template <class R>
__device__ __forceinline__ R dir_normal(const R *g, R eps2, R *nn)
{
    const R m2 = add_rn(fma_rn(g[2], g[2], fma_rn(g[0], g[0], mul_rn(g[1], g[1]))), eps2);
    const R im = frsqrt(m2);
    for (int a = 0; a < 3; a++) nn[a] = mul_rn(g[a], im);
    return mul_rn(m2, im);
}

// The colour record of a node of the stored state (see the top of this
// file): the order parameter phi of the collision that produced it and
// a = b n, one 16-byte (FP64: 32-byte) aligned record, so that a pulled source
// costs one vector load.
template <class R>
struct alignas(4 * sizeof(R)) ColRec {
    R p, a0, a1, a2;
};

// What the gradient pass leaves at a fluid node for the collision and the
// capillary force: the corrected grad(phi) g and the curvature k = div(n) of
// the regularised normals n = g/sqrt(|g|^2 + eps^2), one aligned record (one
// vector load; the normal is formed again from g where it is needed)
template <class R>
struct alignas(4 * sizeof(R)) GradRec {
    R g0, g1, g2, k;
    // the gradient alone (the curvature follows two planes later)
    __device__ __forceinline__ void set_gradient(const R *g)
    {
        struct alignas(2 * sizeof(R)) Pair { R a, b; };
        *reinterpret_cast<Pair *>(&g0) = Pair{g[0], g[1]};
        g2 = g[2];
    }
};

// The curvature slot of a node that was solid in the step's gradient pass: a
// NaN of its own (arithmetic makes the canonical one), so that the FP32 and
// FP64 collision knows its nodes without their flags, which the owner update
// beside it may be changing.  Written when the solid map is built or changed.
__device__ __forceinline__ void set_solid_mark(GradRec<float> &r) { r.k = __int_as_float(0x7fc0dead); }
__device__ __forceinline__ void set_solid_mark(GradRec<double> &r) { r.k = __longlong_as_double(0x7ff8dead00000000ll); }
__device__ __forceinline__ bool solid_mark(const GradRec<float> &r) { return __float_as_int(r.k) == 0x7fc0dead; }
__device__ __forceinline__ bool solid_mark(const GradRec<double> &r)
{
    return __double_as_longlong(r.k) == 0x7ff8dead00000000ll;
}

// entry a of a particle's record (the layout of lbm_particle_forces)
__device__ __forceinline__ double record_entry(const PartDev &q, int a)
{
    static_assert(offsetof(PartDev, Tc) == offsetof(PartDev, Feta) + 15 * sizeof(double) &&
                      offsetof(PartDev, q) == offsetof(PartDev, x) + 9 * sizeof(double) &&
                      offsetof(PartDev, Fb) == offsetof(PartDev, sub) + sizeof(double),
                  "the record's parts are contiguous");
    if (a < 18) return (&q.Feta[0])[a];  // F_eta, T_eta, F_sig, T_sig, F_c, T_c
    if (a < 31) return (&q.x[0])[a - 18];  // x, v, w, q
    return a == 31 ? q.m : (&q.sub)[a - 32];  // sub, F_b
}

// entry of a boundary list: instance and instance-local node
__device__ __forceinline__ long long list_entry(int inst, int n) { return (long long)inst << 32 | (unsigned)n; }

// (c_i . a)/|c_i|: the colour offset G*_i of a record beyond phi (1 + F*_i)
template <class R>
__device__ __forceinline__ R col_rec(int i, const ColRec<R> &c)
{
    R t = 0;
    if (cx(i)) t += cx(i) * c.a0;
    if (cy(i)) t += cy(i) * c.a1;
    if (cz(i)) t += cz(i) * c.a2;
    return csq(i) == 1 ? t : t * R(0.70710678118654752440);
}

// one node's record slot (write side)
template <class R>
struct ColSlot {
    ColRec<R> *p;
    __device__ __forceinline__ void set(const ColRec<R> &c) const { *p = c; }
    // the slot n nodes further on
    __device__ __forceinline__ ColSlot shifted(long long n) const { return ColSlot{p + n}; }
    // phi of the record n nodes further on
    __device__ __forceinline__ R phi(long long n) const { return p[n].p; }
};

// the colour records of an instance (read side)
template <class R>
struct Colour {
    const ColRec<R> *c;
    __device__ __forceinline__ Colour(const Lattice &L, const InstDev &I)
        : c((const ColRec<R> *)L.col + I.node_off)
    {
    }
    __device__ __forceinline__ ColRec<R> at(int m) const { return c[m]; }
};

template <class S>
using ColourOf = Colour<typename Store<S>::real>;
template <class S>
using ColSlotOf = ColSlot<typename Store<S>::real>;

// the record slot of global node g
template <class S>
__device__ __forceinline__ ColSlotOf<S> col_slot(const Lattice &L, long long g)
{
    return ColSlotOf<S>{(ColRec<typename Store<S>::real> *)L.col + g};
}

// Pull streaming (Sec. IV) into fluid node n next to a solid, with the Sec. V A
// halfway bounce-back where the source node is solid:
//   f_i(x) = f*_ibar(x) + 6 w_i rho^{a,b}(x) c_i.u_w,
// rho^{a,b}(x) of the node's own pre-streaming state, u_w at the link midpoint.
// A source on a pressure face (Sec. V D) gives the anti-bounce-back value
//   f_i = -f*_ibar(x) + 2 w_i rho_w [1 + (c_i.u_w)^2/(2 cs^4) - u_w^2/(2 cs^2)],
// rho_w the face's density (inlet below, outlet above), u_w = j*/rho* of the
// node's own post-collision state.  own[i] and F[i] receive the owner of
// direction i's source and the streamed total offset.
// Every flag and population load is issued before any is used, and a
// particle's state is read once per particle met (mostly one), not per link:
// a chain of round trips per link is what these passes would wait on.
template <class S>
__device__ __forceinline__ void gather_links(const InstDev &I, const PartDev *parts, const uint8_t *fli, const Nbr &nb,
                                             const Pop<S> &in, int n, int x, int y, int z, int (&own)[Q],
                                             typename Store<S>::real (&F)[Q])
{
    using R = typename Store<S>::real;
    R oF[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) {
        const int s = nb.at(-cx(i), -cy(i), -cz(i));
        own[i] = fli[s];
        F[i] = in.F_beside_writes(i, s);
        oF[i] = in.F_beside_writes(i, n);
    }
    R sF = 0;
    unsigned long long met = 0;
#pragma unroll
    for (int i = 0; i < Q; i++) {
        sF += wgt<R>(i) * oF[i];
        own[i] &= OWNER_MASK;
        met |= 1ull << own[i];
    }
    const R rr = R(1) + sF;
    if (met >> OWN_WALL & 1) {
        R uw[3];
        for (int a = 0; a < 3; a++) uw[a] = sizeof(R) == 8 ? (R)I.wall_u[a] : (R)I.f_wall_u[a];
#pragma unroll
        for (int i = 1; i < Q; i++)
            if (own[i] == OWN_WALL)
                F[i] = oF[opp(i)] + R(6) * rr * (cx(i) * uw[0] + cy(i) * uw[1] + cz(i) * uw[2]);
    }
    if (met >> OWN_PRESS & 1) {
        R j[3] = {0, 0, 0};
#pragma unroll
        for (int i = 1; i < Q; i++) {
            if (cx(i)) j[0] += wgt<R>(i) * cx(i) * oF[i];
            if (cy(i)) j[1] += wgt<R>(i) * cy(i) * oF[i];
            if (cz(i)) j[2] += wgt<R>(i) * cz(i) * oF[i];
        }
        const R irr = R(1) / rr;
        const R u0 = j[0] * irr, u1 = j[1] * irr, u2 = j[2] * irr;
#pragma unroll
        for (int i = 1; i < Q; i++) {
            if (own[i] != OWN_PRESS) continue;
            const R cu = cx(i) * u0 + cy(i) * u1 + cz(i) * u2;
            const R rw = sizeof(R) == 8 ? (R)(cz(i) > 0 ? I.rin : I.rout) : (R)(cz(i) > 0 ? I.f_rin : I.f_rout);
            F[i] = R(-2) - oF[opp(i)] + R(2) * rw * (R(1) + R(4.5) * cu * cu - R(1.5) * (u0 * u0 + u1 * u1 + u2 * u2));
        }
    }
    met &= ~(1ull << OWN_FLUID | 1ull << OWN_WALL | 1ull << OWN_PRESS);
    while (met) {
        const int o = __ffsll((long long)met) - 1;
        met &= met - 1;
        const PartDev &P = parts[I.part_off + o - 2];
        R c[3], v[3], w[3];
        for (int a = 0; a < 3; a++) {
            c[a] = sizeof(R) == 8 ? (R)P.x[a] : (R)P.xf[a];
            v[a] = (R)P.v[a];
            w[a] = (R)P.w[a];
        }
        // c_i.u_w at the link midpoint is that at the node, since c_i.(w x c_i) = 0:
        // in FP64, whose every instruction counts, one lever for all links instead
        // of 32 instructions a link (48x32x32 with a wall and a sphere: order-
        // parameter boundary pass 28 -> 12 us).  FP32 keeps the other form: with
        // both the pass spills more (66 against 61 us in a tube of radius 40)
        R d[3];
        if (sizeof(R) == 8 && node_lever<R>(I, x, y, z, c, d)) {
            const R u0 = v[0] + (w[1] * d[2] - w[2] * d[1]), u1 = v[1] + (w[2] * d[0] - w[0] * d[2]),
                    u2 = v[2] + (w[0] * d[1] - w[1] * d[0]);
            const R r6 = R(6) * rr;
#pragma unroll
            for (int i = 1; i < Q; i++)
                if (own[i] == o) F[i] = oF[opp(i)] + r6 * (cx(i) * u0 + cy(i) * u1 + cz(i) * u2);
            continue;
        }
#pragma unroll
        for (int i = 1; i < Q; i++) {
            if (own[i] != o) continue;
            // u_w = v + w x (link midpoint - centre), in R: the midpoints are half-integers, exact in either
            const R d0 = min_image_r<R>((x - R(0.5) * cx(i)) - c[0], I.nx), d1 = min_image_r<R>((y - R(0.5) * cy(i)) - c[1], I.ny),
                    d2 = min_image_r<R>((z - R(0.5) * cz(i)) - c[2], I.nz);
            const R u0 = v[0] + (w[1] * d2 - w[2] * d1), u1 = v[1] + (w[2] * d0 - w[0] * d2),
                    u2 = v[2] + (w[0] * d1 - w[1] * d0);
            F[i] = oF[opp(i)] + R(6) * rr * (cx(i) * u0 + cy(i) * u1 + cz(i) * u2);
        }
    }
}

// sum_i w_i G_i of the streamed colour offsets of that node:
// G_i(x) = G*_i(x - c_i) from a fluid source; from a solid one
// G*_ibar(x) + 6 (rho^a - rho^b)(x)/rho0 c_i.u_w, and since
// (rho^a - rho^b)(x) = phi(x) rho(x) that is phi(x)(1 + F_i(x)) - (c_i . a(x))/|c_i|;
// from a pressure face, whose colour split follows the node's own state,
// phi(x)(1 + F_i) + (c_i . a(x))/|c_i|.  The sources' records are read in three
// batches, whatever their owner (a solid node's record is not used).
template <class S>
__device__ __forceinline__ typename Store<S>::real gather_colour(const Nbr &nb, const ColourOf<S> &C, int n,
                                                                 const int (&own)[Q],
                                                                 const typename Store<S>::real (&F)[Q])
{
    using R = typename Store<S>::real;
    const ColRec<R> cn = C.at(n);
    R g = wgt<R>(0) * (cn.p * (R(1) + F[0]));
#pragma unroll
    for (int b = 0; b < 3; b++) {
        ColRec<R> r[6];
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const int i = 1 + 6 * b + k;
            r[k] = C.at(nb.at(-cx(i), -cy(i), -cz(i)));
        }
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const int i = 1 + 6 * b + k;
            const bool fluid = own[i] == OWN_FLUID;
            const ColRec<R> s = {fluid ? r[k].p : cn.p, fluid ? r[k].a0 : cn.a0, fluid ? r[k].a1 : cn.a1,
                                 fluid ? r[k].a2 : cn.a2};
            const R t = col_rec(i, s), st = fluid || own[i] == OWN_PRESS ? t : -t;
            if constexpr (BY_DIRECTION<S>) g = fma_rn(wgt<R>(i), fma_rn(s.p, add_rn(R(1), F[i]), st), g);
            else g += wgt<R>(i) * (s.p * (R(1) + F[i]) + st);
        }
    }
    return g;
}

// Sec. V E geometric wetting: rotate g so that -g/|g| makes the angle theta
// with the outward solid normal ns, keeping |g|; of the two candidates the one
// closer to the original direction is kept.
template <class R>
__device__ __forceinline__ void wetting_rotate(R *g, const R *ns, R cth, R sth)
{
    R gm = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
    if (gm == R(0)) return;
    R st[3] = {-g[0] / gm, -g[1] / gm, -g[2] / gm};
    R ca = ns[0] * st[0] + ns[1] * st[1] + ns[2] * st[2];
    ca = ca > R(1) ? R(1) : (ca < R(-1) ? R(-1) : ca);
    // cos and sin of the angle alpha* between n* and n_s: the FP64 path takes
    // acos / sin / cos as the oracle does; single precision uses the dot and
    // the norm of the cross product (alpha* in [0, pi]), which need no
    // transcendental calls and keep sin alpha* to relative precision where
    // sqrt(1 - cos^2) would lose it (cos alpha* near +-1)
    R sa, cal;
    if (sizeof(R) == 8) {
        const R al = acos(ca);
        sa = sin(al);
        cal = cos(al);
    } else {
        cal = ca;
        const R x0 = ns[1] * st[2] - ns[2] * st[1], x1 = ns[2] * st[0] - ns[0] * st[2],
                x2 = ns[0] * st[1] - ns[1] * st[0];
        sa = sqrt(x0 * x0 + x1 * x1 + x2 * x2);
    }
    if (sa < R(1e-4)) return;  // contact-line direction undefined (n* parallel to n_s)
    R ap1 = cth - sth * cal / sa, ap2 = sth / sa;
    R am1 = cth + sth * cal / sa, am2 = -sth / sa;
    R np_[3], nm_[3];
    for (int a = 0; a < 3; a++) {
        np_[a] = ap1 * ns[a] + ap2 * st[a];
        nm_[a] = am1 * ns[a] + am2 * st[a];
    }
    R dp = np_[0] * st[0] + np_[1] * st[1] + np_[2] * st[2];
    R dm = nm_[0] * st[0] + nm_[1] * st[1] + nm_[2] * st[2];
    const R *nc = dp >= dm ? np_ : nm_;
    for (int a = 0; a < 3; a++) g[a] = -gm * nc[a];
}

// kernel stages, in launch order within a step (for per-kernel timing)
enum Stage {
    STAGE_PHI = 0, STAGE_SOLIDPHI, STAGE_GRAD, STAGE_COLLIDE, STAGE_MEM, STAGE_CAPILLARY, STAGE_DEM,
    STAGE_GEOM_OWNER, STAGE_GEOM_BOUND, STAGE_REFILL, STAGE_FUSED, STAGE_REGION, STAGE_CURV, STAGE_SURROGATE,
    STAGE_PHI_BOUND, STAGE_COLLIDE_BOUND, STAGE_CONTACTS, N_STAGES
};

// optional per-kernel marker: called right before and right after each launch
struct Marker {
    void (*fn)(void *self, int stage, int after) = nullptr;
    void *self = nullptr;
    void operator()(int stage, int after) const
    {
        if (fn) fn(self, stage, after);
    }
};

// host-side hook of the fluid launcher
struct Hook {
    void (*fn)(void *self) = nullptr;
    void *self = nullptr;
    void operator()() const
    {
        if (fn) fn(self);
    }
};

// a second stream with two events: the boundary passes run there, beside the
// bulk kernels (they write disjoint nodes), and what the hooks enqueue
struct SideLane {
    cudaStream_t side = nullptr;
    cudaEvent_t a = nullptr, b = nullptr;
    Hook after_phi_bound;      // after the order parameter's boundary pass and the solid-phi fill
    Hook after_grad;           // once grad(phi) and the curvature of the step are final
    Hook after_collide_bound;  // after the collision's boundary pass (16-bit storage)
};

// host-side kernel launchers (defined in the .cu files)
constexpr int FORM_PLAIN = 2;  // the launch form of the fluid update (the value the ABI names)
struct FluidLaunch {
    int tile;           // 0: node-pair bulk collision where possible; 1: one node per thread
    long long items;    // collision work items (all instances)
    long long ph_items; // order-parameter work items (all instances): marching tiles
    long long pn_items; // and a node per thread
    long long gc_items; // gradient + curvature work items (all instances)
    bool pair;          // every instance has an even nx: node-pair kernels for 16-bit storage
};
// The gradient pass takes a node per thread in FP64 runs and up to this many
// nodes of a context, marching tiles beyond (measured beside the kernels)
constexpr long long GRAD_NODES_MAX = 768 * 1024;
// z-planes per work item of the gradient + curvature kernel for a grid's size and
// the n_sm SMs; dir: FP32 storage
int planned_zchunk(const std::vector<InstDev> &inst, int n_sm, bool dir);
// plan the work items of the gradient + curvature kernel into fz (z-planes per
// item: zc_inst[k] for instance k where set (> 0), else zc_request where set,
// else planned_zchunk); used where L.nrm is null
void plan_gradcurv(std::vector<InstDev> &inst, int zc_request, const std::vector<int> &zc_inst, int n_sm, bool dir,
                   FluidLaunch *fz);
// plan the work items of the order-parameter kernel into fz
void plan_phi(std::vector<InstDev> &inst, int n_sm, bool fp64, FluidLaunch *fz);
// plan the collision's work items into fz (and the divisions by nx and ny)
void plan_items(std::vector<InstDev> &inst, bool fp64, FluidLaunch *fz);
template <class S>
void launch_fluid_step(const Lattice &L, int cur, cudaStream_t st, long long *launches, const Marker &mk,
                       const FluidLaunch &fz, const SideLane &lane = SideLane());
// Verlet prediction and contact forces (from the state before the step)
template <class S>
void launch_contacts(const Lattice &L, cudaStream_t st, long long *launches, const Marker &mk);
// momentum exchange (needs only the step's input populations) and capillary
// force (needs the step's phi and gradients)
template <class S>
void launch_momentum_exchange(const Lattice &L, int cur, cudaStream_t st, long long *launches, const Marker &mk);
template <class S>
void launch_capillary(const Lattice &L, cudaStream_t st, long long *launches, const Marker &mk);
// sum_fluid: gather the momentum-exchange and capillary partial sums first
// (false when the surrogate has written the fluid forces)
template <class S>
void launch_dem(const Lattice &L, cudaStream_t st, long long *launches, const Marker &mk, bool sum_fluid);
// geometry: owners and fresh bits, then boundary bits and lists, and the
// refill of fresh nodes (after the collision)
void launch_geom_owner(const Lattice &L, cudaStream_t st, long long *launches, const Marker &mk);
void launch_geom_surface(const Lattice &L, cudaStream_t st, long long *launches, const Marker &mk);
template <class S>
void launch_refill(const Lattice &L, int nxt, cudaStream_t st, long long *launches, const Marker &mk);

// ---------------------------------------------------------------------------
// learned force surrogate (lbm_mlp.cu)
// ---------------------------------------------------------------------------
constexpr int MLP_NIN = 387, MLP_KIN = 400, MLP_HIDDEN = 128, MLP_NOUT = 6, MLP_SHELL = 96;
constexpr int MLP_OFF_W1 = 0;
constexpr int MLP_OFF_B1 = MLP_OFF_W1 + MLP_HIDDEN * MLP_KIN;
constexpr int MLP_OFF_W2 = MLP_OFF_B1 + MLP_HIDDEN;
constexpr int MLP_OFF_B2 = MLP_OFF_W2 + MLP_HIDDEN * MLP_HIDDEN;
constexpr int MLP_OFF_W3 = MLP_OFF_B2 + MLP_HIDDEN;
constexpr int MLP_OFF_B3 = MLP_OFF_W3 + MLP_NOUT * MLP_HIDDEN;
constexpr int MLP_NPARAM = MLP_OFF_B3 + MLP_NOUT;
constexpr int MLP_CAP = 4096;  // batch rows at most

struct Mlp {
    float *theta = nullptr, *grad = nullptr, *adam_m = nullptr, *adam_v = nullptr;  // [MLP_NPARAM]
    __nv_bfloat16 *W1b = nullptr, *W2b = nullptr, *W3b = nullptr;                   // BF16 operand copies
    __nv_bfloat16 *X = nullptr, *H1 = nullptr, *H2 = nullptr, *dZ1 = nullptr, *dZ2 = nullptr, *dYb = nullptr;
    float *Y = nullptr, *dY = nullptr;                // [cap][16]
    double *loss_part = nullptr, *loss = nullptr;     // loss[0]: last batch, loss[1]: accumulator
    double *dirs = nullptr;  // [96][3] unit vectors of the shell points
    int cap = 0;
    long long t = 0;  // Adam steps taken
    bool fault_no_commit = false;  // host-set fault injection (lbm_inject_fault)
};
cudaError_t mlp_alloc(Mlp &m, int cap);
void mlp_free(Mlp &m);
void mlp_refresh(const Mlp &m, cudaStream_t st);
// outputs m.Y [n][16] (6 used) for device inputs X [n][387]
cudaError_t mlp_forward(const Mlp &m, const float *X, int n, unsigned *status, cudaStream_t st);
// loss and gradient of the rows idx[row0 + r] (or row0 + r), r < n, of X [*][387]
// and T [*][6]; the loss is added to *acc where given
cudaError_t mlp_gradient(const Mlp &m, const float *X, const float *T, const long long *idx, long long row0, int n,
                         double *acc, unsigned *status, cudaStream_t st);
void mlp_adam(Mlp &m, double lr, cudaStream_t st);
template <class S>
void launch_shell_features(const Lattice &L, const Mlp &m, int p0, int np, float *feat, cudaStream_t st);
template <class S>
void launch_surrogate_forces(const Lattice &L, const Mlp &m, float *feat, cudaStream_t st, long long *launches,
                             const Marker &mk);
template <class S>
void launch_init_fields(const Lattice &L, int cur, int inst, long long N, const double *phi, const double *rho,
                        const double *u, const double *pops, cudaStream_t st);
template <class S>
void launch_read_fields(const Lattice &L, int cur, int inst, long long N, unsigned mask, double *out,
                        cudaStream_t st);
template <class S>
void launch_mass_sums(const Lattice &L, int cur, int inst, long long N, double *partial, int nblk, double *out,
                      cudaStream_t st);
void launch_boundary_full(const Lattice &L, int inst, long long N, cudaStream_t st);
// a static boundary list, in node order: mode 0 static solid nodes with a
// non-static neighbour, mode 1 non-static nodes with a static solid
// neighbour.  Count: blocks[b] entries of block b (static_bound_blocks of
// them), then offs[b] entries before it, offs[nblocks] all; fill after that.
long long static_bound_blocks(const Lattice &L);
void launch_static_count(const Lattice &L, int *blocks, long long *offs, int mode, cudaStream_t st);
void launch_static_fill(const Lattice &L, const long long *offs, long long *list, int mode, cudaStream_t st);
// solid marks of every node's gradient record (FP32 and FP64 storage)
template <class S>
void launch_mark_solid(const Lattice &L, cudaStream_t st);
void launch_mark_particles(const Lattice &L, cudaStream_t st);
// the first step's particle lists
void launch_first_lists(const Lattice &L, cudaStream_t st);

}  // namespace lbmg
