// Fluid update of one coupled time step (Sec. IV of arXiv 2505.10171).
//
// Per node: pull streaming with bounce-back -> order parameter phi -> phi on
// solid nodes next to fluid (w-weighted fluid mean) -> isotropic grad(phi)
// with the geometric wetting rotation (Sec. V E) -> regularised normal and its
// divergence (curvature) -> CSF + body force -> MRT with Guo forcing, evaluated
// in its two-relaxation-time form -> recolouring -> write.
//
// Kernels of a step: k_phi (z-marching tiles; narrow domains: k_phi_nodes) stores phi;
// the solid-phi fill over the listed static solid nodes and the step's list
// of particle-surface solid nodes; k_gradcurv (z-marching tiles: gradient,
// wetting, normal, curvature; FP64 and small grids: k_grad_nodes and
// k_curv_nodes); k_collide (or k_collide2).  Nodes next
// to a solid go to the boundary pass k_phi_bound and, in 16-bit storage, to
// k_collide_bound, which run beside the bulk kernels on a second stream.
//
// The state between steps is the total offsets F* (pop[cur]) with one colour
// record per node: phi (the order parameter its collision used) and b n (the
// recolouring amplitude times the normal).  The order-parameter pass rebuilds
// each pulled colour offset G_i from its source node's record
// (lbm_internal.cuh); the collision needs the colour offsets only through phi.
// Storage type S in {double, float, __half, __nv_bfloat16}; arithmetic in
// double for S = double and float otherwise.
#include <algorithm>
#include <cmath>

#include "lbm_node.cuh"

// Boundary passes, which run beside the bulk kernels: CTAs of 64 threads
// (FP64: one warp), so that a short list reaches many SMs (and FP64 pipes); 4
// (8) times this many per SM
template <class S>
constexpr int BOUND_THREADS = sizeof(S) == 8 ? 32 : 64;
#ifndef LBM_BOUND_MINB
#define LBM_BOUND_MINB 2
#endif
// CTAs of 256 threads per SM of the one-node collision.  FP32 storage: 5 (48
// registers, no spill), 119 us per 256x128x128 launch, 6.6 TB/s of the 188 bytes
// a node that it moves; 4 (64) 125 us.  16-bit storage: 4 (64 registers), as the
// gathered form spills with 48
#ifndef LBM_COLLIDE_MINB
#define LBM_COLLIDE_MINB 4
#endif
#ifndef LBM_COLLIDE_MINB_F32
#define LBM_COLLIDE_MINB_F32 5
#endif

namespace lbmg {

// ---------------------------------------------------------------------------
// bulk kernels over all nodes, list kernels over the nodes next to solids
// ---------------------------------------------------------------------------
// a mod n in [0, n): the in-range and one-period cases without a division
__device__ __forceinline__ int wrap_any(int a, int n)
{
    if (a >= 0 && a < n) return a;
    if (a < 0 && a >= -n) return a + n;
    if (a >= n && a < 2 * n) return a - n;
    a %= n;
    return a < 0 ? a + n : a;
}

// place of the in-plane source (x - dx, y - dy), dx or dy 0, among five
__host__ __device__ constexpr int five(int dx, int dy)
{
    return dx < 0 ? 1 : (dx > 0 ? 2 : (dy < 0 ? 3 : (dy > 0 ? 4 : 0)));
}

// ---------------------------------------------------------------------------
// order parameter of the fluid nodes none of whose neighbours is solid (the
// boundary pass k_phi_bound does the others)
// ---------------------------------------------------------------------------
// phi = sum_i w_i G_i / (1 + sum_i w_i F_i) of the streamed offsets, the
// colour offset pulled along direction i rebuilt from its source's record:
//   G_i = p_s (1 + F_i) + (c_i . a_s)/|c_i|,  s = x - c_i.
// Each record is wanted by 19 nodes.  A CTA owns a PH_TX x PH_TY column tile and
// marches through a chunk of z-planes; a plane's records (1-node halo) are
// staged once in shared memory, and every thread takes from each plane its nine
// p and the plane's sums of a: with
//   E = a0(x-1) - a0(x+1) + a1(y-1) - a1(y+1),  V = a2/18 + k (sum of a2 at the
//   four neighbours),  D the diagonal differences,  k = 1/(36 sqrt 2),
// the plane adds E/18 + k D to its own nodes' sum, k E + V to those above and
// k E - V to those below: 26 scalar reads a node instead of 19 16-byte ones.
// FP32 storage sums direction by direction (BY_DIRECTION): there a staged node
// holds the nine values that its record gives along the directions, a_k and
// (a_k +- a_l)/sqrt 2, formed once instead of by every node that pulls them, in
// a ring of three or four planes, and the 18 values and 19 p of a node are read
// where they are wanted: with p and the plane below carried in registers
// (80, spilling) the pass took 111 us on 256x128x128 and 347 on 64 x 96x48x48,
// with nothing carried (72) 94 and 285.
// The 19 pulled offsets of the next plane are loaded as soon as this plane's
// are used, so that they are in flight for a whole iteration.
// Bound by the latency of those loads (96 bytes a node FP32, 58 of 16-bit
// offsets; 24 resident warps per SM, half the issue slots used): 64 x 96x48x48
// FP32 472 -> 284 us (4.8 TB/s), 96-domain FP16 sweep 4297 -> 2692 us,
// 256x128x128 107 -> 93 us (FP16 92 -> 83: two waves of CTAs and little more),
// against the form that loaded every record where it was wanted.  Three CTAs
// per SM (80 registers); two 104 to 119 us, four (64, spilling) 213 (by
// direction 114 and 114).
constexpr int PH_TX = 32, PH_TY = 8;
#ifndef LBM_PHI_MINB
#define LBM_PHI_MINB 3
#endif

// direction i as one of the values +-a_k, +-(a_k +- a_l)/sqrt 2 that it pulls
// from its own plane (four) or a neighbouring one (five): which, and whether
// with the positive sign
__host__ __device__ constexpr int dir_along(int i)
{
    if (cz(i) == 0) return csq(i) == 1 ? (cx(i) ? 0 : 1) : (cx(i) == cy(i) ? 2 : 3);
    if (csq(i) == 1) return 0;
    return cx(i) ? (cx(i) == cz(i) ? 1 : 2) : (cy(i) == cz(i) ? 3 : 4);
}
__host__ __device__ constexpr bool dir_forward(int i)
{
    return cx(i) ? cx(i) > 0 : (cy(i) ? cy(i) > 0 : cz(i) > 0);
}

template <class S>
__global__ void __launch_bounds__(PH_TX *PH_TY, sizeof(S) == 8 ? 1 : LBM_PHI_MINB)
    k_phi(Lattice L, int cur)
{
    using R = typename Store<S>::real;
    constexpr int NT = PH_TX * PH_TY, PW = PH_TX + 2, PN = PW * (PH_TY + 2), PER = (PN + NT - 1) / NT;
    constexpr bool DIR = BY_DIRECTION<S>;
    // staged planes, a ring each: p and a_0, a_1, a_2; by direction p, what nodes
    // of the same plane pull (a_0, a_1, (a_0 +- a_1)/sqrt 2) and what those of the
    // planes beside it do (a_2, (a_0 +- a_2)/sqrt 2, (a_1 +- a_2)/sqrt 2)
    constexpr int SLOTS = DIR ? 4 : 2;
    __shared__ R recS[SLOTS][DIR ? 1 : 4][PN];
    __shared__ R sameS[DIR ? 3 : 1][DIR ? 4 : 1][DIR ? PN : 1], sideS[DIR ? 4 : 1][DIR ? 5 : 1][DIR ? PN : 1];
    pdl_trigger();  // the gradient pass may be scheduled as this grid drains

    const long long item = blockIdx.x;
    int lo = 0, hi = L.n_inst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (L.inst[mid].ph_item_start <= item) lo = mid;
        else hi = mid - 1;
    }
    const InstDev &I = L.inst[lo];
    const int loc = (int)(item - I.ph_item_start);
    const int t2 = I.fd_ph_nchunks.div(loc);
    const int chunk = loc - t2 * I.ph_nchunks;
    const int ty = I.fd_ph_tiles_x.div(t2);
    const int x0 = (t2 - ty * I.ph_tiles_x) * PH_TX, y0 = ty * PH_TY;
    const int z0 = chunk * I.ph_zc, zc = min(I.ph_zc, I.nz - z0);
    const int nx = I.nx, ny = I.ny, nz = I.nz, N = I.pstride, plane = nx * ny;
    const S *const pf = Pop<S>(L.pop[cur], I).f;
    const ColRec<R> *const rec = (const ColRec<R> *)L.col + I.node_off;
    const uint8_t *const fli = L.flags + I.node_off;
    R *const phi = (R *)L.phi + I.node_off;
    const int tid = threadIdx.x, lx = tid % PH_TX, ly = tid / PH_TX;
    const int gx = x0 + lx, gy = y0 + ly;
    const bool inside = gx < nx && gy < ny;
    const int c = (ly + 1) * PW + lx + 1;

    // in-plane offsets of the sources (x - dx, y - dy)
    int off[3][3];
    {
        const int X[3] = {wrap_any(gx + 1, nx), wrap_any(gx, nx), wrap_any(gx - 1, nx)};
        const int Y[3] = {wrap_any(gy + 1, ny) * nx, wrap_any(gy, ny) * nx, wrap_any(gy - 1, ny) * nx};
#pragma unroll
        for (int b = 0; b < 3; b++)
#pragma unroll
            for (int a = 0; a < 3; a++) off[b][a] = Y[b] + X[a];
    }
    int roff[PER];
#pragma unroll
    for (int q = 0; q < PER; q++) {
        const int r = min(tid + q * NT, PN - 1);
        roff[q] = wrap_any(y0 - 1 + r / PW, ny) * nx + wrap_any(x0 - 1 + r % PW, nx);
    }
    ColRec<R> rv[PER];
    int zr = wrap_any(z0 - 1, nz);  // plane whose records are fetched next
    auto fetch = [&]() {
        const int zo = zr * plane;
        zr = zr == nz - 1 ? 0 : zr + 1;
#pragma unroll
        for (int q = 0; q < PER; q++) rv[q] = rec[zo + roff[q]];
    };
    int at1 = 2, at0 = 0, atn = 1;  // sameS: slots of the planes j - 1, j and j + 1
    auto store = [&](int j, int same) {
#pragma unroll
        for (int q = 0; q < PER; q++) {
            const int r = tid + q * NT;
            if (r < PN) {
                const int slot = j & (SLOTS - 1);
                const R a0 = rv[q].a0, a1 = rv[q].a1, a2 = rv[q].a2;
                recS[slot][0][r] = rv[q].p;
                if constexpr (DIR) {
                    const R h = R(0.70710678118654752440);
                    sameS[same][0][r] = a0;
                    sameS[same][1][r] = a1;
                    sameS[same][2][r] = mul_rn(h, add_rn(a0, a1));
                    sameS[same][3][r] = mul_rn(h, sub_rn(a0, a1));
                    sideS[slot][0][r] = a2;
                    sideS[slot][1][r] = mul_rn(h, add_rn(a0, a2));
                    sideS[slot][2][r] = mul_rn(h, sub_rn(a0, a2));
                    sideS[slot][3][r] = mul_rn(h, add_rn(a1, a2));
                    sideS[slot][4][r] = mul_rn(h, sub_rn(a1, a2));
                } else {
                    recS[slot][1][r] = a0;
                    recS[slot][2][r] = a1;
                    recS[slot][3][r] = a2;
                }
            }
        }
    };
    // the pulled offsets and flags of target plane zt, in their stored type
    S F[Q];
    uint8_t fl = 0;
    auto pull = [&](int zt) {
        const int zo[3] = {(zt == nz - 1 ? 0 : zt + 1) * plane, zt * plane, (zt == 0 ? nz - 1 : zt - 1) * plane};
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const S *const base = pf + (i * N + zo[cz(i) + 1]);
            F[i] = pop_load_beside_writes(base + off[cy(i) + 1][cx(i) + 1]);
        }
        fl = fli[zt * plane + off[1][1]];
    };
    fetch();
    store(0, at0);
    pull(z0);
    __syncthreads();

    const R k18 = R(1.0 / 18.0), kd = R(0.70710678118654752440 / 36.0);
    // gathered sums: p of the last plane ([y][x], sources of the target as off) and
    // the five of the plane before that a target above pulls from; sums of a to come
    R p1[3][3], p2[5];
    R above = 0, own = 0;  // of the plane after the last: what is below gives; of the last plane: all but its plane above
#pragma unroll
    for (int b = 0; b < 3; b++)
#pragma unroll
        for (int a = 0; a < 3; a++) p1[b][a] = 0;
#pragma unroll
    for (int a = 0; a < 5; a++) p2[a] = 0;
    for (int j = 0; j < zc + 2; j++) {
        // plane z0-1+j is staged; the target is plane z0-2+j
        if (j < zc + 1) fetch();
        R p0[3][3], E = 0, V = 0, D = 0;
        if constexpr (!DIR) {
            const R *s = recS[j & 1][0] + c;
#pragma unroll
            for (int b = 0; b < 3; b++)
#pragma unroll
                for (int a = 0; a < 3; a++) p0[b][a] = s[(1 - b) * PW + 1 - a];
            const R *a0 = s + PN, *a1 = a0 + PN, *a2 = a1 + PN;
            E = (a0[-1] - a0[1]) + (a1[-PW] - a1[PW]);
            V = k18 * a2[0] + kd * ((a2[-1] + a2[1]) + (a2[-PW] + a2[PW]));
            D = ((a0[-PW - 1] + a1[-PW - 1]) - (a0[PW + 1] + a1[PW + 1])) +
                ((a0[PW - 1] - a1[PW - 1]) - (a0[-PW + 1] - a1[-PW + 1]));
        }
        if (j >= 2) {
            R f[Q];
#pragma unroll
            for (int i = 0; i < Q; i++) f[i] = Store<S>::cvt(F[i]);
            const int zt = z0 - 2 + j;
            const bool write = inside && !(fl & (OWNER_MASK | BOUND_BIT));  // fluid, no solid beside it
            if (j < zc + 1) pull(zt + 1);
            R num, den;
            if constexpr (DIR) {
                // G_i = p (1 + F_i) + (c_i . a)/|c_i|, then the two sums over i
                R sG = 0, sF = 0;
#pragma unroll
                for (int i = 0; i < Q; i++) {
                    const int at = c - cy(i) * PW - cx(i), slot = (j - 1 - cz(i)) & 3, k = dir_along(i);
                    const R p = recS[slot][0][at], e = add_rn(R(1), f[i]);
                    R G = mul_rn(p, e);
                    if (i > 0) {
                        const R t = cz(i) == 0 ? sameS[at1][k][at] : sideS[slot][k][at];
                        G = fma_rn(p, e, dir_forward(i) ? t : -t);
                    }
                    sF = fma_rn(wgt<R>(i), f[i], sF);
                    sG = fma_rn(wgt<R>(i), G, sG);
                }
                num = sG;
                den = add_rn(R(1), sF);
            } else {
                // p (1 + F) and F summed by weight: rest, axes, diagonals
                const R T = own + (kd * E - V);
                R ga = 0, gd = 0, fa = 0, fd = 0;
#pragma unroll
                for (int i = 1; i < Q; i++) {
                    const R p = cz(i) == 0 ? p1[cy(i) + 1][cx(i) + 1]
                                           : (cz(i) < 0 ? p0[cy(i) + 1][cx(i) + 1] : p2[five(cx(i), cy(i))]);
                    const R g = p + p * f[i];
                    if (csq(i) == 1) {
                        ga += g;
                        fa += f[i];
                    } else {
                        gd += g;
                        fd += f[i];
                    }
                }
                num = R(1.0 / 3.0) * (p1[1][1] + p1[1][1] * f[0]) + (k18 * ga + (R(1.0 / 36.0) * gd + T));
                den = R(1) + (R(1.0 / 3.0) * f[0] + (k18 * fa + R(1.0 / 36.0) * fd));
            }
            if (write) phi[zt * plane + off[1][1]] = num / den;
        }
        if constexpr (!DIR) {
            own = above + (k18 * E + kd * D);
            above = kd * E + V;
            p2[0] = p1[1][1];
            p2[1] = p1[1][0];
            p2[2] = p1[1][2];
            p2[3] = p1[0][1];
            p2[4] = p1[2][1];
#pragma unroll
            for (int b = 0; b < 3; b++)
#pragma unroll
                for (int a = 0; a < 3; a++) p1[b][a] = p0[b][a];
        }
        if (j < zc + 1) store(j + 1, atn);
        __syncthreads();
        const int last = at1;
        at1 = at0;
        at0 = atn;
        atn = last;
    }
}

// ---------------------------------------------------------------------------
// boundary lists
// ---------------------------------------------------------------------------
// instance of global node g (binary search over the node offsets)
__device__ __forceinline__ int inst_of_node(const Lattice &L, long long g)
{
    int lo = 0, hi = L.n_inst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (L.inst[mid].node_off <= g) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// static solid nodes with a neighbour that is not static solid (mode 0), or
// the other way round (mode 1): whether global node g is one, and its entry
__device__ __forceinline__ bool static_bound(const Lattice &L, long long g, int mode, long long *entry)
{
    if (g >= L.Ntot || own_static(L.flags[g] & OWNER_MASK) != (mode == 0)) return false;
    const int k = inst_of_node(L, g);
    const InstDev &I = L.inst[k];
    const int n = (int)(g - I.node_off);
    const int x = n % I.nx, y = (n / I.nx) % I.ny, z = n / (I.nx * I.ny);
    Nbr nb;
    nb.init(x, y, z, I.nx, I.ny, I.nz);
    const uint8_t *fli = L.flags + I.node_off;
    bool hit = false;
#pragma unroll
    for (int i = 1; i < Q; i++) hit |= own_static(fli[nb.at(cx(i), cy(i), cz(i))] & OWNER_MASK) != (mode == 0);
    *entry = list_entry(k, n);
    return hit;
}

// The lists are in node order: consecutive threads of the passes over them
// then work on nodes of one row, whose loads share sectors.  (Appended with one
// atomic per node, 64x64x1024 tube: order-parameter boundary pass 98 us and
// collision boundary pass 187 us for 300 000 nodes; in order 88 us, and the
// latter is gone.)
constexpr int SB_THREADS = 256;
__global__ void __launch_bounds__(SB_THREADS) k_static_count(Lattice L, int mode, int *blocks)
{
    long long e;
    const int c = __syncthreads_count(static_bound(L, (long long)blockIdx.x * SB_THREADS + threadIdx.x, mode, &e));
    if (threadIdx.x == 0) blocks[blockIdx.x] = c;
}

// offs[b] = sum of blocks[0..b), offs[nb] = sum of all: one CTA, a run of
// consecutive blocks per thread
__global__ void __launch_bounds__(1024) k_static_scan(const int *blocks, long long nb, long long *offs)
{
    __shared__ long long sh[1024];
    const int t = threadIdx.x;
    const long long per = (nb + 1023) / 1024, b0 = min(nb, t * per), b1 = min(nb, b0 + per);
    long long s = 0;
    for (long long b = b0; b < b1; b++) s += blocks[b];
    sh[t] = s;
    __syncthreads();
    for (int d = 1; d < 1024; d <<= 1) {
        const long long v = t >= d ? sh[t - d] : 0;
        __syncthreads();
        sh[t] += v;
        __syncthreads();
    }
    long long o = sh[t] - s;
    for (long long b = b0; b < b1; b++) {
        offs[b] = o;
        o += blocks[b];
    }
    if (t == 1023) offs[nb] = sh[1023];
}

__global__ void __launch_bounds__(SB_THREADS) k_static_fill(Lattice L, int mode, const long long *offs, long long *list)
{
    __shared__ int warps[SB_THREADS / 32];
    long long e = 0;
    const bool hit = static_bound(L, (long long)blockIdx.x * SB_THREADS + threadIdx.x, mode, &e);
    const unsigned m = __ballot_sync(0xffffffffu, hit);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) warps[wid] = __popc(m);
    __syncthreads();
    if (!hit) return;
    long long o = offs[blockIdx.x] + __popc(m & ((1u << lane) - 1u));
    for (int w = 0; w < wid; w++) o += warps[w];
    list[o] = e;
}

long long static_bound_blocks(const Lattice &L) { return (L.Ntot + SB_THREADS - 1) / SB_THREADS; }
void launch_static_count(const Lattice &L, int *blocks, long long *offs, int mode, cudaStream_t st)
{
    const long long nb = static_bound_blocks(L);
    k_static_count<<<(unsigned)nb, SB_THREADS, 0, st>>>(L, mode, blocks);
    k_static_scan<<<1, 1024, 0, st>>>(blocks, nb, offs);
}
void launch_static_fill(const Lattice &L, const long long *offs, long long *list, int mode, cudaStream_t st)
{
    k_static_fill<<<(unsigned)static_bound_blocks(L), SB_THREADS, 0, st>>>(L, mode, offs, list);
}

template <class R>
__global__ void __launch_bounds__(256) k_mark_solid(Lattice L)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < L.Ntot && (L.flags[g] & OWNER_MASK) != OWN_FLUID) set_solid_mark(((GradRec<R> *)L.grad)[g]);
}
template <class S>
void launch_mark_solid(const Lattice &L, cudaStream_t st)
{
    k_mark_solid<typename Store<S>::real><<<(unsigned)((L.Ntot + 255) / 256), 256, 0, st>>>(L);
}

// node of a list entry
__device__ __forceinline__ const InstDev &list_node(const Lattice &L, long long e, int *n, int *x, int *y, int *z)
{
    const InstDev &I = L.inst[e >> 32];
    *n = (int)(unsigned)e;
    const int row = I.fd_nx.div(*n);
    *x = *n - row * I.nx;
    *z = I.fd_ny.div(row);
    *y = row - *z * I.ny;
    return I;
}

// The boundary passes: fluid nodes next to a solid, with the bounce-back pull
// (Sec. V A), grid-stride over the listed particle nodes and the static list
// of nodes next to walls; a node listed twice (two cubes, or a cube and the
// static list) is written twice with the same value.
//
// The order-parameter pass forms every bounced offset F_i; FP32 and FP64
// storage keep it in slot i of the solid source itself, which no other node
// pulls and no kernel reads otherwise, so that the bulk collision pulls these
// nodes like all others and has no boundary pass.  (16-bit storage would round
// the offset there; its collision takes these nodes in k_collide_bound.)  The
// bulk order-parameter pass may load such a slot while it is written: for a
// node next to a solid, whose value it drops (pop_load_beside_writes).
template <class S>
__device__ __forceinline__ void phi_bound_node(const Lattice &L, int cur, long long e)
{
    using R = typename Store<S>::real;
    int n, x, y, z;
    const InstDev &I = list_node(L, e, &n, &x, &y, &z);
    const uint8_t *fli = L.flags + I.node_off;
    const uint8_t fl = fli[n];
    const Pop<S> in(L.pop[cur], I);
    const ColourOf<S> C(L, I);
    Nbr nb;
    nb.init(x, y, z, I.nx, I.ny, I.nz);
    int own[Q];
    R F[Q], sF = 0;
    gather_links<S>(I, L.parts, fli, nb, in, n, x, y, z, own, F);
    const R sG = gather_colour<S>(nb, C, n, own, F);
    if ((fl & OWNER_MASK) != OWN_FLUID || !(fl & BOUND_BIT)) return;  // covered by a particle
#pragma unroll
    for (int i = 0; i < Q; i++) sF += wgt<R>(i) * F[i];
    ((R *)L.phi)[I.node_off + n] = sG / (R(1) + sF);
    if (BOUNCE_IN_SLOTS<S>) {
#pragma unroll
        for (int i = 1; i < Q; i++)
            if (own[i] != OWN_FLUID) in.setF(i, nb.at(-cx(i), -cy(i), -cz(i)), F[i]);
    }
}

template <class S>
__global__ void __launch_bounds__(BOUND_THREADS<S>, sizeof(S) == 8 ? 8 : 4 * LBM_BOUND_MINB) k_phi_bound(Lattice L, int cur)
{
    const long long npb = L.n_parts ? (long long)L.list_n[LIST_FLUID] : 0;
    const long long total = npb + L.n_static_bfl;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x)
        phi_bound_node<S>(L, cur, t < npb ? L.pbl[t] : L.static_bfl[t - npb]);
}

template <class S>
__device__ __forceinline__ void collide_bound_node(const Lattice &L, int cur, long long e)
{
    using R = typename Store<S>::real;
    int n, x, y, z;
    const InstDev &I = list_node(L, e, &n, &x, &y, &z);
    const uint8_t *fli = L.flags + I.node_off;
    const long long g = I.node_off + n;
    const uint8_t fl = fli[n];
    const Pop<S> in(L.pop[cur], I);
    const Pop<S> out(L.pop[cur ^ 1], I);
    const GradRec<R> gr = ((const GradRec<R> *)L.grad)[g];
    const R phi = ((const R *)L.phi)[g];
    R *U = I.store_u ? (R *)L.u + I.node_off : nullptr;
    Nbr nb;
    nb.init(x, y, z, I.nx, I.ny, I.nz);
    int own[Q];
    R F[Q];
    gather_links<S>(I, L.parts, fli, nb, in, n, x, y, z, own, F);
    if ((fl & OWNER_MASK) != OWN_FLUID || !(fl & BOUND_BIT)) return;
    FluidPar<R> P;
    load_par(I, P);
    collide_store_phi<S>(P, F, phi, gr, out, n, col_slot<S>(L, g), U, L.Ntot, L.status);
}

template <class S>
__global__ void __launch_bounds__(BOUND_THREADS<S>, 4 * LBM_BOUND_MINB) k_collide_bound(Lattice L, int cur)
{
    const long long npb = L.n_parts ? (long long)L.list_n[LIST_FLUID] : 0;
    const long long total = npb + L.n_static_bfl;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x)
        collide_bound_node<S>(L, cur, t < npb ? L.pbl[t] : L.static_bfl[t - npb]);
}

// phi of the solid nodes next to fluid, the listed static ones and the step's
// list of particle-surface ones: the w-weighted mean over their fluid
// neighbours
template <class R>
__global__ void __launch_bounds__(PART_THREADS) k_solidphi(Lattice L)
{
    const long long nps = L.n_parts ? (long long)L.list_n[LIST_SOLID] : 0;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < nps + L.n_static;
         t += (long long)gridDim.x * blockDim.x) {
        int n, x, y, z;
        const InstDev &I = list_node(L, t < nps ? L.psl[t] : L.static_list[t - nps], &n, &x, &y, &z);
        const uint8_t *fli = L.flags + I.node_off;
        R *ph = (R *)L.phi + I.node_off;
        Nbr nb;
        nb.init(x, y, z, I.nx, I.ny, I.nz);
        const uint8_t fl = fli[n];
        int own[Q];
        R p[Q];
#pragma unroll
        for (int i = 1; i < Q; i++) {
            const int s = nb.at(cx(i), cy(i), cz(i));
            own[i] = fli[s];
            p[i] = ph[s];
        }
        if ((fl & OWNER_MASK) == OWN_FLUID || !(fl & BOUND_BIT)) continue;
        R sw = 0, sp = 0;
#pragma unroll
        for (int i = 1; i < Q; i++) {
            if ((own[i] & OWNER_MASK) != OWN_FLUID) continue;
            sw += wgt<R>(i);
            sp += wgt<R>(i) * p[i];
        }
        ph[n] = sw > R(0) ? sp / sw : R(0);
    }
}

template <class S>
__device__ __forceinline__ void collide_body(const Lattice &L, const InstDev &I, int cur, int n, int x, int y, int z)
{
    using R = typename Store<S>::real;
    const long long g = I.node_off + n;
    const Pop<S> in(L.pop[cur], I);
    const Pop<S> out(L.pop[cur ^ 1], I);
    // every load is issued before the node's kind is tested
    const uint8_t fl = BOUNCE_IN_SLOTS<S> ? 0 : L.flags[g];
    const GradRec<R> gr = ((const GradRec<R> *)L.grad)[g];
    const R phi = ((const R *)L.phi)[g];
    Nbr nb;
    nb.init(x, y, z, I.nx, I.ny, I.nz);
    R F[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) F[i] = in.F(i, nb.at(-cx(i), -cy(i), -cz(i)));
#pragma unroll
    for (int i = 0; i < Q; i++) keep(F[i]);
    R *U = I.store_u ? (R *)L.u + I.node_off : nullptr;
    if (BOUNCE_IN_SLOTS<S> ? solid_mark(gr) : (fl & OWNER_MASK) != OWN_FLUID) {
        if (U) { U[n] = 0; U[L.Ntot + n] = 0; U[2 * L.Ntot + n] = 0; }
        return;
    }
    // 16-bit storage: nodes next to a solid belong to the boundary pass
    if (fl & BOUND_BIT) return;
    FluidPar<R> P;
    load_par(I, P);
    collide_store_phi<S>(P, F, phi, gr, out, n, col_slot<S>(L, g), U, L.Ntot, L.status);
}

// Node pairs (x even, x + 1) of one row per thread, for 16-bit storage: the
// pulls along directions with c_x = 0 are one 32-bit load of the pair, every
// output a pair store (half2 or bfloat162), and the arithmetic handles both
// nodes per instruction (F2), which halves what binds this kernel: issue slots.
// Each node's arithmetic is that of collide_store_phi (which may leave other
// multiply-adds fused, so the results agree to rounding); a node of the pair
// that the bulk kernel skips (solid, next to a solid) is computed but not
// written.
template <class S>
__device__ __forceinline__ void collide_body2(const Lattice &L, const InstDev &I, int cur, int n, int x, int y, int z)
{
    using R = typename Store<S>::real;
    using FT = typename Pop<S>::FT;
    static_assert(sizeof(FT) == 2 && sizeof(R) == 4, "pair kernel: 16-bit total offsets, FP32 arithmetic");
    const long long g = I.node_off + n;  // even
    const Pop<S> in(L.pop[cur], I);
    const Pop<S> out(L.pop[cur ^ 1], I);
    const int N = in.N;
    const uint8_t fl0 = L.flags[g], fl1 = L.flags[g + 1];
    const long long Nt = L.Ntot;
    const GradRec<R> grA = ((const GradRec<R> *)L.grad)[g], grB = ((const GradRec<R> *)L.grad)[g + 1];
    const float2 pv = *reinterpret_cast<const float2 *>((const R *)L.phi + g);
    Nbr nb;
    nb.init(x, y, z, I.nx, I.ny, I.nz);
    const int xp2 = x + 2 == I.nx ? 0 : x + 2;
    F2 F[Q];
    {
        R F0[Q], F1[Q];
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const FT *row = in.f + i * N + nb.ZO[1 - cz(i)] + nb.YO[1 - cy(i)];
            if (cx(i) == 0) {
                ld_pair(row + x, F0[i], F1[i]);
            } else if (cx(i) == 1) {
                F0[i] = Store<FT>::ld(row + nb.X[0]);
                F1[i] = Store<FT>::ld(row + x);
            } else {
                F0[i] = Store<FT>::ld(row + x + 1);
                F1[i] = Store<FT>::ld(row + xp2);
            }
        }
#pragma unroll
        for (int i = 0; i < Q; i++) {
            keep(F0[i]);
            keep(F1[i]);
            F[i] = f2(F0[i], F1[i]);
        }
    }
    const bool fluid0 = (fl0 & OWNER_MASK) == OWN_FLUID, fluid1 = (fl1 & OWNER_MASK) == OWN_FLUID;
    const bool a0 = fluid0 && !(fl0 & BOUND_BIT), a1 = fluid1 && !(fl1 & BOUND_BIT);
    R *U = I.store_u ? (R *)L.u + I.node_off : nullptr;
    if (U) {
        if (!fluid0) { U[n] = 0; U[Nt + n] = 0; U[2 * Nt + n] = 0; }
        if (!fluid1) { U[n + 1] = 0; U[Nt + n + 1] = 0; U[2 * Nt + n + 1] = 0; }
    }
    if (!a0 && !a1) return;
    FluidPar<R> P;
    load_par(I, P);
    const F2 gr[3] = {f2(grA.g0, grB.g0), f2(grA.g1, grB.g1), f2(grA.g2, grB.g2)};
    const Collision<F2> c = collide_setup(CollidePar<F2>(P), F, f2(pv.x, pv.y), gr, f2(grA.k, grB.k));
    float rA, rB, bA, bB;
    unpack(c.rr, rA, rB);
    unpack(c.bq, bA, bB);
    if ((a0 && (!(rA > R(0)) || !(pv.x == pv.x))) || (a1 && (!(rB > R(0)) || !(pv.y == pv.y))))
        atomicOr(L.status, ST_UNSTABLE);
    if (U) {
#pragma unroll
        for (int k = 0; k < 3; k++) {
            float uA, uB;
            unpack(c.u[k], uA, uB);
            if (a0) U[k * Nt + n] = uA;
            if (a1) U[k * Nt + n + 1] = uB;
        }
    }
    FT *const of = out.f + n;
    const bool both = a0 && a1;
    auto put = [&](FT *p, F2 v) {
        float v0, v1;
        unpack(v, v0, v1);
        if (both) {
            st_pair(p, v0, v1);
        } else if (a0) {
            Store<FT>::st(p, v0);
        } else {
            Store<FT>::st(p + 1, v1);
        }
    };
    if (a0) col_slot<S>(L, g).set(colour_record(bA, P.eps2, pv.x, grA.g0, grA.g1, grA.g2));
    if (a1) col_slot<S>(L, g + 1).set(colour_record(bB, P.eps2, pv.y, grB.g0, grB.g1, grB.g2));
    put(of, collide_rest(c, F[0]));
    PairLoop<R>::run([&](auto ic) {
        constexpr int i = decltype(ic)::value, ib = i + 9;
        F2 Fi, Fib;
        collide_pair<i>(c, F[i], F[ib], Fi, Fib);
        put(of + i * N, Fi);
        put(of + ib * N, Fib);
    });
}

// CTAs of 128 threads per SM the node-pair collision is compiled for: 4 (128
// registers, no spill); 5, 6 and 7 spill and took 3445, 3699 and 3703 us against
// 3393 on the 96-domain sweep.  With two scalar nodes per thread, the relaxation
// direction by direction and items of whole rows it was bound by issue and took
// 3915 us (36 x 200x90x36: 634 -> 545); now 4.8 TB/s.
#ifndef LBM_COLLIDE2_MINB
#define LBM_COLLIDE2_MINB 4
#endif
// Work items of the collision: consecutive nodes of an instance, whatever their
// rows (items of whole rows leave lanes idle wherever rows do not fill a CTA: 22%
// at nx = 200, 25% at 96).  FP64 items are small: its runs are bound by the
// FP64 pipes of the SMs they reach, and 224 CTAs of 240 nodes on 152 SMs took
// 66 us for 48x32x32; CTAs of 64 and a third fewer FP64 instructions 31.
template <class S>
constexpr int COLLIDE_NODES = sizeof(S) == 8 ? 64 : 256;

// the node of item `item` for thread offset j; false past the instance's end
__device__ __forceinline__ bool item_node(const Lattice &L, long long item, int per_item, int j, const InstDev **Ip,
                                          int *n, int *x, int *y, int *z)
{
    int lo = 0, hi = L.n_inst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (L.inst[mid].item_start <= item) lo = mid;
        else hi = mid - 1;
    }
    const InstDev &I = L.inst[lo];
    const int m = (int)(item - I.item_start) * per_item + j;
    if (m >= I.pstride) return false;
    const int row = I.fd_nx.div(m);
    *x = m - row * I.nx;
    *z = I.fd_ny.div(row);
    *y = row - *z * I.ny;
    *n = m;
    *Ip = &I;
    return true;
}

// The form without tiles, for domains that fill few of the tiles' lanes or planes:
// a node per thread, direction by direction, every record loaded where it is
// wanted.  Bound by the latency of those loads and by L1 (19 records of 16 bytes a
// node).  Marching against this form, FP32 (FP16), by the share of the tiles'
// work that is nodes, nx ny nz over 256 tiles nz + 2 planes: 0.25 (8x8x16384) 82
// and 34 us (70, 27); 0.33 (1024x1024x1) 49 and 35 (42, 27); 0.45 (34x34x1024) 58
// and 41 (50, 33); 0.47 (512 x 16^3) 102 and 85 (92, 84); 0.57 (42x42x1024) 70 and
// 57 (60, 52); 0.60 (64 x 40^3) 135 and 131 (117, 125); 0.75 (48x48x1024) 72 and 69
// (62, 65); 1 (256x128x128) 94 and 113 (82, 114).  FP64 keeps the tiles, which
// spare it instructions.
// Four CTAs per SM (64 registers); three 43 us on 34x34x1024, two 43.
constexpr int PN_NODES = 256;
constexpr double PN_SHARE = 0.58;
#ifndef LBM_PHI_NODES_MINB
#define LBM_PHI_NODES_MINB 4
#endif
template <class S>
__global__ void __launch_bounds__(PN_NODES, LBM_PHI_NODES_MINB) k_phi_nodes(Lattice L, int cur)
{
    using R = typename Store<S>::real;
    int lo = 0, hi = L.n_inst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (L.inst[mid].pn_item_start <= (long long)blockIdx.x) lo = mid;
        else hi = mid - 1;
    }
    const InstDev &I = L.inst[lo];
    const int n = (int)((long long)blockIdx.x - I.pn_item_start) * PN_NODES + (int)threadIdx.x;
    pdl_trigger();  // the gradient pass may be scheduled as this grid drains
    if (n >= I.pstride) return;
    const int row = I.fd_nx.div(n), z = I.fd_ny.div(row), x = n - row * I.nx, y = row - z * I.ny;
    Nbr nb;
    nb.init(x, y, z, I.nx, I.ny, I.nz);
    const Pop<S> in(L.pop[cur], I);
    const ColRec<R> *const rec = (const ColRec<R> *)L.col + I.node_off;
    const uint8_t fl = L.flags[I.node_off + n];
    R sF = 0, sG = 0;
#pragma unroll
    for (int i = 0; i < Q; i++) {
        const int s = nb.at(-cx(i), -cy(i), -cz(i));
        const R F = in.F_beside_writes(i, s), e = add_rn(R(1), F);
        const ColRec<R> r = rec[s];
        const R G = i ? fma_rn(r.p, e, col_rec(i, r)) : mul_rn(r.p, e);
        sF = fma_rn(wgt<R>(i), F, sF);
        sG = fma_rn(wgt<R>(i), G, sG);
    }
    R v = sG / add_rn(R(1), sF);
    keep(v);
    if (!(fl & (OWNER_MASK | BOUND_BIT))) ((R *)L.phi)[I.node_off + n] = v;
}

template <class S>
__global__ void __launch_bounds__(COLLIDE_NODES<S> / 2, LBM_COLLIDE2_MINB) k_collide2(Lattice L, int cur)
{
    const InstDev *I;
    int n, x, y, z;
    const bool have = item_node(L, blockIdx.x, COLLIDE_NODES<S>, 2 * (int)threadIdx.x, &I, &n, &x, &y, &z);
    pdl_wait();  // the gradient pass's grad(phi) and curvature
    if (have) collide_body2<S>(L, *I, cur, n, x, y, z);
}

template <class S>
__global__ void __launch_bounds__(COLLIDE_NODES<S>, sizeof(S) == 8 ? 4 : (sizeof(S) == 4 ? LBM_COLLIDE_MINB_F32 : LBM_COLLIDE_MINB)) k_collide(Lattice L, int cur)
{
    const InstDev *I;
    int n, x, y, z;
    const bool have = item_node(L, blockIdx.x, COLLIDE_NODES<S>, (int)threadIdx.x, &I, &n, &x, &y, &z);
    pdl_wait();  // the gradient pass's grad(phi) and curvature
    if (have) collide_body<S>(L, *I, cur, n, x, y, z);
}

// ---------------------------------------------------------------------------
// gradient, wetting, normal and curvature in one z-marching pass
// ---------------------------------------------------------------------------
// FP32 arithmetic: a CTA owns a GC_TX x (ROWS RP) column tile and a chunk of z-planes and
// marches through the chunk's planes of phi (2-node halo).  FP32 storage (DIR)
// takes both stencils direction by direction from the planes around a node, kept
// in two rings.  16-bit storage splits them into in-plane sums of one plane
// each: with X, Y the differences of the
// +-x and +-y neighbours, S the sum of the four, A and B the sum and difference
// of the two diagonal differences of a plane,
//   gx(z) = X/6 + A/12 + [X(z+1) + X(z-1)]/12,   gy alike with Y and B,
//   gz(z) = q(z+1) - q(z-1),  q = phi/6 + S/12,
// and the curvature is the same operator applied to the normal's components.
// So a plane is read from shared memory once and its sums are carried to the
// planes below and above in registers, instead of 18 + 30 reads of three
// stored planes.  Iteration j: gradient and normal of plane z0-3+j on the
// 1-halo tile (written to one of two normal planes), curvature of plane
// z0-5+j from the normals of the iteration before, and phi of plane z0-1+j
// into the plane ring; one barrier, which also tells whether any node of the
// plane carries a flag (most planes of most tiles do not: no flag is looked at
// then).  The first 32 ROWS threads own RP rows of one column each; further
// threads take the nodes around the tile, whose normals the curvature needs.
//
// Bound by the chain of a plane's iteration (shared-memory reads, the normal's
// inverse root, a barrier: 58% of the issue slots at 20 to 24 resident warps per
// SM), not by memory: 24 bytes a node, most of which stay in L2.  With the two
// rows in two-float instructions it executes a fifth fewer and takes as long
// (75.5 against 73 us on 256x128x128, 1720 against 1746 us in the sweep).  The
// form with three stored planes and 48 reads a node executed 14.2 warp
// instructions per node, this one 9.6: 96-domain sweep (1.5e8 nodes) 2796 -> 1738 us, 256x128x128
// 75 -> 73 us.  By direction the 48 reads stay: 64 x 96x48x48 254 -> 212 us by
// one barrier a plane instead of three and planes without flags passed by
// (184 with gathered sums), 256x128x128 75 -> 74 us.
constexpr int GC_TX = 32;

// the sums of the gradient carried from plane to plane for one column
template <class R>
struct GcColumn {
    R px = 0, py = 0, pz = 0;  // gradient of the last plane but for the plane above it
    R hx = 0, hy = 0, q = 0;   // X/12, Y/12 and q of the last plane
    // next plane: the rows y-1, y, y+1 of its 3 x 3 nodes; g receives the last plane's gradient
    __device__ __forceinline__ void advance(const R (&s)[3], const R (&c)[3], const R (&n)[3], R *g)
    {
        const R d1 = sub_rn(n[2], s[0]), d2 = sub_rn(s[2], n[0]);
        const R X = sub_rn(c[2], c[0]), Y = sub_rn(n[1], s[1]);
        const R hx1 = mul_rn(R(1.0 / 12.0), X), hy1 = mul_rn(R(1.0 / 12.0), Y);
        const R q1 =
            fma_rn(R(1.0 / 6.0), c[1], mul_rn(R(1.0 / 12.0), add_rn(add_rn(c[2], c[0]), add_rn(n[1], s[1]))));
        g[0] = add_rn(px, hx1);
        g[1] = add_rn(py, hy1);
        g[2] = add_rn(pz, q1);
        px = fma_rn(R(1.0 / 6.0), X, fma_rn(R(1.0 / 12.0), add_rn(d1, d2), hx));
        py = fma_rn(R(1.0 / 6.0), Y, fma_rn(R(1.0 / 12.0), sub_rn(d1, d2), hy));
        pz = -q;
        hx = hx1;
        hy = hy1;
        q = q1;
    }
};

template <class R>
__device__ __forceinline__ void load_row(const R *p, R (&v)[3])
{
    v[0] = p[-1];
    v[1] = p[0];
    v[2] = p[1];
}

// a particle of the instance as the wetting needs it, in shared memory: centre,
// radius, cos and sin of the contact angle
template <class R>
struct GcPart {
    R x[3], rad, c, s;
};

// a fluid node next to a solid (flag(i): flags of its neighbour i, part(p):
// particle p): the wetting rotation of its gradient g, and
// s = 3 sum w_i c_i over its solid neighbours, which take the node's own normal
// in the curvature (their share is n . s).  The outward solid normal and
// contact angle: the nearest particle surface if a neighbour belongs to a
// particle, otherwise the normalised -sum w_i c_i over substrate neighbours.
// A CTA's march waits for its slowest thread on every plane, so a surface
// must not cost a chain of memory round trips: the sums are integers (36 w_i
// is 2 or 1), the owners met are collected as a mask, and distances are taken
// only where two particles meet.  With the owners' particle records read from
// memory per direction the pass took 195 us instead of 75 on 256x128x128
// nodes with eight spheres.
// DIR: the substrate's sum in floating point, direction by direction, for nodes
// that the wetting turns only (the walls of a 64x64x1024 tube: the pass 119 us with
// it for every node, 93 so); returns a bit per solid neighbour, direction i at bit i.
template <bool DIR, class R, class Flag, class Part>
__device__ __forceinline__ unsigned gc_solid(const InstDev &I, const Part &part, const Flag &flag, R phi, int x, int y,
                                             int z, R *g, R *s)
{
    int all[3] = {0, 0, 0}, wall[3] = {0, 0, 0};
    R ws[3] = {0, 0, 0};
    unsigned solid = 0;
    unsigned long long met = 0;
    const R wet_max = sizeof(R) == 8 ? (R)I.wet_max : (R)I.f_wet_max;
    if constexpr (DIR) {
#pragma unroll
        for (int i = 1; i < Q; i++)
            if ((flag(i) & OWNER_MASK) != OWN_FLUID) solid |= 1u << i;
        if (!(fabs(phi) < wet_max)) return solid;
    }
#pragma unroll
    for (int i = 1; i < Q; i++) {
        const int own = flag(i) & OWNER_MASK;
        const int k = own == OWN_FLUID ? 0 : (csq(i) == 1 ? 2 : 1);
        const int kw = own == OWN_WALL ? k : 0;
        if constexpr (DIR) {
            const R w = kw ? wgt<R>(i) : R(0);
            if (cx(i)) ws[0] = sub_rn(ws[0], cx(i) * w);
            if (cy(i)) ws[1] = sub_rn(ws[1], cy(i) * w);
            if (cz(i)) ws[2] = sub_rn(ws[2], cz(i) * w);
        } else {
            if (cx(i)) { all[0] += cx(i) * k; wall[0] += cx(i) * kw; }
            if (cy(i)) { all[1] += cy(i) * k; wall[1] += cy(i) * kw; }
            if (cz(i)) { all[2] += cz(i) * k; wall[2] += cz(i) * kw; }
        }
        met |= 1ull << own;
    }
    if constexpr (!DIR)
        for (int a = 0; a < 3; a++) s[a] = R(1.0 / 12.0) * all[a];
    if (!DIR && !(fabs(phi) < wet_max)) return solid;
    met &= ~(1ull << OWN_FLUID | 1ull << OWN_WALL | 1ull << OWN_PRESS);  // a pressure face carries no contact angle
    R d[3] = {DIR ? ws[0] : R(-wall[0]), DIR ? ws[1] : R(-wall[1]), DIR ? ws[2] : R(-wall[2])};
    R cth = (R)I.cos_tw, sth = (R)I.sin_tw;
    if (met) {
        // lowest index first: it wins a tie
        R bestd = 0;
        bool first = true;
        do {
            const GcPart<R> &P = part(__ffsll((long long)met) - 1 - 2);
            met &= met - 1;
            R e[3];
            if (sizeof(R) == 8) {
                e[0] = (R)min_image(x - P.x[0], I.nx); e[1] = (R)min_image(y - P.x[1], I.ny);
                e[2] = (R)min_image(z - P.x[2], I.nz);
            } else {
                e[0] = (R)min_image_f((float)(x - P.x[0]), I.nx); e[1] = (R)min_image_f((float)(y - P.x[1]), I.ny);
                e[2] = (R)min_image_f((float)(z - P.x[2]), I.nz);
            }
            const R dist = first && !met ? R(0) : sqrt(e[0] * e[0] + e[1] * e[1] + e[2] * e[2]) - P.rad;
            if (first || dist < bestd) {
                bestd = dist;
                d[0] = e[0]; d[1] = e[1]; d[2] = e[2];
                cth = P.c;
                sth = P.s;
            }
            first = false;
        } while (met);
    }
    const R l = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    if (l == R(0)) return solid;
    const R ns[3] = {d[0] / l, d[1] / l, d[2] / l};
    wetting_rotate<R>(g, ns, cth, sth);
    return solid;
}

// The sums direction by direction.  at(dx, dy, dz): phi of that neighbour;
// gradient 3 sum_i w_i c_i phi
template <class R, class At>
__device__ __forceinline__ void dir_gradient(const At &at, R *g)
{
    g[0] = g[1] = g[2] = 0;
#pragma unroll
    for (int i = 1; i < Q; i++) {
        const R p = at(cx(i), cy(i), cz(i)), w = R(3) * wgt<R>(i);
        if (cx(i)) g[0] = fma_rn(cx(i) * w, p, g[0]);
        if (cy(i)) g[1] = fma_rn(cy(i) * w, p, g[1]);
        if (cz(i)) g[2] = fma_rn(cz(i) * w, p, g[2]);
    }
}

// nf(a, i): component a of the normal of neighbour i (the node's own normal where
// that is solid); curvature 3 sum_i w_i c_i . n over opposite pairs, as
// w_i c_i . (n_i - n_ib)
template <class R, class NF>
__device__ __forceinline__ R dir_curvature(const NF &nf)
{
    R k = 0;
#pragma unroll
    for (int i = 1; i <= 9; i++) {
        R t = 0;
        if (cx(i)) t = sub_rn(nf(0, i), nf(0, i + 9));
        if (cy(i)) {
            const R d = sub_rn(nf(1, i), nf(1, i + 9));
            t = cx(i) ? (cy(i) > 0 ? add_rn(t, d) : sub_rn(t, d)) : d;
        }
        if (cz(i)) {
            const R d = sub_rn(nf(2, i), nf(2, i + 9));
            t = cx(i) || cy(i) ? (cz(i) > 0 ? add_rn(t, d) : sub_rn(t, d)) : d;
        }
        k = fma_rn(wgt<R>(i), t, k);
    }
    return mul_rn(R(3), k);
}

// Threads of the pass.  Two rows per thread share most of their shared-memory
// reads (75 against 72 us with one on 256x128x128 nodes, but 1738 against
// 1993 us on the 96-domain sweep); 8 warps of own nodes beat 4 (80 and 1864 us)
// and 6 (82 and 1956 us).
// By direction a node reads the three planes around it for each sum (18 + 30
// values; two rows share few of them), one row a thread: 74 us on 256x128x128 and
// 212 on 64 x 96x48x48 (78 and 218 when two rows took 83 and 225, and 12 rows of
// threads 80 and 227).
template <bool DIR>
struct GcShape {
    static constexpr int RP = DIR ? 1 : 2, ROWS = 8;
    static constexpr int TY = ROWS * RP;
    static constexpr int RING = (GC_TX + 2) * (TY + 2) - GC_TX * TY;  // nodes around the tile
    static constexpr int OWN = GC_TX * ROWS;
    static constexpr int NT = OWN + (RING + 31) / 32 * 32;
};

// CTAs per SM: 2 (80 registers); with 3 (56) the march spills and took 139 to
// 168 us.  By direction 3 (56, no spill); 2 took as long on one domain and 6%
// more on 64, 4 spill and took a quarter longer
#ifndef LBM_GC_MINB
#define LBM_GC_MINB 2
#endif
#ifndef LBM_GC_MINB_DIR
#define LBM_GC_MINB_DIR 3
#endif
template <bool DIR>
__global__ void __launch_bounds__(GcShape<DIR>::NT, DIR ? LBM_GC_MINB_DIR : LBM_GC_MINB) k_gradcurv(Lattice L)
{
    using R = float;
    using Shape = GcShape<DIR>;
    constexpr int RP = Shape::RP, TY = Shape::TY, NT = Shape::NT, OWN = Shape::OWN;
    constexpr int PW = GC_TX + 4, PH = TY + 4, PN = PW * PH;  // phi / flag region (2-node halo)
    constexpr int NW = GC_TX + 2, NH = TY + 2, NN = NW * NH;  // normal region (1-node halo)
    constexpr int PER = (PN + NT - 1) / NT;                   // region values per thread
    __shared__ R phS[4][PN];
    __shared__ uint8_t flS[4][PN];
    constexpr int NS = DIR ? 4 : 2;                           // normal planes kept
    __shared__ R nS[NS][3][NN];
    __shared__ GcPart<R> partS[MAX_PART];

    const long long item = blockIdx.x;
    int k = 0;
    {
        int lo = 0, hi = L.n_inst - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (L.inst[mid].gc_item_start <= item) lo = mid;
            else hi = mid - 1;
        }
        k = lo;
    }
    const InstDev &I = L.inst[k];
    const int loc = (int)(item - I.gc_item_start);
    const int t2 = I.fd_nchunks.div(loc);
    const int chunk = loc - t2 * I.gc_nchunks;
    const int ty = I.fd_tiles_x.div(t2);
    const int x0 = (t2 - ty * I.gc_tiles_x) * GC_TX, y0 = ty * TY;
    const int z0 = chunk * I.gc_zc, zc = min(I.gc_zc, I.nz - z0);
    const int nx = I.nx, ny = I.ny, nz = I.nz;
    const uint8_t *const fli = L.flags + I.node_off;
    const R *const ph = (const R *)L.phi + I.node_off;
    const int tid = threadIdx.x;

    // this thread's first node: column (ax, ay) of the 1-halo region
    const bool own = tid < OWN;
    int ax, ay;
    if (own) {
        ax = 1 + tid % GC_TX;
        ay = 1 + tid / GC_TX * RP;
    } else {
        const int r = min(tid - OWN, Shape::RING - 1);  // the last warp's spare threads repeat the last node
        if (r < 2 * NW) {
            ax = r < NW ? r : r - NW;
            ay = r < NW ? 0 : NH - 1;
        } else {
            ax = r & 1 ? NW - 1 : 0;
            ay = 1 + (r - 2 * NW) / 2;
        }
    }
    const int gx = x0 + ax - 1, gy = y0 + ay - 1;  // periodic images for nodes around the tile
    const int pc = (ay + 1) * PW + (ax + 1), nc = ay * NW + ax;
    GradRec<R> *out = (GradRec<R> *)L.grad + I.node_off + ((long long)z0 * ny + gy) * nx + gx;  // of plane z0
    const int plane = nx * ny;

    // this thread's share of a plane region, fetched one iteration ahead
    int roff[PER];
#pragma unroll
    for (int q = 0; q < PER; q++) {
        const int r = min(tid + q * NT, PN - 1);
        roff[q] = wrap_any(y0 - 2 + r / PW, ny) * nx + wrap_any(x0 - 2 + r % PW, nx);
    }
    const R eps2 = I.f_eps2;
    pdl_trigger();  // the collision may be scheduled as this grid drains
    pdl_wait();     // phi of the order-parameter pass
    R pv[PER];
    uint8_t fv[PER];
    int zf = wrap_any(z0 - 2, nz);  // plane to fetch next
    auto fetch = [&]() {
        const int zo = zf * plane;
        zf = zf == nz - 1 ? 0 : zf + 1;
#pragma unroll
        for (int q = 0; q < PER; q++) {
            pv[q] = ph[zo + roff[q]];
            fv[q] = fli[zo + roff[q]];
        }
    };
    // the fetched plane into slot j of the rings; whether it carries any flag
    auto store = [&](int j) {
        bool any = false;
#pragma unroll
        for (int q = 0; q < PER; q++) {
            const int r = tid + q * NT;
            if (PER * NT == PN || r < PN) {
                phS[j & 3][r] = pv[q];
                flS[j & 3][r] = fv[q];
            }
            any |= fv[q] != 0;
        }
        return any;
    };
    for (int p = tid; p < I.np; p += NT) {
        const PartDev &P = L.parts[I.part_off + p];
        for (int a = 0; a < 3; a++) partS[p].x[a] = P.xf[a];
        partS[p].rad = (R)P.R;
        partS[p].c = (R)P.cos_t;
        partS[p].s = (R)P.sin_t;
    }
    fetch();
    bool flagged = false;                          // plane j - 1 carries flags
    bool flagged_next = __syncthreads_or(store(0));  // plane j

    GcColumn<R> col[RP];
    R kp[RP], ud[RP];              // curvature of the last normal plane but for the plane above; its U - V
    R corr1[RP], corr2[RP];        // the solid neighbours' share of it, planes z0-4+j and z0-5+j
    unsigned fl1 = 0, fl2 = 0;     // own fluid nodes of those planes, a bit per row
    unsigned sol1[RP], sol2[RP];   // by direction: their solid neighbours
#pragma unroll
    for (int r = 0; r < RP; r++) sol1[r] = sol2[r] = 0;
#pragma unroll
    for (int r = 0; r < RP; r++) kp[r] = ud[r] = corr1[r] = corr2[r] = 0;
    unsigned inside = 0;           // own nodes inside the domain
#pragma unroll
    for (int r = 0; r < RP; r++)
        if (own && gx < nx && gy + r < ny) inside |= 1u << r;

    for (int j = 0; j < zc + 5; j++) {
        if (j < zc + 3) fetch();
        R corr[RP];
        unsigned sol[RP];
#pragma unroll
        for (int r = 0; r < RP; r++) {
            corr[r] = 0;
            sol[r] = 0;
        }
        unsigned fluid = 0;
        if (j < zc + 4) {
            // (1) gradient and normal of plane z0-3+j; 0 for a solid node
            // (by direction: from the rows of the three planes around it)
            R v[RP + 2][3], vm[DIR ? RP + 2 : 1][3], vp[DIR ? RP + 2 : 1][3];
            {
                const R *pl = phS[(DIR ? j - 1 : j) & 3] + pc;
#pragma unroll
                for (int r = 0; r < RP + 2; r++)
                    if (r < 3 || own) load_row(pl + (r - 1) * PW, v[r]);
            }
            if constexpr (DIR) {
                const R *pm = phS[(j - 2) & 3] + pc, *pp = phS[j & 3] + pc;
#pragma unroll
                for (int r = 0; r < RP + 2; r++)
                    if (r < 3 || own) {
                        load_row(pm + (r - 1) * PW, vm[r]);
                        load_row(pp + (r - 1) * PW, vp[r]);
                    }
            }
#pragma unroll
            for (int r = 0; r < RP; r++) {
                if (r > 0 && !own) break;
                R g[3], nn[3];
                if constexpr (DIR)
                    dir_gradient<R>([&](int dx, int dy, int dz) { return (dz < 0 ? vm : (dz > 0 ? vp : v))[r + 1 + dy][1 + dx]; }, g);
                else
                    col[r].advance(v[r], v[r + 1], v[r + 2], g);
                if (j < 2) continue;
                bool solid = false;
                R s0 = 0, s1 = 0, s2 = 0;
                if (flagged) {
                    const int c = pc + r * PW;
                    const uint8_t fl = flS[(j - 1) & 3][c];
                    solid = (fl & OWNER_MASK) != OWN_FLUID;
                    if (!solid && (fl & BOUND_BIT)) {
                        R sv[3] = {0, 0, 0};
                        const uint8_t *f0 = flS[(j - 2) & 3], *f1 = flS[(j - 1) & 3], *f2 = flS[j & 3];
                        sol[r] = gc_solid<DIR, R>(
                            I, [&](int p) -> const GcPart<R> & { return partS[p]; },
                            [&](int i) { return (cz(i) < 0 ? f0 : (cz(i) > 0 ? f2 : f1))[c + cy(i) * PW + cx(i)]; },
                            phS[(j - 1) & 3][c], wrap_any(gx, nx), wrap_any(gy + r, ny), wrap_any(z0 - 3 + j, nz), g,
                            sv);
                        s0 = sv[0]; s1 = sv[1]; s2 = sv[2];
                    }
                }
                if constexpr (DIR) {
                    dir_normal(g, eps2, nn);
                } else {
                    const R im = frsqrt(fma_rn(g[0], g[0], fma_rn(g[1], g[1], fma_rn(g[2], g[2], eps2))));
                    nn[0] = mul_rn(g[0], im);
                    nn[1] = mul_rn(g[1], im);
                    nn[2] = mul_rn(g[2], im);
                }
                if (solid) nn[0] = nn[1] = nn[2] = 0;
                if (own) {
                    const bool here = !solid && (inside >> r & 1u);
                    if (here && j >= 3 && j < zc + 3) out[(j - 3) * plane + r * nx].set_gradient(g);
                    if (here) fluid |= 1u << r;
                    if constexpr (!DIR) corr[r] = fma_rn(nn[0], s0, fma_rn(nn[1], s1, mul_rn(nn[2], s2)));
                }
                R *d = &nS[j & (NS - 1)][0][nc + r * NW];
                d[0] = nn[0];
                d[NN] = nn[1];
                d[2 * NN] = nn[2];
            }
        }
        if constexpr (DIR) {
            // (2) curvature of plane z0-5+j from the normals of the planes around it
            if (j >= 5 && own) {
                const R *n0 = nS[(j - 3) & 3][0] + nc, *n1 = nS[(j - 2) & 3][0] + nc, *n2 = nS[(j - 1) & 3][0] + nc;
#pragma unroll
                for (int r = 0; r < RP; r++) {
                    auto normal = [&](int i) { return (cz(i) < 0 ? n0 : (cz(i) > 0 ? n2 : n1)) + (r + cy(i)) * NW + cx(i); };
                    // a warp takes one of the two ways, not both in turn
                    R k;
                    if (__any_sync(0xffffffffu, sol2[r] != 0))
                        k = dir_curvature<R>([&](int a, int i) {
                            const R *q = sol2[r] >> i & 1u ? n1 + r * NW : normal(i);
                            return q[a * NN];
                        });
                    else
                        k = dir_curvature<R>([&](int a, int i) { return normal(i)[a * NN]; });
                    if (fl2 >> r & 1u) out[(j - 5) * plane + r * nx].k = k;
                }
            }
        } else
        // (2) curvature of plane z0-5+j: the in-plane sums of the normals of plane z0-4+j
        if (j >= 3 && own) {
            const R *a = nS[(j - 1) & 1][0] + nc, *b = a + NN, *d = b + NN;
            R av[RP + 2][2], bv[RP + 2][3], dv[RP + 2], dw[RP][2];
#pragma unroll
            for (int r = 0; r < RP + 2; r++) {
                av[r][0] = a[(r - 1) * NW - 1];
                av[r][1] = a[(r - 1) * NW + 1];
                load_row(b + (r - 1) * NW, bv[r]);
                dv[r] = d[(r - 1) * NW];
            }
#pragma unroll
            for (int r = 0; r < RP; r++) {
                dw[r][0] = d[r * NW - 1];
                dw[r][1] = d[r * NW + 1];
            }
#pragma unroll
            for (int r = 0; r < RP; r++) {
                const R twelfth = R(1.0 / 12.0), sixth = R(1.0 / 6.0);
                const R e = add_rn(sub_rn(av[r + 1][1], av[r + 1][0]), sub_rn(bv[r + 2][1], bv[r][1]));
                const R U = mul_rn(twelfth, e);
                const R V = fma_rn(sixth, dv[r + 1],
                                   mul_rn(twelfth, add_rn(add_rn(dw[r][1], dw[r][0]), add_rn(dv[r + 2], dv[r]))));
                const R diag = add_rn(sub_rn(add_rn(av[r + 2][1], bv[r + 2][2]), add_rn(av[r][0], bv[r][0])),
                                      sub_rn(sub_rn(av[r][1], bv[r][2]), sub_rn(av[r + 2][0], bv[r + 2][0])));
                if ((fl2 >> r & 1u) && j >= 5)
                    out[(j - 5) * plane + r * nx].k = add_rn(add_rn(kp[r], add_rn(U, V)), corr2[r]);
                kp[r] = fma_rn(sixth, e, fma_rn(twelfth, diag, ud[r]));
                ud[r] = sub_rn(U, V);
            }
        }
#pragma unroll
        for (int r = 0; r < RP; r++) {
            corr2[r] = corr1[r];
            corr1[r] = corr[r];
            sol2[r] = sol1[r];
            sol1[r] = sol[r];
        }
        fl2 = fl1;
        fl1 = fluid;
        flagged = flagged_next;
        flagged_next = __syncthreads_or(j < zc + 3 ? store(j + 1) : false);
    }
}

// The form without tiles: a node per thread and two kernels, the normals going
// through memory, with the roundings of the marching form (the same bits).
//
// FP64: FP64 instructions have 2 lanes a clock on an SM, so that they are the
// cost (about 35 of the gradient, 45 of the normal, 40 of the curvature; on
// 48x32x32 nodes some 10 us of the whole chip), and the marching tiles' work
// around their nodes, 1.6 times the normals in a plane and 4 planes more than a
// chunk has, is what a run cannot afford: 48x32x32 with a sphere 25 us for both
// kernels, 59 us marching.  One warp a CTA, since the FP64 pipe that a CTA lands
// on is shared by its SM.
//
// FP32 arithmetic: bound by latency on a small grid, where a march of some 10
// planes with a barrier each is a chain that few CTAs walk, and by loads (48 a
// node) and 28 bytes a node more on a large one.  Marching against this form,
// with the events' 5 us: 48x32x32 21 and 11 us; 0.44 M nodes as 4 x 48^3 29 and
// 19; 0.7 M as one domain 24 and 23 (201x91x37) or 21 and 23 (128x80x72), as 6
// x 48^3 38 and 25, as 19 x 40x33x29 49 and 29; 0.88 M as 96^3 25 and 27, as 8
// x 48^3 35 and 31; 256x128x64 35 and 49; 256x128x128 73 and 115: taken up to
// GRAD_NODES_MAX nodes of a context.  (Marching with gathered sums.  A uniform
// field in FP32, by direction: 4 x 48^3 19 and 19, 6 x 48^3 22 and 25, 19 x
// 40x33x29 32 and 28, 96^3 22 and 26, 256x128x64 41 and 52.)
template <class R>
constexpr int GN_THREADS = sizeof(R) == 8 ? 32 : 128;
template <class R>
__device__ __forceinline__ bool gn_node(const Lattice &L, const InstDev **I, int *n, int *x, int *y, int *z)
{
    constexpr int PER = COLLIDE_NODES<R> / GN_THREADS<R>;  // CTAs of a work item of the collision
    return item_node(L, blockIdx.x / PER, COLLIDE_NODES<R>,
                     (int)(blockIdx.x % PER) * GN_THREADS<R> + (int)threadIdx.x, I, n, x, y, z);
}

// gradient, wetting and normal (0 at a solid node); the solid neighbours' share
// of the curvature into its slot
template <class R, bool DIR>
__global__ void __launch_bounds__(GN_THREADS<R>) k_grad_nodes(Lattice L)
{
    const InstDev *Ip;
    int n, x, y, z;
    const bool have = gn_node<R>(L, &Ip, &n, &x, &y, &z);
    pdl_trigger();
    pdl_wait();  // phi of the order-parameter pass
    if (!have) return;
    const InstDev &I = *Ip;
    const uint8_t *const fli = L.flags + I.node_off;
    const R *const ph = (const R *)L.phi + I.node_off;
    R *const nrm = (R *)L.nrm + I.node_off;
    Nbr nb;
    nb.init(x, y, z, I.nx, I.ny, I.nz);
    const uint8_t fl = fli[n];
    R v[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) v[i] = ph[nb.at(cx(i), cy(i), cz(i))];
    if ((fl & OWNER_MASK) != OWN_FLUID) {
        for (int a = 0; a < 3; a++) nrm[a * L.Ntot + n] = 0;
        return;
    }
    auto at = [&](int dx, int dy, int dz) { return v[dir_of(dx, dy, dz)]; };
    const R twelfth = R(1.0 / 12.0), sixth = R(1.0 / 6.0);
    R g[3];
    if constexpr (DIR) {
        dir_gradient<R>(at, g);
    } else {
        const R d1 = sub_rn(at(1, 1, 0), at(-1, -1, 0)), d2 = sub_rn(at(1, -1, 0), at(-1, 1, 0));
        const R X = sub_rn(at(1, 0, 0), at(-1, 0, 0)), Y = sub_rn(at(0, 1, 0), at(0, -1, 0));
        R hx[2], hy[2], q[2];  // of the planes below and above
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const int dz = 2 * k - 1;
            hx[k] = mul_rn(twelfth, sub_rn(at(1, 0, dz), at(-1, 0, dz)));
            hy[k] = mul_rn(twelfth, sub_rn(at(0, 1, dz), at(0, -1, dz)));
            q[k] = fma_rn(sixth, at(0, 0, dz),
                          mul_rn(twelfth, add_rn(add_rn(at(1, 0, dz), at(-1, 0, dz)), add_rn(at(0, 1, dz), at(0, -1, dz)))));
        }
        g[0] = add_rn(fma_rn(sixth, X, fma_rn(twelfth, add_rn(d1, d2), hx[0])), hx[1]);
        g[1] = add_rn(fma_rn(sixth, Y, fma_rn(twelfth, sub_rn(d1, d2), hy[0])), hy[1]);
        g[2] = sub_rn(q[1], q[0]);
    }
    R sv[3] = {0, 0, 0};
    if (fl & BOUND_BIT) {
        auto part = [&](int p) {
            const PartDev &P = L.parts[I.part_off + p];
            if constexpr (sizeof(R) == 8) return GcPart<R>{{P.x[0], P.x[1], P.x[2]}, P.R, P.cos_t, P.sin_t};
            else return GcPart<R>{{P.xf[0], P.xf[1], P.xf[2]}, (R)P.R, (R)P.cos_t, (R)P.sin_t};
        };
        gc_solid<DIR, R>(
            I, part, [&](int i) { return fli[nb.at(cx(i), cy(i), cz(i))]; }, v[0], x, y, z, g, sv);
    }
    const R eps2 = sizeof(R) == 8 ? (R)(I.grad_eps * I.grad_eps) : (R)I.f_eps2;
    R nn[3];
    if constexpr (DIR) {
        dir_normal(g, eps2, nn);
    } else {
        const R im = frsqrt(fma_rn(g[0], g[0], fma_rn(g[1], g[1], fma_rn(g[2], g[2], eps2))));
        for (int a = 0; a < 3; a++) nn[a] = mul_rn(g[a], im);
    }
    for (int a = 0; a < 3; a++) nrm[a * L.Ntot + n] = nn[a];
    const R share = fma_rn(nn[0], sv[0], fma_rn(nn[1], sv[1], mul_rn(nn[2], sv[2])));
    ((GradRec<R> *)L.grad)[I.node_off + n] = GradRec<R>{g[0], g[1], g[2], share};
}

// curvature
template <class R, bool DIR>
__global__ void __launch_bounds__(GN_THREADS<R>) k_curv_nodes(Lattice L)
{
    const InstDev *Ip;
    int n, x, y, z;
    const bool have = gn_node<R>(L, &Ip, &n, &x, &y, &z);
    pdl_trigger();  // the collision may be scheduled as this grid drains
    pdl_wait();     // the normals
    if (!have) return;
    const InstDev &I = *Ip;
    const R *const nrm = (const R *)L.nrm + I.node_off;
    R *const k = &((GradRec<R> *)L.grad)[I.node_off + n].k;
    Nbr nb;
    nb.init(x, y, z, I.nx, I.ny, I.nz);
    const uint8_t *const fli = L.flags + I.node_off;
    const uint8_t fl = fli[n];
    if constexpr (DIR) {
        if ((fl & OWNER_MASK) != OWN_FLUID) return;
        auto normal = [&](int a, int i) { return nrm[a * L.Ntot + nb.at(cx(i), cy(i), cz(i))]; };
        if (fl & BOUND_BIT) {
            unsigned solid = 0;
#pragma unroll
            for (int i = 1; i < Q; i++)
                if ((fli[nb.at(cx(i), cy(i), cz(i))] & OWNER_MASK) != OWN_FLUID) solid |= 1u << i;
            *k = dir_curvature<R>([&](int a, int i) { return solid >> i & 1u ? nrm[a * L.Ntot + n] : normal(a, i); });
        } else
            *k = dir_curvature<R>(normal);
        return;
    }
    const R share = *k;
    // normals' components where the curvature takes them: n_a of the neighbours with c_a != 0
    auto at = [&](int a, int dx, int dy, int dz) { return nrm[a * L.Ntot + nb.at(dx, dy, dz)]; };
    const R twelfth = R(1.0 / 12.0), sixth = R(1.0 / 6.0);
    R e[3];
#pragma unroll
    for (int dz = -1; dz <= 1; dz++)
        e[dz + 1] = add_rn(sub_rn(at(0, 1, 0, dz), at(0, -1, 0, dz)), sub_rn(at(1, 0, 1, dz), at(1, 0, -1, dz)));
    R U[2], W[2];  // of the planes below and above
#pragma unroll
    for (int m = 0; m < 2; m++) {
        const int dz = 2 * m - 1;
        U[m] = mul_rn(twelfth, e[2 * m]);
        W[m] = fma_rn(sixth, at(2, 0, 0, dz),
                      mul_rn(twelfth, add_rn(add_rn(at(2, 1, 0, dz), at(2, -1, 0, dz)),
                                             add_rn(at(2, 0, 1, dz), at(2, 0, -1, dz)))));
    }
    const R diag = add_rn(sub_rn(add_rn(at(0, 1, 1, 0), at(1, 1, 1, 0)), add_rn(at(0, -1, -1, 0), at(1, -1, -1, 0))),
                          sub_rn(sub_rn(at(0, 1, -1, 0), at(1, 1, -1, 0)), sub_rn(at(0, -1, 1, 0), at(1, -1, 1, 0))));
    const R kp = fma_rn(sixth, e[1], fma_rn(twelfth, diag, sub_rn(U[0], W[0])));
    if ((fl & OWNER_MASK) == OWN_FLUID) *k = add_rn(add_rn(kp, add_rn(U[1], W[1])), share);
}

// Cost of marching chunks of zc planes (and `halo` planes more) through column
// tiles of tx x ty nodes over all instances, in plane iterations: the waves of
// CTAs, counted as full ones (a CTA of the last wave runs as long as any) and
// as what they hold (an SM with fewer CTAs runs them faster) alike, and half a
// wave of drain.  Measured against it on 256x128x128 FP32, order parameter by
// planes per chunk 4, 8, 13, 16, 19, 32, 43: 106, 99, 97, 105, 93, 120, 97 us
// (cost 111, 100, 95, 104, 94, 124, 105); gradient pass 8, 15, 16, 22, 26,
// 32, 43: 75, 73, 75, 80, 92, 78, 97 us (94, 83, 84, 98, 106, 84, 100).
static double march_cost(const std::vector<InstDev> &inst, int tx, int ty, int zc, int halo, double slots)
{
    double items = 0.0;
    for (const auto &I : inst)
        items += (double)((I.nx + tx - 1) / tx) * ((I.ny + ty - 1) / ty) * ((I.nz + zc - 1) / zc);
    const double waves = items / slots;
    return (std::ceil(waves) + waves + 0.5) * (zc + halo);
}
constexpr int ZC_MAX = 64;

// The FP32 gradient pass's work items.  Where no z-chunk is asked for, the
// planes per item of the least cost; slots are the resident CTAs.  128x64x64, 4
// planes against 16: 24 against 37 us.  Every choice gives the same bits.
int planned_zchunk(const std::vector<InstDev> &inst, int n_sm, bool dir)
{
    const double slots = n_sm * (double)(dir ? LBM_GC_MINB_DIR : LBM_GC_MINB);
    const int TY = dir ? GcShape<true>::TY : GcShape<false>::TY;
    int planned = 16;
    double least = -1.0;
    for (int zc = ZC_MAX; zc >= 2; zc--) {
        const double cost = march_cost(inst, GC_TX, TY, zc, 4, slots);
        if (least < 0.0 || cost < least) {
            least = cost;
            planned = zc;
        }
    }
    return planned;
}

void plan_gradcurv(std::vector<InstDev> &inst, int zc_request, const std::vector<int> &zc_inst, int n_sm, bool dir,
                   FluidLaunch *fz)
{
    const int TY = dir ? GcShape<true>::TY : GcShape<false>::TY;
    const int zc_auto = planned_zchunk(inst, n_sm, dir);
    long long items = 0;
    for (size_t k = 0; k < inst.size(); k++) {
        InstDev &I = inst[k];
        const int req = k < zc_inst.size() && zc_inst[k] > 0 ? zc_inst[k] : zc_request;
        I.gc_tiles_x = (I.nx + GC_TX - 1) / GC_TX;
        I.gc_tiles_y = (I.ny + TY - 1) / TY;
        const int zc = std::min(req > 0 ? req : zc_auto, I.nz);
        I.gc_nchunks = (I.nz + zc - 1) / zc;
        I.gc_zc = (I.nz + I.gc_nchunks - 1) / I.gc_nchunks;
        I.fd_nchunks.set(I.gc_nchunks);
        I.fd_tiles_x.set(I.gc_tiles_x);
        I.gc_item_start = items;
        items += (long long)I.gc_tiles_x * I.gc_tiles_y * I.gc_nchunks;
    }
    fz->gc_items = items;
}

// The order-parameter pass's work items, planned alike: one plane of halo
// staged on each side of a chunk.  An instance's form follows from its own shape
// (its results must not depend on what else a context holds).
static bool phi_by_node(const InstDev &I, bool fp64)
{
    const double tiles = (double)((I.nx + PH_TX - 1) / PH_TX) * ((I.ny + PH_TY - 1) / PH_TY);
    return !fp64 && (double)I.nx * I.ny * I.nz < PN_SHARE * (PH_TX * PH_TY) * tiles * (I.nz + 2);
}

void plan_phi(std::vector<InstDev> &inst, int n_sm, bool fp64, FluidLaunch *fz)
{
    const double slots = n_sm * (fp64 ? 1.0 : (double)LBM_PHI_MINB);
    std::vector<InstDev> tiled;
    for (const auto &I : inst)
        if (!phi_by_node(I, fp64)) tiled.push_back(I);
    int best = 16;
    double least = -1.0;
    for (int zc = ZC_MAX; zc >= 2; zc--) {
        const double cost = march_cost(tiled, PH_TX, PH_TY, zc, 2, slots);
        if (least < 0.0 || cost < least) {
            least = cost;
            best = zc;
        }
    }
    long long items = 0, nodes = 0;
    for (auto &I : inst) {
        I.ph_tiles_x = (I.nx + PH_TX - 1) / PH_TX;
        const int tiles_y = (I.ny + PH_TY - 1) / PH_TY;
        I.pn_item_start = nodes;
        I.ph_item_start = items;
        if (phi_by_node(I, fp64)) {
            nodes += (I.N + PN_NODES - 1) / PN_NODES;
            continue;
        }
        const int zc = std::min(best, I.nz);
        I.ph_nchunks = (I.nz + zc - 1) / zc;
        I.ph_zc = (I.nz + I.ph_nchunks - 1) / I.ph_nchunks;
        I.fd_ph_nchunks.set(I.ph_nchunks);
        I.fd_ph_tiles_x.set(I.ph_tiles_x);
        items += (long long)I.ph_tiles_x * tiles_y * I.ph_nchunks;
    }
    fz->ph_items = items;
    fz->pn_items = nodes;
}

// the collision's work items
void plan_items(std::vector<InstDev> &inst, bool fp64, FluidLaunch *fz)
{
    const long long per = fp64 ? COLLIDE_NODES<double> : COLLIDE_NODES<float>;
    long long total = 0;
    for (auto &I : inst) {
        I.fd_nx.set(I.nx);
        I.fd_ny.set(I.ny);
        I.item_start = total;
        total += (I.N + per - 1) / per;
    }
    fz->items = total;
}

// launch with programmatic stream serialisation: the kernel may be scheduled
// while its predecessor in the stream drains (it calls pdl_wait first)
template <class... P, class... A>
static void launch_after(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <class S>
void launch_fluid_step(const Lattice &L, int cur, cudaStream_t st, long long *launches, const Marker &mk,
                       const FluidLaunch &fz, const SideLane &lane)
{
    using R = typename Store<S>::real;
    const dim3 grid((unsigned)fz.items);  // one CTA per work item of the collision
    const bool pair = sizeof(S) == 2 && fz.pair;
    // boundary passes: grid-stride over the listed particle nodes and the
    // static list of nodes next to walls
    const dim3 bgrid((unsigned)std::max(L.bound_ctas, 1));
    const bool any_bound = L.n_parts > 0 || L.n_static_bfl > 0;
    // phi of solid nodes next to fluid reads phi only at fluid nodes next to a
    // solid, which the boundary pass writes, so it follows that pass beside the
    // bulk kernel
    auto fill_solid_phi = [&](cudaStream_t s) {
        if (L.n_static == 0 && L.n_parts == 0) return;
        const long long ctas = (L.n_static + PART_THREADS - 1) / PART_THREADS + (L.n_parts ? L.bound_ctas / 8 : 0);
        mk(STAGE_SOLIDPHI, 0);
        k_solidphi<R><<<(unsigned)std::max(std::min(ctas, 8ll * L.bound_ctas), 1ll), PART_THREADS, 0, s>>>(L);
        mk(STAGE_SOLIDPHI, 1);
        *launches += 1;
    };
    // a boundary pass beside the bulk kernels (side lane), from here in the
    // main stream on; profiling (no side lane) times it alone
    auto bound_pass = [&](auto kernel, int stage) {
        if (!any_bound) return;
        cudaStream_t s = lane.side ? lane.side : st;
        if (lane.side) {
            cudaEventRecord(lane.a, st);
            cudaStreamWaitEvent(lane.side, lane.a, 0);
        }
        mk(stage, 0);
        kernel<<<bgrid, BOUND_THREADS<S>, 0, s>>>(L, cur);
        mk(stage, 1);
        *launches += 1;
    };
    bound_pass(k_phi_bound<S>, STAGE_PHI_BOUND);
    fill_solid_phi(lane.side && any_bound ? lane.side : st);
    if (lane.side && any_bound) cudaEventRecord(lane.b, lane.side);
    lane.after_phi_bound();
    mk(STAGE_PHI, 0);
    if constexpr (sizeof(S) < 8)
        if (fz.pn_items > 0) k_phi_nodes<S><<<(unsigned)fz.pn_items, PN_NODES, 0, st>>>(L, cur);
    if (fz.ph_items > 0) k_phi<S><<<(unsigned)fz.ph_items, PH_TX * PH_TY, 0, st>>>(L, cur);
    if (fz.pn_items > 0 && fz.ph_items > 0) *launches += 1;
    mk(STAGE_PHI, 1);
    if (lane.side && any_bound) cudaStreamWaitEvent(st, lane.b, 0);
    mk(STAGE_GRAD, 0);
    if (L.nrm) {
        const dim3 ctas((unsigned)(fz.items * (COLLIDE_NODES<R> / GN_THREADS<R>)));
        launch_after(k_grad_nodes<R, BY_DIRECTION<S>>, ctas, dim3(GN_THREADS<R>), st, L);
        launch_after(k_curv_nodes<R, BY_DIRECTION<S>>, ctas, dim3(GN_THREADS<R>), st, L);
        *launches += 1;
    } else
        launch_after(k_gradcurv<BY_DIRECTION<S>>, dim3((unsigned)fz.gc_items), dim3(GcShape<BY_DIRECTION<S>>::NT), st, L);
    mk(STAGE_GRAD, 1);
    lane.after_grad();
    if constexpr (BOUNCE_IN_SLOTS<S>) {
        lane.after_collide_bound();
        mk(STAGE_COLLIDE, 0);
        launch_after(k_collide<S>, grid, dim3(COLLIDE_NODES<S>), st, L, cur);
        mk(STAGE_COLLIDE, 1);
    } else {
        bound_pass(k_collide_bound<S>, STAGE_COLLIDE_BOUND);
        if (lane.side && any_bound) cudaEventRecord(lane.b, lane.side);
        lane.after_collide_bound();
        mk(STAGE_COLLIDE, 0);
        if (pair) launch_after(k_collide2<S>, grid, dim3(COLLIDE_NODES<S> / 2), st, L, cur);
        else launch_after(k_collide<S>, grid, dim3(COLLIDE_NODES<S>), st, L, cur);
        mk(STAGE_COLLIDE, 1);
        if (lane.side && any_bound) cudaStreamWaitEvent(st, lane.b, 0);
    }
    *launches += 3;
}


#define INST(S)                                                                                                   \
    template void launch_mark_solid<S>(const Lattice &, cudaStream_t);                                             \
    template void launch_fluid_step<S>(const Lattice &, int, cudaStream_t, long long *, const Marker &,            \
                                       const FluidLaunch &, const SideLane &);
INST(double)
INST(float)
INST(__half)
INST(__nv_bfloat16)
#undef INST

}  // namespace lbmg
