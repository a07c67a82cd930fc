// Learned particle-force surrogate (an extension of the method, not in the
// paper): samples of the flow on a shell around each sphere feed a
// 400-128-128-6 tanh network whose output replaces the momentum-exchange and
// capillary forces.  The network runs and trains with BF16 operands on the
// fifth-generation tensor cores: tcgen05.mma with the accumulator in tensor
// memory, operands staged in shared memory, FP32 master weights, Adam.
//
// The products are small (0.14 GFLOP forward for 1000 rows), so what they cost
// is latency: launches, round trips to memory, and barriers.  Two kernels:
//   k_mlp_rows   a CTA takes 32 rows through the whole network: inputs gathered
//                and rounded to BF16 on the way into shared memory, the three
//                layers with their activations, and in training the loss and
//                both layers' deltas; weights and activations stay in shared
//                memory from one product to the next;
//   k_mlp_grads  the weight gradients (sums over the batch) with the bias
//                gradients and the loss, a CTA per output tile.
// The rows are the N side of the products and the layer's units the M side, so
// that a CTA may have few rows (a batch of 512 is 16 CTAs) and yet every lane of
// the tensor memory a value.
// One GEMM launch per product with operands staged 64 columns at a time by a
// loop of dependent loads took 36 to 46 us each, 17 launches and 285 us a batch
// of 512; with 128 rows to a CTA (the M side) the two kernels and Adam took 31,
// 18 and 4 us, now 21, 16 and 4.  Each is scheduled while the one before drains,
// and does before its wait what does not depend on it (the rows' gather, Adam's
// moments).  An epoch of 20000 samples 11.4 -> 2.5 -> 2.06 ms, with the
// overlap 1.53 ms; 512 predictions with their copies 132 -> 61 -> 56 us (and 47
// with one synchronisation), to the same bits.
//
// Shared-memory operands are in the canonical layout without swizzle: 8 x
// 16-byte core matrices of 128 bytes.  Read K-major, a core matrix holds 8 rows
// (M or N) of 8 k each; read MN-major, 8 k of 8 consecutive m or n each - the
// same bytes serve a product with the operand and one with its transpose.
// Descriptors give the distance between core matrices along k (leading) and
// along M or N (stride).
#include <cmath>
#include <mutex>
#include <vector>

#include "lbm_async.cuh"
#include "lbm_internal.cuh"

namespace lbmg {

using bf16 = __nv_bfloat16;

namespace {

// ---------------------------------------------------------------------------
// tcgen05 wrappers
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// 16 consecutive FP32 columns of this warp's 32 TMEM lanes
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}

// 8 columns
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float *v)
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]);
}

// shared-memory matrix descriptor: start address, leading (k) and stride
// (row-group) byte offsets, descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: BF16 A and B, FP32 D, M = 128, N = BN;
// TA, TB: that operand is read MN-major
template <int BN, bool TA = false, bool TB = false>
__host__ __device__ constexpr uint32_t idesc_bf16()
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((TA ? 1u : 0u) << 15) | ((TB ? 1u : 0u) << 16) |
           ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// the same with the last 16 - bytes of them zero
__device__ __forceinline__ void cp_async16z(uint32_t dst, const void *src, uint32_t bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait_group()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

constexpr int GM = 128;        // M of a product (TMEM lanes)
constexpr int NR = 32;         // rows of a CTA of the row kernel
constexpr int MLP_THREADS = 256;   // gradients: two warps per quarter of the TMEM lanes
constexpr int ROW_THREADS = 512;   // rows: four, of 8 rows each

// STEPS products of K = 16 each into tmem (the first one overwrites it where
// fresh), issued and committed by one thread; a_step, b_step: bytes between
// the k = 16 slices of the operands
template <uint32_t IDESC, int STEPS>
__device__ __forceinline__ void mma_steps(uint32_t tmem, uint32_t a, uint32_t a_lbo, uint32_t a_sbo, uint32_t a_step,
                                          uint32_t b, uint32_t b_lbo, uint32_t b_sbo, uint32_t b_step, bool fresh,
                                          uint32_t bar)
{
    tc_fence_after();
#pragma unroll
    for (int j = 0; j < STEPS; j++)
        tc_mma_bf16(tmem, smem_desc(a + j * a_step, a_lbo, a_sbo), smem_desc(b + j * b_step, b_lbo, b_sbo), IDESC,
                    fresh && j == 0 ? 0u : 1u);
    tc_commit(bar);
}

__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// ---------------------------------------------------------------------------
// the network over rows
// ---------------------------------------------------------------------------
struct RowArgs {
    const float *X;        // inputs [*][387]
    const float *T;        // targets [*][6] (training)
    const long long *idx;  // rows idx[row0 + r] of both, or row0 + r
    long long row0;
    int n;
    const bf16 *W1, *W2, *W3;
    const float *b1, *b2, *b3;
    bf16 *Xb, *H1, *H2, *dZ1, *dZ2, *dYb;  // for the gradients (training)
    float *Y, *dY;
    double *loss_part;
    unsigned *status;
    int no_mma;            // fault injection: issue no MMA and no commit (the wait finds nothing arriving)
    long long wait_limit;  // clock cycles a wait on the commit barrier may take
};

// shared memory: barrier, TMEM slot and biases; the input tile; activations and
// deltas; the weights.  W3 has 16 rows (6..15 zero); a product with it on the M
// side reads 128, whose results past the sixth are not used: up to 1920 bytes
// behind the last slice's, kept in bounds by W3_BYTES
struct RowSmem {
    static constexpr int BIAS = 128;                      // b1[128], b2[128], b3[16]
    static constexpr int RED = BIAS + 4 * (128 + 128 + 16);
    static constexpr int XA = 2048;
    static constexpr int TILE = NR * MLP_HIDDEN * 2;      // 32 x 128
    static constexpr int H1 = XA + NR * MLP_KIN * 2, H2 = H1 + TILE, DZ2 = H2 + TILE, DY = DZ2 + TILE;  // DY: 32 x 16
    static constexpr int W1 = DY + NR * 16 * 2;
    static constexpr int W2 = W1 + MLP_HIDDEN * MLP_KIN * 2;
    static constexpr int W3 = W2 + MLP_HIDDEN * MLP_HIDDEN * 2;
    static constexpr int W3_BYTES = 16 * MLP_HIDDEN * 2 + 2048;
    static constexpr int BYTES = W3 + W3_BYTES;
};
static_assert(RowSmem::RED + 128 <= RowSmem::XA, "regions");
static_assert((MLP_HIDDEN / 8 - 1) * 256 + GM / 8 * 128 <= RowSmem::W3_BYTES, "rows read past W3");
static_assert(RowSmem::BYTES <= 227 * 1024, "shared memory of a CTA");

// bytes between neighbouring core matrices along k and along rows: 128 rows of
// weights, NR rows of the batch
constexpr uint32_t T_LBO = GM / 8 * 128, R_LBO = NR / 8 * 128, T_SBO = 128;

// a weight matrix of 128 rows and K columns, row-major, into shared memory.  A
// warp takes 8 rows by 64 bytes: whole sectors, and whole core matrices
template <int K>
__device__ __forceinline__ void load_weights(uint32_t dst, const bf16 *W, int tid)
{
    constexpr int KB = K / 8, QUADS = (KB + 3) / 4;
    for (int i = tid; i < QUADS * 16 * 32; i += ROW_THREADS) {
        const int r = (i & 7) + 8 * ((i >> 5) & 15), kb = ((i >> 3) & 3) + 4 * (i >> 9);
        if (kb < KB) cp_async16(dst + (kb * 16 + (r >> 3)) * 128 + (r & 7) * 16, W + r * K + kb * 8);
    }
}

template <bool TRAIN>
__global__ void __launch_bounds__(ROW_THREADS, 1) k_mlp_rows(RowArgs g)
{
    using Sm = RowSmem;
    extern __shared__ __align__(1024) unsigned char sm[];
    const uint32_t base = smem_addr(sm), bar = base, slot = base + 16;
    float *const bias = (float *)(sm + Sm::BIAS);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int r0 = blockIdx.x * NR;
    constexpr uint32_t NCOLS = 2 * NR;

    if (warp == 0) {
        tmem_alloc(slot, NCOLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_fence_init();
    }
    // A training batch's inputs and targets do not depend on the kernels before,
    // so their gather runs before the wait for those; a prediction's inputs may
    // be the preceding kernel's.  Programmatic launches (also of the other two
    // kernels) are triggered only after the own wait, so that a kernel running
    // ahead of its wait knows the last but one to be complete.
    if (!TRAIN) {
        pdl_wait();
        pdl_trigger();
    }
    // inputs: a warp takes 2 rows, all loads in flight
    constexpr int NC = (MLP_KIN + 31) / 32;
    float v[2][NC];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int r = r0 + warp * 2 + h;
        const bool have = r < g.n;
        const long long src = have ? (g.idx ? g.idx[g.row0 + r] : g.row0 + r) : 0;
        const float *x = g.X + src * MLP_NIN;
#pragma unroll
        for (int j = 0; j < NC; j++) {
            const int k = lane + 32 * j;
            v[h][j] = have && k < MLP_NIN ? x[k] : 0.0f;
        }
    }
    // this thread's unit (TMEM lane) and its 8 rows (TMEM columns) of the CTA's
    const int unit = (warp & 3) * 32 + lane, row = (warp >> 2) * 8;
    const bool out_unit = unit < MLP_NOUT;
    float target[8];
    if (TRAIN && out_unit) {
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const int r = r0 + row + j;
            target[j] = r < g.n ? g.T[(g.idx ? g.idx[g.row0 + r] : g.row0 + r) * MLP_NOUT + unit] : 0.0f;
        }
    }
    // two values of neighbouring units (or inputs) and one row from lanes 2i and
    // 2i + 1 with one value a and b of two rows each: the even lane's are of the
    // first row, the odd lane's of the second
    const bool odd = lane & 1;
    auto exchange = [&](float a, float b) {
        const float other = __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
        return odd ? pack2(other, b) : pack2(a, other);
    };
    uint32_t xw[NC];
    const int xr = warp * 2 + (int)odd;
    auto store_inputs = [&]() {
#pragma unroll
        for (int j = 0; j < NC; j++) {
            const int k = (lane & ~1) + 32 * j;
            xw[j] = exchange(v[0][j], v[1][j]);
            if (k < MLP_KIN)
                *(uint32_t *)(sm + Sm::XA + (k >> 3) * R_LBO + (xr >> 3) * 128 + (xr & 7) * 16 + (k & 7) * 2) = xw[j];
        }
    };
    if (TRAIN) {
        store_inputs();
        pdl_wait();
        pdl_trigger();
    }
    load_weights<MLP_KIN>(base + Sm::W1, g.W1, tid);
    load_weights<MLP_HIDDEN>(base + Sm::W2, g.W2, tid);
    if (tid < 256) {
        const int r = tid & 15, kb = tid >> 4;
        unsigned char *d = sm + Sm::W3 + (kb * 2 + (r >> 3)) * 128 + (r & 7) * 16;
        *(uint4 *)d = r < MLP_NOUT ? *(const uint4 *)(g.W3 + r * MLP_HIDDEN + kb * 8) : make_uint4(0, 0, 0, 0);
    } else if (tid < 256 + NR * 2) {
        *(uint4 *)(sm + Sm::DY + (tid - 256) * 16) = make_uint4(0, 0, 0, 0);
    }
    if (tid < 128) {
        bias[tid] = g.b1[tid];
        bias[128 + tid] = g.b2[tid];
        if (tid < 16) bias[256 + tid] = tid < MLP_NOUT ? g.b3[tid] : 0.0f;
    }
    if (TRAIN) {
        if (r0 + xr < g.n)
#pragma unroll
            for (int j = 0; j < NC; j++) {
                const int k = (lane & ~1) + 32 * j;
                if (k < MLP_KIN) *(uint32_t *)(g.Xb + (long long)(r0 + xr) * MLP_KIN + k) = xw[j];
            }
    } else {
        store_inputs();
    }
    cp_async_wait();
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *(volatile uint32_t *)(sm + 16);
    const uint32_t d1 = tmem, d2 = tmem + NR;

    unsigned phase = 0;
    bool ok = true;
    // every thread waits for the products committed last; false once a wait gave up
    auto wait = [&]() {
        ok = mbar_wait_bounded(bar, phase & 1, g.wait_limit);
        phase++;
        ok = !__syncthreads_or(!ok);
        tc_fence_after();
        return ok;
    };
    const bool issuer = tid == 0 && !g.no_mma;
    const uint32_t mine = ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)row;
    // the epilogue of a product of 128 units: f(j, value) of this thread's rows,
    // rounded to BF16, kept where asked, into the shared-memory tile at `tile`
    // and, in training, row-major to `out`
    auto epilogue = [&](uint32_t d, int tile, bf16 *out, float *kept, auto &&f) {
        float a[8];
        tmem_ld8(d + mine, a);
#pragma unroll
        for (int j = 0; j < 8; j++) {
            a[j] = __bfloat162float(__float2bfloat16_rn(f(j, a[j])));
            if (kept) kept[j] = a[j];
        }
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            const uint32_t w = exchange(a[j], a[j + 1]);
            const int u = unit & ~1, r = row + j + (int)odd;
            if (tile >= 0) *(uint32_t *)(sm + tile + (u >> 3) * R_LBO + (r >> 3) * 128 + (r & 7) * 16 + (u & 7) * 2) = w;
            if (TRAIN && out && r0 + r < g.n) *(uint32_t *)(out + (long long)(r0 + r) * MLP_HIDDEN + u) = w;
        }
    };
    auto ready = [&]() {  // shared-memory writes of all threads before the next products
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
    };
    float h1[8], h2[8];

    do {
        // h1 = tanh(W1 x + b1)
        if (issuer)
            mma_steps<idesc_bf16<NR>(), MLP_KIN / 16>(d1, base + Sm::W1, T_LBO, T_SBO, 2 * T_LBO, base + Sm::XA, R_LBO,
                                                      T_SBO, 2 * R_LBO, true, bar);
        if (!wait()) break;
        epilogue(d1, Sm::H1, g.H1, h1, [&](int, float a) { return tanhf(a + bias[unit]); });
        ready();
        // h2 = tanh(W2 h1 + b2)
        if (issuer)
            mma_steps<idesc_bf16<NR>(), MLP_HIDDEN / 16>(d2, base + Sm::W2, T_LBO, T_SBO, 2 * T_LBO, base + Sm::H1, R_LBO,
                                                         T_SBO, 2 * R_LBO, true, bar);
        if (!wait()) break;
        epilogue(d2, Sm::H2, g.H2, h2, [&](int, float a) { return tanhf(a + bias[128 + unit]); });
        ready();
        // y = W3 h2 + b3
        if (issuer)
            mma_steps<idesc_bf16<NR>(), MLP_HIDDEN / 16>(d1, base + Sm::W3, 256, T_SBO, 512, base + Sm::H2, R_LBO, T_SBO,
                                                         2 * R_LBO, true, bar);
        if (!wait()) break;
        double e2 = 0.0;
        if ((warp & 3) == 0) {
            float a[8];
            tmem_ld8(d1 + mine, a);
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const int r = row + j;
                const bool have = r0 + r < g.n;
                float d = 0.0f;
                if (out_unit && have) {
                    const float y = a[j] + bias[256 + unit];
                    g.Y[(long long)(r0 + r) * 16 + unit] = y;
                    if (TRAIN) {
                        const float diff = y - target[j];
                        e2 += (double)diff * diff;
                        d = 2.0f * diff / (float)(MLP_NOUT * g.n);
                        g.dY[(long long)(r0 + r) * 16 + unit] = d;
                    }
                }
                if (TRAIN && unit < 16) {
                    // dY = 2 (Y - T)/(6 n), 16 columns of which 6 count
                    const bf16 o = __float2bfloat16_rn(d);
                    if (out_unit) *(bf16 *)(sm + Sm::DY + (r >> 3) * 128 + (r & 7) * 16 + unit * 2) = o;
                    if (have) g.dYb[(long long)(r0 + r) * 16 + unit] = o;
                }
            }
        }
        if constexpr (TRAIN) {
            // squared error of the tile: lanes, then rows by eights, in a fixed order
            for (int o = 16; o > 0; o >>= 1) e2 += __shfl_down_sync(0xffffffffu, e2, o);
            double *const red = (double *)(sm + Sm::RED);
            if (lane == 0 && (warp & 3) == 0) red[warp >> 2] = e2;
            ready();
            if (tid == 0) g.loss_part[blockIdx.x] = ((red[0] + red[1]) + red[2]) + red[3];
            // dz2 = (W3^T dY) (1 - h2^2): W3 read MN-major, m its columns, k its rows
            if (issuer)
                mma_steps<idesc_bf16<NR, true, false>(), 1>(d2, base + Sm::W3, 128, 256, 0, base + Sm::DY, R_LBO, T_SBO, 0,
                                                            true, bar);
            if (!wait()) break;
            epilogue(d2, Sm::DZ2, g.dZ2, nullptr, [&](int j, float a) { return a * (1.0f - h2[j] * h2[j]); });
            ready();
            // dz1 = (W2^T dz2) (1 - h1^2): W2 read MN-major
            if (issuer)
                mma_steps<idesc_bf16<NR, true, false>(), MLP_HIDDEN / 16>(d1, base + Sm::W2, 128, T_LBO, 256,
                                                                          base + Sm::DZ2, R_LBO, T_SBO, 2 * R_LBO, true,
                                                                          bar);
            if (!wait()) break;
            epilogue(d1, -1, g.dZ1, nullptr, [&](int j, float a) { return a * (1.0f - h1[j] * h1[j]); });
        }
    } while (false);
    if (!ok && tid == 0) {
        atomicOr(g.status, ST_TIMEOUT);
        // MMAs still in flight (none are issued under the fault injection) must
        // finish before the tensor memory is freed
        if (!g.no_mma) mbar_wait_bounded(bar, (phase - 1) & 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, NCOLS);
}

// ---------------------------------------------------------------------------
// weight gradients: C[m][n] = sum_b A[b][m] B[b][n] over the batch, A and B
// row-major BF16: both operands are read MN-major, so that their rows go into
// shared memory as they lie, 16 bytes at a time.  A chunk of 64 rows per
// stage, eight stages filled by asynchronous copies, so that a batch of 512 has
// all its loads in flight at once; a stage is refilled only once the commit of
// the chunk that read it has arrived (bounded waits).  Two stages took 17.8 us for
// a batch of 512, eight 16.5.
// ---------------------------------------------------------------------------
struct GradArgs {
    int n;
    const bf16 *Xb, *H1, *H2, *dZ1, *dZ2, *dYb;
    const float *dY;
    float *grad;
    const double *loss_part;
    int parts;
    double *loss, *acc;  // *loss: the batch's; added to *acc where given
    unsigned *status;
    int no_mma;
    long long wait_limit;
};

constexpr int GB = 64;  // batch rows per chunk
constexpr int GN = 64;  // columns of an output tile
constexpr int GRAD_W1 = (MLP_KIN + GN - 1) / GN, GRAD_W2 = MLP_HIDDEN / GN;  // tiles of dW1 and dW2
constexpr int GRAD_TILES = GRAD_W1 + GRAD_W2 + 1;                            // and one of dW3
constexpr int GRAD_CTAS = GRAD_TILES + 2 * (MLP_HIDDEN / 8) + 2;             // bias sums 8 at a time, loss

struct GradSmem {
    static constexpr int STAGES = 8;
    static constexpr int SLOT = 64, HEAD = 128;  // STAGES barriers, the TMEM slot
    static constexpr int A_STAGE = GB * GM * 2, B_STAGE = GB * GN * 2;
    static constexpr int BYTES = HEAD + STAGES * (A_STAGE + B_STAGE);
};
static_assert(GradSmem::BYTES <= 227 * 1024, "shared memory of a CTA");
static_assert(MLP_KIN % 16 == 0 && MLP_OFF_W1 % 4 == 0 && MLP_OFF_W2 % 4 == 0, "16-byte stores of gradient rows");

// one tile: BN columns from n0 of B (ldb apart per row, nb 16-byte groups of it valid)
template <int BN>
__device__ __forceinline__ void grad_tile(const GradArgs &g, unsigned char *sm, const bf16 *A, const bf16 *B, int ldb, int n0,
                                          int nb, float *C, long long scm, long long scn, int ncols)
{
    using Sm = GradSmem;
    constexpr int ST = Sm::STAGES;
    const uint32_t base = smem_addr(sm);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr uint32_t NCOLS = BN < 32 ? 32 : BN;
    constexpr int VA = GB * GM / 8 / MLP_THREADS;                       // 16-byte copies of A a thread
    constexpr int NB8 = BN / 8, VB = (GB * NB8 + MLP_THREADS - 1) / MLP_THREADS;
    const int nchunks = (g.n + GB - 1) / GB;
    // vector i of a chunk: core matrix (k group, m group), row b of 8 in it; the
    // shared-memory place is 16 i.  One group of copies per call, an empty one
    // past the last chunk
    auto fetch = [&](int c) {
        const uint32_t As = base + Sm::HEAD + (c % ST) * Sm::A_STAGE;
        const uint32_t Bs = base + Sm::HEAD + ST * Sm::A_STAGE + (c % ST) * Sm::B_STAGE;
        if (c < nchunks) {
#pragma unroll
            for (int q = 0; q < VA; q++) {
                const int i = tid + q * MLP_THREADS, b = c * GB + (i >> 7) * 8 + (i & 7), mb = (i >> 3) & 15;
                const bool have = b < g.n;
                cp_async16z(As + i * 16, A + (have ? (long long)b * MLP_HIDDEN + mb * 8 : 0), have ? 16 : 0);
            }
#pragma unroll
            for (int q = 0; q < VB; q++) {
                const int i = tid + q * MLP_THREADS, kb = i / (8 * NB8), b = c * GB + kb * 8 + (i & 7), j = (i >> 3) % NB8;
                const bool have = b < g.n && j < nb;
                if (i < GB * NB8) cp_async16z(Bs + i * 16, B + (have ? (long long)b * ldb + n0 + j * 8 : 0), have ? 16 : 0);
            }
        }
        cp_async_commit();
    };
    if (warp == 0) {
        tmem_alloc(base + Sm::SLOT, NCOLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < ST; i++) mbar_init(base + 8 * i, 1);
        mbar_fence_init();
    }
    pdl_wait();  // the batch's activations and deltas
    pdl_trigger();
    for (int c = 0; c < ST; c++) fetch(c);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *(volatile uint32_t *)(sm + Sm::SLOT);
    bool ok = true;
    int last = -1;
    for (int c = 0; c < nchunks; c++) {
        if (c >= 1 && c - 1 + ST < nchunks) {
            // chunk c - 1 + ST takes the stage that the MMAs of chunk c - 1 read
            ok = mbar_wait_bounded(base + 8 * ((c - 1) % ST), (unsigned)(((c - 1) / ST) & 1), g.wait_limit);
            if (__syncthreads_or(!ok)) {
                ok = false;
                break;
            }
            tc_fence_after();
        }
        if (c >= 1) fetch(c - 1 + ST);
        cp_async_wait_group<ST - 1>();  // ST + c groups committed: chunk c has landed
        fence_async_smem();
        __syncthreads();
        if (tid == 0 && !g.no_mma)
            mma_steps<idesc_bf16<BN, true, true>(), GB / 16>(
                tmem, base + Sm::HEAD + (c % ST) * Sm::A_STAGE, 2048, 128, 4096,
                base + Sm::HEAD + ST * Sm::A_STAGE + (c % ST) * Sm::B_STAGE, NB8 * 128, 128, 2 * NB8 * 128, c == 0,
                base + 8 * (c % ST));
        last = c;
    }
    cp_async_wait();
    // a commit covers every MMA this thread issued before it: the last one's
    // arrival means the accumulator is complete
    if (ok && last >= 0) {
        ok = mbar_wait_bounded(base + 8 * (last % ST), (unsigned)((last / ST) & 1), g.wait_limit);
        ok = !__syncthreads_or(!ok);
        tc_fence_after();
    }
    if (!ok) {
        if (tid == 0) {
            atomicOr(g.status, ST_TIMEOUT);
            // MMAs still in flight (none are issued under the fault injection)
            // must finish before the tensor memory is freed
            if (!g.no_mma && last >= 0) mbar_wait_bounded(base + 8 * (last % ST), (unsigned)((last / ST) & 1));
        }
    } else if (warp < 4 || BN > 16) {
        const int m = (warp & 3) * 32 + lane;
        for (int c0 = (warp >> 2) * (BN / 2); c0 < (BN > 16 ? (warp >> 2) * (BN / 2) + BN / 2 : 16); c0 += 16) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, v);
            if (BN > 16) {  // rows of C (scn 1), whole groups of 16 columns
                if (c0 < ncols)
#pragma unroll
                    for (int i = 0; i < 16; i += 4)
                        *(float4 *)(C + m * scm + c0 + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
            } else {
#pragma unroll
                for (int i = 0; i < 16; i++)
                    if (c0 + i < ncols) C[m * scm + (c0 + i) * scn] = v[i];
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, NCOLS);
}

// sums of 8 neighbouring columns in a fixed order (bias gradients), `cols` of
// them wanted
template <class T>
__device__ __forceinline__ void column_sums(const T *src, int rows, int ld, float *sh, float *out, int cols)
{
    float s[8];
#pragma unroll
    for (int e = 0; e < 8; e++) s[e] = 0.0f;
    for (int r = threadIdx.x; r < rows; r += MLP_THREADS) {
        alignas(16) T v[8];
#pragma unroll
        for (int k = 0; k < (int)sizeof v / 16; k++) ((uint4 *)v)[k] = ((const uint4 *)(src + (long long)r * ld))[k];
#pragma unroll
        for (int e = 0; e < 8; e++) s[e] += (float)v[e];
    }
#pragma unroll
    for (int e = 0; e < 8; e++) sh[e * MLP_THREADS + threadIdx.x] = s[e];
    __syncthreads();
    for (int k = MLP_THREADS / 2; k > 0; k >>= 1) {
        if ((int)threadIdx.x < k)
#pragma unroll
            for (int e = 0; e < 8; e++)
                sh[e * MLP_THREADS + threadIdx.x] += sh[e * MLP_THREADS + threadIdx.x + k];
        __syncthreads();
    }
    if ((int)threadIdx.x < cols) out[threadIdx.x] = sh[threadIdx.x * MLP_THREADS];
}

__global__ void __launch_bounds__(MLP_THREADS) k_mlp_grads(GradArgs g)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    int t = blockIdx.x;
    if (t < GRAD_W1) {  // dW1[o][i] = sum_b dz1[b][o] x[b][i]
        const int n0 = t * GN, left = MLP_KIN - n0;
        grad_tile<GN>(g, sm, g.dZ1, g.Xb, MLP_KIN, n0, left / 8, g.grad + MLP_OFF_W1 + n0, MLP_KIN, 1, left);
        return;
    }
    t -= GRAD_W1;
    if (t < GRAD_W2) {  // dW2[o][i] = sum_b dz2[b][o] h1[b][i]
        const int n0 = t * GN;
        grad_tile<GN>(g, sm, g.dZ2, g.H1, MLP_HIDDEN, n0, GN / 8, g.grad + MLP_OFF_W2 + n0, MLP_HIDDEN, 1, GN);
        return;
    }
    t -= GRAD_W2;
    if (t == 0) {  // dW3[j][i] = sum_b dY[b][j] h2[b][i]  (M = hidden i, N = output j)
        grad_tile<16>(g, sm, g.H2, g.dYb, 16, 0, 2, g.grad + MLP_OFF_W3, 1, MLP_HIDDEN, MLP_NOUT);
        return;
    }
    t -= 1;
    float *const sh = (float *)sm;
    pdl_wait();
    pdl_trigger();
    if (t < MLP_HIDDEN / 8) {
        column_sums(g.dZ1 + 8 * t, g.n, MLP_HIDDEN, sh, g.grad + MLP_OFF_B1 + 8 * t, 8);
        return;
    }
    t -= MLP_HIDDEN / 8;
    if (t < MLP_HIDDEN / 8) {
        column_sums(g.dZ2 + 8 * t, g.n, MLP_HIDDEN, sh, g.grad + MLP_OFF_B2 + 8 * t, 8);
        return;
    }
    t -= MLP_HIDDEN / 8;
    if (t == 0) {  // columns 6 and 7 of dY are not written and not wanted
        column_sums(g.dY, g.n, 16, sh, g.grad + MLP_OFF_B3, MLP_NOUT);
        return;
    }
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < g.parts; i++) s += g.loss_part[i];
        const double l = s / ((double)g.n * MLP_NOUT);
        *g.loss = l;
        if (g.acc) *g.acc += l;
    }
}

// these kernels need more than 48 KiB of dynamic shared memory, a function
// attribute of each device: set once per device (under a lock, since
// contexts on several threads may reach here first together), with its result
// checked, before the first launch there
cudaError_t mlp_setup()
{
    constexpr int MAXDEV = 64;
    static std::mutex mu;
    static bool done[MAXDEV] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAXDEV) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return cudaSuccess;
    const auto size = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if ((e = cudaFuncSetAttribute(k_mlp_rows<false>, size, RowSmem::BYTES)) == cudaSuccess &&
        (e = cudaFuncSetAttribute(k_mlp_rows<true>, size, RowSmem::BYTES)) == cudaSuccess &&
        (e = cudaFuncSetAttribute(k_mlp_grads, size, GradSmem::BYTES)) == cudaSuccess)
        done[dev] = true;
    return e;
}

// the row kernel's arguments; under the network's fault-injection setting no
// MMA is issued and the commit barrier is never signalled, so the bounded wait
// (shortened to about a millisecond) runs out and reports a timeout
RowArgs row_args(const Mlp &m, const float *X, const float *T, const long long *idx, long long row0, int n,
                 unsigned *status)
{
    RowArgs a;
    memset(&a, 0, sizeof a);
    a.X = X; a.T = T; a.idx = idx; a.row0 = row0; a.n = n;
    a.W1 = m.W1b; a.W2 = m.W2b; a.W3 = m.W3b;
    a.b1 = m.theta + MLP_OFF_B1; a.b2 = m.theta + MLP_OFF_B2; a.b3 = m.theta + MLP_OFF_B3;
    a.Xb = m.X; a.H1 = m.H1; a.H2 = m.H2; a.dZ1 = m.dZ1; a.dZ2 = m.dZ2; a.dYb = m.dYb;
    a.Y = m.Y; a.dY = m.dY; a.loss_part = m.loss_part;
    a.status = status;
    a.no_mma = m.fault_no_commit ? 1 : 0;
    a.wait_limit = m.fault_no_commit ? 1ll << 21 : WAIT_CYCLES;
    return a;
}

// with programmatic stream serialisation: the kernel may be scheduled while its
// predecessor in the stream drains (it calls pdl_wait first)
template <class... P, class... A>
cudaError_t launch_after(void (*kernel)(P...), int ctas, int threads, int bytes, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)bytes;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// the set-up's or this launch's own error
template <class A>
cudaError_t mlp_launch(void (*kernel)(A), int ctas, int threads, int bytes, const A &a, cudaStream_t st)
{
    const cudaError_t e = mlp_setup();
    return e != cudaSuccess ? e : launch_after(kernel, ctas, threads, bytes, st, a);
}

// ---------------------------------------------------------------------------
// element-wise kernels
// ---------------------------------------------------------------------------
constexpr int EW = 256;

// master weights -> bf16 copies used as GEMM operands
__global__ void k_refresh(const float *theta, bf16 *W1b, bf16 *W2b, bf16 *W3b)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < MLP_HIDDEN * MLP_KIN) W1b[i] = __float2bfloat16_rn(theta[MLP_OFF_W1 + i]);
    if (i < MLP_HIDDEN * MLP_HIDDEN) W2b[i] = __float2bfloat16_rn(theta[MLP_OFF_W2 + i]);
    if (i < MLP_NOUT * MLP_HIDDEN) W3b[i] = __float2bfloat16_rn(theta[MLP_OFF_W3 + i]);
}

// Adam (Kingma and Ba 2015) on the FP32 master weights, and their BF16 copies
__global__ void k_adam(float *theta, const float *grad, float *m, float *v, float lr, float c1, float c2, bf16 *W1b,
                       bf16 *W2b, bf16 *W3b)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool have = i < MLP_NPARAM;
    // the moments and weights are this kernel's own: loaded before the gradients are waited for
    const float m0 = have ? m[i] : 0.0f, v0 = have ? v[i] : 0.0f, t0 = have ? theta[i] : 0.0f;
    pdl_wait();
    pdl_trigger();
    if (!have) return;
    const float g = grad[i];
    const float mi = 0.9f * m0 + 0.1f * g;
    const float vi = 0.999f * v0 + 0.001f * g * g;
    m[i] = mi;
    v[i] = vi;
    const float t = t0 - lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
    theta[i] = t;
    if (i < MLP_OFF_B1) W1b[i] = __float2bfloat16_rn(t);
    else if (i >= MLP_OFF_W2 && i < MLP_OFF_B2) W2b[i - MLP_OFF_W2] = __float2bfloat16_rn(t);
    else if (i >= MLP_OFF_W3 && i < MLP_OFF_B3) W3b[i - MLP_OFF_W3] = __float2bfloat16_rn(t);
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
cudaError_t mlp_alloc(Mlp &m, int cap)
{
    m.cap = cap;
    auto A = [&](void **p, size_t b) { return cudaMalloc(p, b); };
    cudaError_t e;
    if ((e = A((void **)&m.theta, sizeof(float) * MLP_NPARAM)) || (e = A((void **)&m.grad, sizeof(float) * MLP_NPARAM)) ||
        (e = A((void **)&m.adam_m, sizeof(float) * MLP_NPARAM)) ||
        (e = A((void **)&m.adam_v, sizeof(float) * MLP_NPARAM)) ||
        (e = A((void **)&m.W1b, sizeof(bf16) * MLP_HIDDEN * MLP_KIN)) ||
        (e = A((void **)&m.W2b, sizeof(bf16) * MLP_HIDDEN * MLP_HIDDEN)) ||
        (e = A((void **)&m.W3b, sizeof(bf16) * MLP_NOUT * MLP_HIDDEN)) ||
        (e = A((void **)&m.X, sizeof(bf16) * (size_t)cap * MLP_KIN)) ||
        (e = A((void **)&m.H1, sizeof(bf16) * (size_t)cap * MLP_HIDDEN)) ||
        (e = A((void **)&m.H2, sizeof(bf16) * (size_t)cap * MLP_HIDDEN)) ||
        (e = A((void **)&m.dZ1, sizeof(bf16) * (size_t)cap * MLP_HIDDEN)) ||
        (e = A((void **)&m.dZ2, sizeof(bf16) * (size_t)cap * MLP_HIDDEN)) ||
        (e = A((void **)&m.dYb, sizeof(bf16) * (size_t)cap * 16)) || (e = A((void **)&m.Y, sizeof(float) * (size_t)cap * 16)) ||
        (e = A((void **)&m.dY, sizeof(float) * (size_t)cap * 16)) ||
        (e = A((void **)&m.loss_part, sizeof(double) * ((size_t)cap / NR + 1))) ||
        (e = A((void **)&m.loss, sizeof(double) * 2)) || (e = A((void **)&m.dirs, sizeof(double) * 3 * MLP_SHELL)))
        return e;
    // directions of the shell points: a Fibonacci sphere
    double dirs[3 * MLP_SHELL];
    for (int k = 0; k < MLP_SHELL; k++) {
        const double ez = 1.0 - (2.0 * k + 1.0) / MLP_SHELL, er = std::sqrt(1.0 - ez * ez);
        const double az = k * (3.14159265358979323846 * (3.0 - std::sqrt(5.0)));
        dirs[3 * k] = er * std::cos(az);
        dirs[3 * k + 1] = er * std::sin(az);
        dirs[3 * k + 2] = ez;
    }
    if ((e = cudaMemcpy(m.dirs, dirs, sizeof dirs, cudaMemcpyHostToDevice))) return e;
    cudaMemset(m.adam_m, 0, sizeof(float) * MLP_NPARAM);
    cudaMemset(m.adam_v, 0, sizeof(float) * MLP_NPARAM);
    cudaMemset(m.loss, 0, sizeof(double) * 2);
    return cudaSuccess;
}

void mlp_free(Mlp &m)
{
    void *ps[] = {m.theta, m.grad, m.adam_m, m.adam_v, m.W1b, m.W2b, m.W3b, m.X, m.H1, m.H2,
                  m.dZ1, m.dZ2, m.dYb, m.Y, m.dY, m.loss_part, m.loss, m.dirs};
    for (void *p : ps) cudaFree(p);
    m = Mlp();
}

void mlp_refresh(const Mlp &m, cudaStream_t st)
{
    k_refresh<<<(MLP_HIDDEN * MLP_KIN + EW - 1) / EW, EW, 0, st>>>(m.theta, m.W1b, m.W2b, m.W3b);
}

cudaError_t mlp_forward(const Mlp &m, const float *X, int n, unsigned *status, cudaStream_t st)
{
    return mlp_launch(k_mlp_rows<false>, (n + NR - 1) / NR, ROW_THREADS, RowSmem::BYTES,
                      row_args(m, X, nullptr, nullptr, 0, n, status), st);
}

cudaError_t mlp_gradient(const Mlp &m, const float *X, const float *T, const long long *idx, long long row0, int n,
                         double *acc, unsigned *status, cudaStream_t st)
{
    const int tiles = (n + NR - 1) / NR;
    const RowArgs r = row_args(m, X, T, idx, row0, n, status);
    const cudaError_t e = mlp_launch(k_mlp_rows<true>, tiles, ROW_THREADS, RowSmem::BYTES, r, st);
    if (e != cudaSuccess) return e;
    GradArgs a;
    memset(&a, 0, sizeof a);
    a.n = n;
    a.Xb = m.X; a.H1 = m.H1; a.H2 = m.H2; a.dZ1 = m.dZ1; a.dZ2 = m.dZ2; a.dYb = m.dYb; a.dY = m.dY;
    a.grad = m.grad; a.loss_part = m.loss_part; a.parts = tiles; a.loss = m.loss; a.acc = acc;
    a.status = status; a.no_mma = r.no_mma; a.wait_limit = r.wait_limit;
    return mlp_launch(k_mlp_grads, GRAD_CTAS, MLP_THREADS, GradSmem::BYTES, a, st);
}

void mlp_adam(Mlp &m, double lr, cudaStream_t st)
{
    m.t += 1;
    const float c1 = (float)(1.0 - std::pow(0.9, (double)m.t));
    const float c2 = (float)(1.0 - std::pow(0.999, (double)m.t));
    launch_after(k_adam, (MLP_NPARAM + EW - 1) / EW, EW, 0, st, m.theta, m.grad, m.adam_m, m.adam_v, (float)lr, c1, c2,
                 m.W1b, m.W2b, m.W3b);
}

// ---------------------------------------------------------------------------
// shell sampling and the surrogate forces in the step
// ---------------------------------------------------------------------------
namespace {

// fields at point X (lattice units, wrapped) as the trilinear mean over the
// fluid corners of its cell, whose loads are issued together; false when no
// corner is fluid
template <class R>
__device__ __forceinline__ bool interp_fluid(const Lattice &L, const InstDev &I, const double *X, double *phi, double *u)
{
    const int n3[3] = {I.nx, I.ny, I.nz};
    int lo[3], hi[3];
    double f[3];
    for (int a = 0; a < 3; a++) {
        const int b = (int)floor(X[a]);
        f[a] = X[a] - b;
        lo[a] = b % n3[a];
        hi[a] = (b + 1) % n3[a];
    }
    const uint8_t *fli = L.flags + I.node_off;
    const R *ph = (const R *)L.phi + I.node_off;
    const R *U = (const R *)L.u + I.node_off;
    uint8_t fl[8];
    R p[8], v[3][8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const int n = ((k & 4 ? hi[2] : lo[2]) * I.ny + (k & 2 ? hi[1] : lo[1])) * I.nx + (k & 1 ? hi[0] : lo[0]);
        fl[k] = fli[n];
        p[k] = ph[n];
        for (int a = 0; a < 3; a++) v[a][k] = U[a * L.Ntot + n];
    }
    double ap = 0.0, au[3] = {0.0, 0.0, 0.0}, ws = 0.0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        if ((fl[k] & OWNER_MASK) != OWN_FLUID) continue;
        const double w = (k & 1 ? f[0] : 1.0 - f[0]) * (k & 2 ? f[1] : 1.0 - f[1]) * (k & 4 ? f[2] : 1.0 - f[2]);
        ap = ap + w * (double)p[k];
        for (int a = 0; a < 3; a++) au[a] = au[a] + w * (double)v[a][k];
        ws += w;
    }
    if (ws <= 0.0) return false;
    *phi = ap / ws;
    for (int a = 0; a < 3; a++) u[a] = au[a] / ws;
    return true;
}

// features of particles p0..p0+gridDim.x-1: 96 shell points (one thread
// each, directions from the table), then cos(theta), sin(theta), R/R_ref
template <class R>
__global__ void __launch_bounds__(MLP_SHELL + 32) k_shell(Lattice L, int p0, const double *dirs, float *feat)
{
    const int p = p0 + blockIdx.x;
    const PartDev &P = L.parts[p];
    const InstDev &I = L.inst[P.inst];
    float *f = feat + (long long)blockIdx.x * MLP_NIN;
    const int k = threadIdx.x;
    if (k < MLP_SHELL) {
        const double e[3] = {dirs[3 * k], dirs[3 * k + 1], dirs[3 * k + 2]};
        const double rs = P.R + I.sh_gap;
        const int n3[3] = {I.nx, I.ny, I.nz};
        double lev[3];
        for (int a = 0; a < 3; a++) lev[a] = rs * e[a];
        // with a box filter (width sh_box) the mean over the 3 x 3 x 3 points
        // of the box, offsets -w/3, 0, +w/3 per axis, of those whose cell has
        // a fluid corner (the midpoint rule of the box average); with a wall
        // at z = 0 a point outside [0, nz) in z lies in or beyond the wall and
        // is left out (no wrap across the wall)
        const int nsub = I.sh_box > 0.0 ? 27 : 1;
        double ph = 0.0, u[3] = {0.0, 0.0, 0.0};
        int used = 0;
        for (int s = 0; s < nsub; s++) {
            const double d[3] = {nsub == 1 ? 0.0 : (s % 3 - 1) * I.sh_box / 3.0,
                                 nsub == 1 ? 0.0 : ((s / 3) % 3 - 1) * I.sh_box / 3.0,
                                 nsub == 1 ? 0.0 : (s / 9 - 1) * I.sh_box / 3.0};
            double X[3];
            bool in_wall = false;
            for (int a = 0; a < 3; a++) {
                const double v = P.x[a] + lev[a] + d[a];
                if (a == 2 && I.wall_z0 && !(v >= 0.0 && v < n3[2])) in_wall = true;
                // in [0, n) already, or one period off (the common cases), without a division
                X[a] = v >= 0.0 && v < n3[a] ? v
                                             : (v < 0.0 && v >= -n3[a] ? v + n3[a] : v - n3[a] * floor(v / n3[a]));
            }
            if (in_wall) continue;
            double p1 = 0.0, u1[3] = {0.0, 0.0, 0.0};
            if (!interp_fluid<R>(L, I, X, &p1, u1)) continue;
            ph += p1;
            for (int a = 0; a < 3; a++) u[a] += u1[a];
            used++;
        }
        float o[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (used > 0) {
            if (nsub > 1) {
                ph /= used;
                for (int a = 0; a < 3; a++) u[a] /= used;
            }
            const double us[3] = {P.v[0] + (P.w[1] * lev[2] - P.w[2] * lev[1]),
                                  P.v[1] + (P.w[2] * lev[0] - P.w[0] * lev[2]),
                                  P.v[2] + (P.w[0] * lev[1] - P.w[1] * lev[0])};
            o[0] = (float)ph;
            for (int a = 0; a < 3; a++) o[1 + a] = (float)((u[a] - us[a]) / I.sh_uref);
        }
        for (int a = 0; a < 4; a++) f[4 * k + a] = o[a];
    } else if (k == MLP_SHELL) {
        f[4 * MLP_SHELL] = (float)P.cos_t;
        f[4 * MLP_SHELL + 1] = (float)P.sin_t;
        f[4 * MLP_SHELL + 2] = (float)(P.R / I.sh_rref);
    }
}

// surrogate output -> fluid forces of the particles: F = sigma R_p y[0..2],
// T = sigma R_p^2 y[3..5]; the capillary share is folded into these
__global__ void k_surrogate_apply(Lattice L, const float *Y, int p0, int np)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= np) return;
    PartDev &P = L.parts[p0 + r];
    const double s = L.inst[P.inst].sigma * P.R;
    for (int a = 0; a < 3; a++) {
        P.Feta[a] = s * (double)Y[r * 16 + a];
        P.Teta[a] = s * P.R * (double)Y[r * 16 + 3 + a];
        P.Fsig[a] = 0.0;
        P.Tsig[a] = 0.0;
    }
}

}  // namespace

template <class S>
void launch_shell_features(const Lattice &L, const Mlp &m, int p0, int np, float *feat, cudaStream_t st)
{
    using R = typename Store<S>::real;
    k_shell<R><<<np, MLP_SHELL + 32, 0, st>>>(L, p0, m.dirs, feat);
}

template <class S>
void launch_surrogate_forces(const Lattice &L, const Mlp &m, float *feat, cudaStream_t st, long long *launches,
                             const Marker &mk)
{
    if (L.n_parts == 0) return;
    mk(STAGE_SURROGATE, 0);
    for (int p0 = 0; p0 < L.n_parts; p0 += m.cap) {
        const int np = std::min(m.cap, L.n_parts - p0);
        launch_shell_features<S>(L, m, p0, np, feat, st);
        // a failed set-up or launch stays in the runtime's last error, which
        // lbm_step checks after enqueueing the step
        if (mlp_forward(m, feat, np, L.status, st) != cudaSuccess) return;
        k_surrogate_apply<<<(np + 127) / 128, 128, 0, st>>>(L, m.Y, p0, np);
        *launches += 3;
    }
    mk(STAGE_SURROGATE, 1);
}

#define INST(S)                                                                                        \
    template void launch_shell_features<S>(const Lattice &, const Mlp &, int, int, float *, cudaStream_t); \
    template void launch_surrogate_forces<S>(const Lattice &, const Mlp &, float *, cudaStream_t, long long *, \
                                             const Marker &);
INST(double)
INST(float)
INST(__half)
INST(__nv_bfloat16)
#undef INST

}  // namespace lbmg
