// mlp.cu -- the network of the learned warm start: a multilayer perceptron
// 3 -> 256 -> 256 -> 256 -> 64 (tanh hidden units, linear output) that maps
// (theta_eq, R0, lambda) to the equilibrium radial profile g(phi) = G(phi)/R0
// of the droplet about its centre (App. B parametrisation, 64 polar samples),
// trained by mean squared error with Adam.  The paper has no network; this
// is the warm start that shortens the runs to equilibrium.
//
// Two kernels.  net_kernel takes 128 samples per cluster of eight CTAs
// through the whole forward pass and, when training, the loss and the
// backward pass; update_kernel forms the parameter gradients (sums over the
// batch) and applies Adam.  Their matrix products run on the
// fifth-generation tensor cores: BF16 operands in shared memory in the
// canonical core-matrix layouts (K-major, or MN-major where the operand is a
// transpose), tcgen05.mma issued by one thread, FP32 accumulators in tensor
// memory (TMEM) read back with tcgen05.ld for the fused epilogues.
// Parameters: FP32 master copy + BF16 copies of the three tensor-core weight
// matrices, refreshed by the update.
#include <math.h>
#include <string.h>

#include <cmath>

#include <algorithm>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/iblb.h"
#include "iblb_internal.h"
#include "mlp_exchange.h"

using namespace iblb;

namespace {

constexpr int NIN = 3, NH = 256, NOUT = 64;
constexpr int64_t NPARAM = (int64_t)NH * NIN + NH + 2 * ((int64_t)NH * NH + NH) + (int64_t)NOUT * NH + NOUT;
constexpr float BETA1 = 0.9f, BETA2 = 0.999f, ADAM_EPS = 1e-8f;

// ----------------------------------------------------------------- tcgen05
constexpr int TC_M = 128;            // rows of one tcgen05.mma (samples, or units of a weight gradient)
constexpr int THREADS = 256;         // update kernel: warp w reads TMEM lanes 32 (w mod 4) .., columns of half w / 4
constexpr int NET_THREADS = 512;     // forward / backward kernel: columns of quarter w / 4
constexpr int CLUSTER = EX_CTAS;     // CTAs per 128 samples
constexpr int UNITS = NH / CLUSTER;
constexpr int OUT_CTAS = EX_OUT, OUT_UNITS = NOUT / OUT_CTAS;   // the output layer: 16 units on each of four CTAs
static_assert(EX_H1.units == UNITS && EX_DY.units == OUT_UNITS, "pieces of a layer");
constexpr long long TC_WAIT_CYCLES = 1000000000LL;   // ~0.5 s: bounded barrier wait

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor (tcgen05), no swizzle: start address,
// leading byte offset, stride byte offset, all in 16-byte units; descriptor
// version 1 at bits 46-47.  An operand is staged as 8 x 8 core matrices of
// 128 contiguous bytes (8 rows of 16 bytes).  K-major: a core matrix holds
// 8 rows of 8 elements along K; LBO = bytes between core matrices adjacent in
// K, SBO = between 8-row groups.  MN-major: a core matrix holds 8 values of K
// with 8 elements along M or N each; SBO = bytes between core matrices
// adjacent in M or N, LBO = between groups of 8 along K.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// Instruction descriptor of kind::f16: D in F32, A and B in BF16, MN-major
// flags at bits 15 (A) and 16 (B), N >> 3 at bits 17-22, M >> 4 at bits 24-28.
__device__ __forceinline__ uint32_t instr_desc(int N, bool a_mn, bool b_mn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}

// a staged operand: shared address, descriptor offsets, bytes per K = 16 step
struct Operand {
    uint32_t addr, lbo, sbo, step;
};
// K-major, row groups `sbo` apart (8 core matrices of K per 1024 bytes)
__device__ __forceinline__ Operand k_major(const void *p, uint32_t sbo) { return {smem_addr(p), 128, sbo, 256}; }
// activations: K-major with the 16 row groups of a K group adjacent (2048
// bytes per K group), so that a CTA's units are one contiguous piece
constexpr uint32_t A_KGROUP = TC_M * 16;
__device__ __forceinline__ Operand activations(const void *p) { return {smem_addr(p), A_KGROUP, 128, 2 * A_KGROUP}; }
// MN-major with mn elements along M or N
__device__ __forceinline__ Operand mn_major(const void *p, int mn)
{
    return {smem_addr(p), (uint32_t)mn * 16, 128, (uint32_t)mn * 32};
}

// D (+)= A . B over ksteps K = 16 steps; completion arrives on bar
__device__ __forceinline__ void issue_mma(uint32_t tmem, Operand A, Operand B, int ksteps, uint32_t idesc,
                                          bool accumulate, uint64_t *bar)
{
    for (int s = 0; s < ksteps; ++s) {
        const uint64_t ad = smem_desc(A.addr + s * A.step, A.lbo, A.sbo);
        const uint64_t bd = smem_desc(B.addr + s * B.step, B.lbo, B.sbo);
        const uint32_t acc = (accumulate || s > 0) ? 1u : 0u;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
            : "memory");
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity)
{
    const long long t0 = clock64();
    while (true) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_addr(bar)), "r"(parity)
            : "memory");
        if (ok)
            return true;
        if (clock64() - t0 > TC_WAIT_CYCLES)
            return false;
    }
}

// 8 / 4 accumulator columns of the thread's row, from column c0
__device__ __forceinline__ void read_acc(uint32_t tmem, int c0, float (&v)[8])
{
    const uint32_t a = tmem + ((threadIdx.x & 96u) << 16) + (uint32_t)c0;
    uint32_t r[8];
    __syncwarp();
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(a)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int e = 0; e < 8; ++e)
        v[e] = __uint_as_float(r[e]);
}
__device__ __forceinline__ void read_acc(uint32_t tmem, int c0, float (&v)[4])
{
    const uint32_t a = tmem + ((threadIdx.x & 96u) << 16) + (uint32_t)c0;
    uint32_t r[4];
    __syncwarp();
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int e = 0; e < 4; ++e)
        v[e] = __uint_as_float(r[e]);
}

// 16 bytes to shared memory asynchronously; zeros when !valid (src is not read)
__device__ __forceinline__ void cp16(void *dst, const void *src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// `rows` rows of 256 BF16 (row-major) as a K-major operand, row groups 4096
// bytes apart: eight consecutive lanes write one core matrix (no bank
// conflicts) and a warp reads 64-byte pieces of eight rows
__device__ __forceinline__ void stage_k_major(uint8_t *dst, const __nv_bfloat16 *src, int rows)
{
    for (int v = threadIdx.x; v < rows * 32; v += NET_THREADS) {
        const int r = (v >> 8) * 8 + (v & 7), kg = (v >> 3) & 31;
        cp16(dst + (r >> 3) * 4096 + kg * 128 + (r & 7) * 16, src + (int64_t)r * NH + kg * 8, true);
    }
}
// columns 0 .. mn - 1 of `nk` rows (row length ld) as an MN-major operand:
// row = index along K; rows at or beyond k_valid and columns at or beyond
// mn_valid read as zero.  mn: 16, 32 or 128
template <int NT>
__device__ __forceinline__ void stage_mn_major(uint8_t *dst, const __nv_bfloat16 *src, int64_t ld, int nk, int mn,
                                               int k_valid, int mn_valid)
{
    const int vecs = mn >> 3, shift = vecs == 16 ? 4 : (vecs == 4 ? 2 : 1);
    for (int v = threadIdx.x; v < nk * vecs; v += NT) {
        const int k = (v >> (3 + shift)) * 8 + (v & 7), j = (v >> 3) & (vecs - 1);
        const bool ok = k < k_valid && j * 8 < mn_valid;
        cp16(dst + (k >> 3) * mn * 16 + j * 128 + (k & 7) * 16, src + (ok ? k * ld + j * 8 : 0), ok);
    }
}

// all threads of all CTAs of the cluster
__device__ __forceinline__ void cluster_arrive()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// the thread's row of an activation operand, from K column k0
__device__ __forceinline__ uint8_t *row_at(uint8_t *buf, int k0)
{
    const int r = threadIdx.x & 127;
    return buf + (k0 >> 3) * A_KGROUP + (r >> 3) * 128 + (r & 7) * 16 + (k0 & 7) * 2;
}
// `bytes` at `src` to the same place in CTA c of the cluster; their arrival
// counts on the same mbarrier there
__device__ __forceinline__ void send(const uint8_t *src, uint32_t bytes, uint64_t *bar, int c)
{
    uint32_t dst, rbar;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(smem_addr(src)), "r"(c));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rbar) : "r"(smem_addr(bar)), "r"(c));
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "r"(smem_addr(src)), "r"(bytes), "r"(rbar)
                 : "memory");
}

__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a)) |
           ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(b)) << 16);
}
__device__ __forceinline__ float unpack(uint32_t w, int hi)
{
    return __bfloat162float(__ushort_as_bfloat16((unsigned short)(hi ? w >> 16 : w & 0xFFFFu)));
}
__device__ __forceinline__ uint4 pack8(const float (&v)[8])
{
    return make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
}
// n (a multiple of 4) floats at p, 16-byte aligned
template <int N>
__device__ __forceinline__ void load_floats(const float *p, float (&v)[N])
{
#pragma unroll
    for (int i = 0; i < N; i += 4) {
        const float4 q = *reinterpret_cast<const float4 *>(p + i);
        v[i] = q.x;
        v[i + 1] = q.y;
        v[i + 2] = q.z;
        v[i + 3] = q.w;
    }
}
template <int N>
__device__ __forceinline__ void store_floats(float *p, const float (&v)[N])
{
#pragma unroll
    for (int i = 0; i < N; i += 4)
        *reinterpret_cast<float4 *>(p + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
}

struct Net {
    int S;
    const float *x;              // raw inputs (theta_eq deg, R0, lambda); row idx[s] of sample s if idx
    const float *y;              // labels, same rows (training)
    const int *idx;
    const float *p;              // FP32 parameters
    const __nv_bfloat16 *W1b, *W2b, *W3b;
    float *yhat;                 // inference: S x 64
    float *u;                    // training: features S x 3, hidden activations and pre-activation gradients
    __nv_bfloat16 *h1, *h2, *h3, *d3b, *d2b, *dyb;
    float *d3, *d2, *d1, *dy, *sq;
    int *err;
};

// parameter offsets
constexpr int64_t OFF_W0 = 0, OFF_B0 = (int64_t)NH * NIN;
constexpr int64_t OFF_W1 = OFF_B0 + NH, OFF_B1 = OFF_W1 + (int64_t)NH * NH;
constexpr int64_t OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + (int64_t)NH * NH;
constexpr int64_t OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + (int64_t)NOUT * NH;

// shared memory of net_kernel: two activation operands (128 x 256, K-major)
// and this CTA's slices of the weights
constexpr int A_BYTES = TC_M * NH * 2, SLICE_BYTES = UNITS * NH * 2;
constexpr int OFF_SA = 0, OFF_SW1 = 2 * A_BYTES, OFF_SW2 = OFF_SW1 + SLICE_BYTES, OFF_SW3 = OFF_SW2 + SLICE_BYTES;
constexpr int FWD_SMEM = OFF_SW3 + OUT_UNITS * NH * 2;
constexpr int OFF_TW3 = FWD_SMEM, OFF_TW2 = OFF_TW3 + NOUT * UNITS * 2, OFF_TW1 = OFF_TW2 + SLICE_BYTES;
constexpr int TRAIN_SMEM = OFF_TW1 + SLICE_BYTES;
static_assert(TRAIN_SMEM <= 226 * 1024, "shared memory of one CTA");

// Forward pass (and with TRAIN the loss and the backward pass) of 128
// samples per cluster.  A layer's product needs every unit of the previous
// layer, so each CTA writes its 32 units' outputs into its own operand buffer
// and sends that 8 KB piece to the seven others (bulk copies between shared
// memories, counted on an mbarrier there): no launch, no pass through global
// memory and no cluster barrier stands between the layers.  Two buffers
// suffice with the senders and receivers of mlp_exchange.h, which shows that a
// CTA sends into a buffer only after every receiver's last product from it.
// What bounds it is the chain of copies, products and tanh epilogues (8 per
// thread), not a throughput: eight CTAs of 512 threads per 128 samples keep
// each link short, and everything a thread reads from global memory (weights'
// slices by asynchronous copies in the order of use, biases, labels) is
// requested before the first layer.
// Measured: a training step at batch 128 39 -> 32 us against stores into the
// other CTAs and a cluster barrier per layer; inference of 200 samples 38 us
// a call, 14 of them here (262 with four launches and three copies).
template <bool TRAIN>
__global__ void __cluster_dims__(CLUSTER, 1, 1) __launch_bounds__(NET_THREADS, 1) net_kernel(Net g)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t bar, full[2];     // a product is done; an operand buffer's pieces have arrived
    __shared__ uint32_t tslot;
    __shared__ int gave_up;                            // a wait of an earlier launch did
    uint8_t *sa[2] = {smem + OFF_SA, smem + OFF_SA + A_BYTES};
    const int cta = blockIdx.x & (CLUSTER - 1), m0 = (blockIdx.x / CLUSTER) * TC_M, n0 = cta * UNITS;
    const int warp = threadIdx.x >> 5, row = threadIdx.x & 127, quarter = threadIdx.x >> 7;
    const int s = m0 + row;
    const bool live = s < g.S;
    const int c0 = n0 + 8 * quarter;                        // the thread's 8 units of a hidden layer
    const int o0 = (cta & (OUT_CTAS - 1)) * OUT_UNITS + 4 * quarter;   // its 4 outputs (CTAs below OUT_CTAS)

    if (threadIdx.x == 0) {
        for (uint64_t *m : {&bar, &full[0], &full[1]})
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(m)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(smem_addr(&tslot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    cluster_arrive();    // waited for before the first write to another CTA
    griddep_wait();
    const int err = threadIdx.x == 0 ? *g.err : 0;
    float w0[24], b0[8], b1[8], b2[8], b3[4], f[3] = {0.f, 0.f, 0.f}, yl[4] = {0.f, 0.f, 0.f, 0.f};
    int src = 0;
    if (live)
        src = g.idx ? g.idx[s] : s;
    load_floats(g.p + OFF_W0 + NIN * c0, w0);
    load_floats(g.p + OFF_B0 + c0, b0);
    load_floats(g.p + OFF_B1 + c0, b1);
    load_floats(g.p + OFF_B2 + c0, b2);
    load_floats(g.p + OFF_B3 + o0, b3);
    stage_k_major(smem + OFF_SW1, g.W1b + n0 * NH, UNITS);
    cp_commit();
    stage_k_major(smem + OFF_SW2, g.W2b + n0 * NH, UNITS);
    cp_commit();
    if (cta < OUT_CTAS)
        stage_k_major(smem + OFF_SW3, g.W3b + cta * OUT_UNITS * NH, OUT_UNITS);
    cp_commit();
    if (TRAIN) {
        stage_mn_major<NET_THREADS>(smem + OFF_TW3, g.W3b + n0, NH, NOUT, UNITS, NOUT, UNITS);
        cp_commit();
        stage_mn_major<NET_THREADS>(smem + OFF_TW2, g.W2b + n0, NH, NH, UNITS, NH, UNITS);
        cp_commit();
        stage_mn_major<NET_THREADS>(smem + OFF_TW1, g.W1b + n0, NH, NH, UNITS, NH, UNITS);
        cp_commit();
    }
    if (live) {
        f[0] = g.x[3 * src];
        f[1] = g.x[3 * src + 1];
        f[2] = g.x[3 * src + 2];
        if (TRAIN)
            load_floats(g.y + (int64_t)src * NOUT + o0, yl);
    }
    constexpr Exchange h1 = EX_H1, h2 = EX_H2, h3 = EX_H3, dy = EX_DY, d3 = EX_D3, d2 = EX_D2;
    uint32_t parity = 0, fparity[2] = {0, 0};
    bool failed = false;
    uint32_t tmem = 0;
    // The CTA's piece of the exchange is written: make it and the staged
    // weights visible to the tensor core and the copies, order the
    // accumulator's readers before its next use, and send it to the receivers.
    // A CTA whose wait gave up sends no more: the others' waits for it give up
    // in turn, long after what they sent it has landed.
    auto publish = [&](const Exchange &x, bool first = false) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (first)
            failed = gave_up != 0;
        if (!failed && cta < x.senders && (int)threadIdx.x < x.receivers && (int)threadIdx.x != cta)
            send(sa[x.buffer] + (x.units * cta >> 3) * A_KGROUP, (uint32_t)(x.units >> 3) * A_KGROUP, &full[x.buffer],
                 threadIdx.x);
    };
    // a receiver's product of the exchange's buffer with B, once the other
    // senders' pieces are in
    auto product = [&](const Exchange &x, Operand B, int N, bool b_mn) {
        if (!failed && cta < x.receivers) {
            const int b = x.buffer, ksteps = x.senders * x.units / 16;
            const uint32_t bytes = (uint32_t)(x.senders - (cta < x.senders)) * (uint32_t)(x.units >> 3) * A_KGROUP;
            bool ok = true;
            if (threadIdx.x == 0) {
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&full[b])),
                             "r"(bytes)
                             : "memory");
                ok = mbar_wait_bounded(&full[b], fparity[b]);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (ok)
                    issue_mma(tmem, activations(sa[b]), B, ksteps, instr_desc(N, false, b_mn), false, &bar);
            }
            fparity[b] ^= 1u;
            ok = ok && mbar_wait_bounded(&bar, parity);
            parity ^= 1u;
            if (__syncthreads_or(!ok)) {
                failed = true;
                if (threadIdx.x == 0)
                    atomicExch(g.err, 1);
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
    };
    uint4 hk1, hk2, hk3, w;              // its activations, kept for the backward pass
    float v[8] = {};
    // the backward pass's dz = dh (1 - h^2)
    auto dtanh = [&](uint4 h) {
        const uint32_t q[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float hv = unpack(q[e >> 1], e & 1);
            v[e] = v[e] * (1.0f - hv * hv);
        }
    };
    auto store = [&](__nv_bfloat16 *o, uint4 h) {
        if (live)
            *reinterpret_cast<uint4 *>(o + (int64_t)s * NH + c0) = h;
    };
    auto store_f = [&](float *o) {
        if (live)
            store_floats(o + (int64_t)s * NH + c0, v);
    };

    // features and the input layer (K = 3) on the CUDA cores
    if (live) {
        f[0] = (f[0] - 90.0f) / 70.0f;
        f[1] = (f[1] - 16.0f) / 8.0f;
        f[2] = log10f(f[2]);
        if (TRAIN && cta == 0 && quarter == 0) {
            g.u[3 * s] = f[0];
            g.u[3 * s + 1] = f[1];
            g.u[3 * s + 2] = f[2];
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const float z = b0[e] + w0[3 * e] * f[0] + w0[3 * e + 1] * f[1] + w0[3 * e + 2] * f[2];
        v[e] = live ? tanhf(z) : 0.0f;
    }
    hk1 = pack8(v);
    *reinterpret_cast<uint4 *>(row_at(sa[0], c0)) = hk1;
    cp_wait<TRAIN ? 5 : 2>();
    if (threadIdx.x == 0)
        gave_up = err;
    cluster_wait();      // every CTA of the cluster runs: its shared memory and barriers may be written
    publish(h1, true);
    tmem = tslot;
    if (TRAIN)
        store(g.h1, hk1);
    // hidden layers 2 and 3
    product(h1, k_major(smem + OFF_SW1, 4096), UNITS, false);
    if (!failed)
        read_acc(tmem, 8 * quarter, v);
#pragma unroll
    for (int e = 0; e < 8; ++e)
        v[e] = tanhf(v[e] + b1[e]);
    hk2 = pack8(v);
    *reinterpret_cast<uint4 *>(row_at(sa[1], c0)) = hk2;
    cp_wait<TRAIN ? 4 : 1>();
    publish(h2);
    if (TRAIN)
        store(g.h2, hk2);
    product(h2, k_major(smem + OFF_SW2, 4096), UNITS, false);
    if (!failed)
        read_acc(tmem, 8 * quarter, v);
#pragma unroll
    for (int e = 0; e < 8; ++e)
        v[e] = tanhf(v[e] + b2[e]);
    hk3 = pack8(v);
    *reinterpret_cast<uint4 *>(row_at(sa[0], c0)) = hk3;
    cp_wait<TRAIN ? 3 : 0>();
    publish(h3);
    if (TRAIN)
        store(g.h3, hk3);
    // output layer, loss gradient 2 (yhat - y) / (S 64) and squared errors
    const bool out_cta = cta < OUT_CTAS;
    float o[4] = {}, q[4] = {};
    product(h3, k_major(smem + OFF_SW3, 4096), OUT_UNITS, false);
    if (out_cta) {
        if (!failed)
            read_acc(tmem, 4 * quarter, o);
#pragma unroll
        for (int e = 0; e < 4; ++e)
            o[e] = o[e] + b3[e];
        if (!TRAIN && live)
            store_floats(g.yhat + (int64_t)s * NOUT + o0, o);
    }
    if constexpr (TRAIN) {
        uint2 t = make_uint2(0, 0);
        if (out_cta) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float d = live ? o[e] - yl[e] : 0.0f;
                o[e] = 2.0f * d / (float)(g.S * NOUT);
                q[e] = d * d;
            }
            t = make_uint2(pack2(o[0], o[1]), pack2(o[2], o[3]));
            *reinterpret_cast<uint2 *>(row_at(sa[1], o0)) = t;
        }
        cp_wait<2>();
        publish(dy);
        if (live && out_cta) {
            *reinterpret_cast<uint2 *>(g.dyb + (int64_t)s * NOUT + o0) = t;
            store_floats(g.dy + (int64_t)s * NOUT + o0, o);
            store_floats(g.sq + (int64_t)s * NOUT + o0, q);
        }
        // d3 = (dy W3) (1 - h3^2)
        product(dy, mn_major(smem + OFF_TW3, UNITS), UNITS, true);
        if (!failed)
            read_acc(tmem, 8 * quarter, v);
        dtanh(hk3);
        w = pack8(v);
        *reinterpret_cast<uint4 *>(row_at(sa[0], c0)) = w;
        cp_wait<1>();
        publish(d3);
        store_f(g.d3);
        store(g.d3b, w);
        // d2 = (d3 W2) (1 - h2^2)
        product(d3, mn_major(smem + OFF_TW2, UNITS), UNITS, true);
        if (!failed)
            read_acc(tmem, 8 * quarter, v);
        dtanh(hk2);
        w = pack8(v);
        *reinterpret_cast<uint4 *>(row_at(sa[1], c0)) = w;
        cp_wait<0>();
        publish(d2);
        store_f(g.d2);
        store(g.d2b, w);
        // d1 = (d2 W1) (1 - h1^2)
        product(d2, mn_major(smem + OFF_TW1, UNITS), UNITS, true);
        if (!failed)
            read_acc(tmem, 8 * quarter, v);
        dtanh(hk1);
        store_f(g.d1);
    }
    cluster_arrive();    // no CTA leaves while its pieces are read or its buffers written
    cluster_wait();
    if (failed) {   // give MMAs and copies still in flight a bounded chance to finish before TMEM and shared memory go
        mbar_wait_bounded(&bar, parity ^ 1u);
        if (threadIdx.x == 0)
            for (int b = 0; b < 2; ++b)
                mbar_wait_bounded(&full[b], fparity[b] ^ 1u);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(tmem) : "memory");
    }
}

struct Update {
    int S;
    const __nv_bfloat16 *h1, *h2, *h3, *d3b, *d2b, *dyb;
    const float *d3, *d2, *d1, *dy, *u, *sq;
    double *loss;
    float *grad;                 // gradient out (adam false)
    bool adam;
    float *p, *m, *v;
    __nv_bfloat16 *W1b, *W2b, *W3b;
    float lr, c1, c2;
    int *err;
};

// one Adam step of a parameter with gradient gi
__device__ __forceinline__ void adam(const Update &g, float gi, float &p, float &m, float &v)
{
    m = BETA1 * m + (1.0f - BETA1) * gi;
    v = BETA2 * v + (1.0f - BETA2) * gi * gi;
    p = p - g.lr * (m / g.c1) / (sqrtf(v / g.c2) + ADAM_EPS);
}

constexpr int UP_N = 16;                             // columns of a weight gradient per CTA
constexpr int UP_K = 256;                            // samples staged at a time
constexpr int UP_A = TC_M * UP_K * 2, UP_B = UP_N * UP_K * 2;
constexpr int TILES = NH / UP_N;                     // CTAs per 128 rows of a weight gradient
constexpr int UP_GEMM = 5 * TILES;                   // dW2 (two row tiles), dW1 (two), dW3
constexpr int UP_RED = (NOUT + 3 * NH) / 32;         // 32 units per CTA: bias gradients (and dW0)
constexpr int UP_BLOCKS = UP_GEMM + UP_RED + 1;      // and the loss

// Weight gradient tile dW(o, i) = sum_s dz(s, o) h(s, i): both operands are
// stored sample-major, so they are staged MN-major as they are; the samples
// run along K in order, UP_K at a time through two buffers.
__device__ __forceinline__ void weight_grad(const Update &g, uint8_t *smem, uint64_t *bar, uint32_t *tslot, int *gave_up)
{
    const int t = blockIdx.x / TILES, n0 = (blockIdx.x % TILES) * UP_N;
    const __nv_bfloat16 *A = t < 2 ? g.d3b : (t < 4 ? g.d2b : g.dyb);
    const __nv_bfloat16 *B = t < 2 ? g.h2 : (t < 4 ? g.h1 : g.h3);
    const int64_t off = t < 2 ? OFF_W2 : (t < 4 ? OFF_W1 : OFF_W3);
    __nv_bfloat16 *Wb = t < 2 ? g.W2b : (t < 4 ? g.W1b : g.W3b);
    const int m0 = t < 4 ? (t & 1) * TC_M : 0, rows = t < 4 ? TC_M : NOUT, lda = t < 4 ? NH : NOUT;
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(smem_addr(tslot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    griddep_wait();
    const int err = threadIdx.x == 0 ? *g.err : 0;
    const int chunks = (g.S + UP_K - 1) / UP_K;
    // the thread's 8 parameters and moments, in flight with the operands
    const int row = threadIdx.x & 127, c0 = 8 * (threadIdx.x >> 7);
    const int64_t o = (int64_t)(m0 + row) * NH + n0 + c0;
    const bool mine = row < rows;
    float pn[8] = {}, mn[8] = {}, vn[8] = {};
    if (g.adam && mine) {
        load_floats(g.p + off + o, pn);
        load_floats(g.m + off + o, mn);
        load_floats(g.v + off + o, vn);
    }
    auto stage = [&](int c) {
        uint8_t *sa = smem + (c & 1) * (UP_A + UP_B), *sb = sa + UP_A;
        const int k0 = c * UP_K, kn = min(UP_K, g.S - k0), nk = (kn + 15) & ~15;
        stage_mn_major<THREADS>(sa, A + (int64_t)k0 * lda + m0, lda, nk, TC_M, kn, rows);
        stage_mn_major<THREADS>(sb, B + (int64_t)k0 * NH + n0, NH, nk, UP_N, kn, UP_N);
        cp_commit();
    };
    stage(0);
    if (threadIdx.x == 0)
        *gave_up = err;
    uint32_t tmem = 0, parity = 0;
    bool failed = false;
    for (int c = 0; c < chunks; ++c) {
        cp_wait<0>();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem = *tslot;
        if (*gave_up) {
            failed = true;
            break;
        }
        const uint8_t *sa = smem + (c & 1) * (UP_A + UP_B), *sb = sa + UP_A;
        if (threadIdx.x == 0)
            issue_mma(tmem, mn_major(sa, TC_M), mn_major(sb, UP_N), (min(UP_K, g.S - c * UP_K) + 15) / 16,
                      instr_desc(UP_N, true, true), c > 0, bar);
        if (c + 1 < chunks)
            stage(c + 1);        // its buffer's products finished one iteration ago
        const bool ok = mbar_wait_bounded(bar, parity);
        parity ^= 1u;
        if (__syncthreads_or(!ok)) {
            failed = true;
            if (threadIdx.x == 0)
                atomicExch(g.err, 1);
            break;
        }
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (failed) {
        cp_wait<0>();
        mbar_wait_bounded(bar, parity ^ 1u);
    } else {
        float acc[8];
        read_acc(tmem, c0, acc);
        if (mine && g.adam) {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                adam(g, acc[e], pn[e], mn[e], vn[e]);
            store_floats(g.p + off + o, pn);
            store_floats(g.m + off + o, mn);
            store_floats(g.v + off + o, vn);
            *reinterpret_cast<uint4 *>(Wb + o) = pack8(pn);
        } else if (mine) {
            store_floats(g.grad + off + o, acc);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(tmem) : "memory");
    }
}

// Sums over the batch for 32 units: slot l of 32 adds samples l, l + 32, ...
// in order and the slots meet in a fixed tree.  A warp takes four slots of
// the 32 units (128-byte reads), their loads in flight together.  dz: S x ld
// from the first unit; U: with the features u, the input layer's weight
// gradient too.
template <bool U>
__device__ __forceinline__ void unit_sums(const Update &g, const float *dz, int ld, int64_t off_b, int unit0,
                                          float (*sh)[32][33], int *gave_up)
{
    constexpr int NV = U ? 1 + NIN : 1;
    const int err = threadIdx.x == 0 ? *g.err : 0;
    const int o = threadIdx.x & 31, w = threadIdx.x >> 5;
    // the parameter that this thread updates: value w of unit o
    const bool mine = w < NV;
    const int64_t i = w == 0 ? off_b + unit0 + o : OFF_W0 + NIN * (unit0 + o) + (w - 1);
    float p = 0.f, m = 0.f, v = 0.f;
    if (mine && g.adam) {
        p = g.p[i];
        m = g.m[i];
        v = g.v[i];
    }
    float acc[4][NV] = {};
    for (int s0 = 0; s0 < g.S; s0 += 32) {
        float d[4], u[4][NIN];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int s = s0 + 4 * w + q;
            d[q] = s < g.S ? dz[(int64_t)s * ld + unit0 + o] : 0.0f;
            if (U)
                for (int k = 0; k < NIN; ++k)
                    u[q][k] = s < g.S ? g.u[3 * s + k] : 0.0f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (s0 + 4 * w + q >= g.S)
                continue;
            acc[q][0] += d[q];
            if (U)
                for (int k = 0; k < NIN; ++k)
                    acc[q][1 + k] += d[q] * u[q][k];
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        for (int k = 0; k < NV; ++k)
            sh[k][4 * w + q][o] = acc[q][k];
    if (threadIdx.x == 0)
        *gave_up = err;
    __syncthreads();
    if (!mine || *gave_up)
        return;
    float t[32];
#pragma unroll
    for (int l = 0; l < 32; ++l)
        t[l] = sh[w][l][o];
#pragma unroll
    for (int h = 16; h >= 1; h >>= 1)
#pragma unroll
        for (int l = 0; l < h; ++l)
            t[l] += t[l + h];
    if (!g.adam) {
        g.grad[i] = t[0];
        return;
    }
    adam(g, t[0], p, m, v);
    g.p[i] = p;
    g.m[i] = m;
    g.v[i] = v;
}

// Every parameter's gradient (sums over the batch) and its Adam step, and
// the loss: CTAs [0, UP_GEMM) one 128 x 16 tile of a weight matrix each on
// the tensor cores, the next 32 units' biases each (with the input layer's
// weights), the last the loss.  Small tiles because the time of a CTA is its
// loads and its divisions: 107 CTAs share both.  Once a wait of the net kernel
// (or of an earlier update) gave up, nothing is updated any more: what the
// gradients would be formed from is not there.  Measured: an Adam step at
// batch 128 766 -> 32 us (15 launches before), 10 of them here.
__global__ void __launch_bounds__(THREADS, 1) update_kernel(Update g)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tslot;
    __shared__ int gave_up;
    if (blockIdx.x < UP_GEMM) {
        weight_grad(g, smem, &bar, &tslot, &gave_up);
        return;
    }
    griddep_wait();
    const int b = blockIdx.x - UP_GEMM;
    float(*sh)[32][33] = reinterpret_cast<float(*)[32][33]>(smem);
    if (b < NOUT / 32) {
        unit_sums<false>(g, g.dy, NOUT, OFF_B3, 32 * b, sh, &gave_up);
    } else if (b < UP_RED) {
        const int k = b - NOUT / 32, layer = k / (NH / 32), u0 = 32 * (k % (NH / 32));
        if (layer == 0)
            unit_sums<false>(g, g.d3, NH, OFF_B2, u0, sh, &gave_up);
        else if (layer == 1)
            unit_sums<false>(g, g.d2, NH, OFF_B1, u0, sh, &gave_up);
        else
            unit_sums<true>(g, g.d1, NH, OFF_B0, u0, sh, &gave_up);
    } else {     // loss = mean of the squared errors, FP64, fixed order
        double *red = reinterpret_cast<double *>(smem);
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        const int64_t n = (int64_t)g.S * NOUT;
#pragma unroll 4
        for (int64_t k = 4 * threadIdx.x; k < n; k += 4 * THREADS) {     // n is a multiple of 4
            const float4 q = *reinterpret_cast<const float4 *>(g.sq + k);
            a[0] += (double)q.x;
            a[1] += (double)q.y;
            a[2] += (double)q.z;
            a[3] += (double)q.w;
        }
        red[threadIdx.x] = (a[0] + a[1]) + (a[2] + a[3]);
        for (int h = THREADS / 2; h >= 1; h >>= 1) {
            __syncthreads();
            if (threadIdx.x < h)
                red[threadIdx.x] += red[threadIdx.x + h];
        }
        if (threadIdx.x == 0)
            *g.loss = red[0] / ((double)g.S * NOUT);
    }
}

__global__ void to_bf16_kernel(const float *src, __nv_bfloat16 *dst, int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        dst[i] = __float2bfloat16_rn(src[i]);
}

constexpr int HEAD = 64;             // floats before the outputs: the error flag, padded to 256 bytes
constexpr int ROWS_OUT = 4096;       // outputs brought to the host at a time, at most

inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

struct iblb_mlp {
    cudaStream_t stream = nullptr;
    int max_batch = 0;
    int64_t t = 0;                       // Adam steps taken
    void *slab = nullptr;                // one allocation holds every array below that max_batch sizes
    // parameters
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    __nv_bfloat16 *W1b = nullptr, *W2b = nullptr, *W3b = nullptr;
    // activations (max_batch rows)
    float *u = nullptr, *yhat = nullptr, *dy = nullptr, *sq = nullptr;
    float *d3 = nullptr, *d2 = nullptr, *d1 = nullptr;
    __nv_bfloat16 *h1 = nullptr, *h2 = nullptr, *h3 = nullptr, *dyb = nullptr, *d3b = nullptr, *d2b = nullptr;
    int *err = nullptr;                  // HEAD floats before yhat, so that one copy brings both to the host
    // samples and their order, and the loss of each batch of an epoch (grown on demand)
    float *x = nullptr, *y = nullptr;
    int *idx = nullptr;
    double *loss = nullptr;
    int64_t data_cap = 0, idx_cap = 0, loss_cap = 0;
    float *h_out = nullptr;              // pinned: HEAD + 64 rows_out floats
    int rows_out = 0;
    std::string msg;
};

namespace {

thread_local std::string g_mlp_error;

int mfail(iblb_mlp *m, int code, const std::string &s)
{
    if (m)
        m->msg = s;
    else
        g_mlp_error = s;
    return code;
}

#define MCK(call)                                                                              \
    do {                                                                                       \
        cudaError_t e_ = (call);                                                               \
        if (e_ != cudaSuccess)                                                                 \
            return mfail(m, IBLB_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));  \
    } while (0)

// forward pass of S rows of x (device, raw inputs): outputs into mm->yhat
cudaError_t forward(iblb_mlp *mm, const float *x, int S)
{
    Net g{};
    g.S = S;
    g.x = x;
    g.p = mm->p;
    g.W1b = mm->W1b;
    g.W2b = mm->W2b;
    g.W3b = mm->W3b;
    g.yhat = mm->yhat;
    g.err = mm->err;
    return launch_k(net_kernel<false>, dim3(nblk(S, TC_M) * CLUSTER), dim3(NET_THREADS), FWD_SMEM, mm->stream, true,
                    g);
}

// Forward and backward pass of S samples (rows idx[s] of x and y if idx) and
// the mean squared error into *loss; then the gradient into mm->g, or with
// lr > 0 one Adam step with the bias corrections c1 and c2.
cudaError_t train_step(iblb_mlp *mm, const float *x, const float *y, const int *idx, int S, double *loss, float lr,
                       float c1, float c2)
{
    const Net n{S, x, y, idx, mm->p, mm->W1b, mm->W2b, mm->W3b, nullptr, mm->u, mm->h1, mm->h2, mm->h3, mm->d3b,
                mm->d2b, mm->dyb, mm->d3, mm->d2, mm->d1, mm->dy, mm->sq, mm->err};
    cudaError_t e = launch_k(net_kernel<true>, dim3(nblk(S, TC_M) * CLUSTER), dim3(NET_THREADS), TRAIN_SMEM,
                             mm->stream, true, n);
    if (e != cudaSuccess)
        return e;
    const Update u{S, mm->h1, mm->h2, mm->h3, mm->d3b, mm->d2b, mm->dyb, mm->d3, mm->d2, mm->d1, mm->dy, mm->u,
                   mm->sq, loss, mm->g, lr > 0.0f, mm->p, mm->m, mm->v, mm->W1b, mm->W2b, mm->W3b, lr, c1, c2,
                   mm->err};
    return launch_k(update_kernel, dim3(UP_BLOCKS), dim3(THREADS), (S > UP_K ? 2 : 1) * (UP_A + UP_B), mm->stream,
                    true, u);
}

cudaError_t refresh_bf16(iblb_mlp *mm)
{
    to_bf16_kernel<<<nblk((int64_t)NH * NH, 256), 256, 0, mm->stream>>>(mm->p + OFF_W1, mm->W1b, (int64_t)NH * NH);
    to_bf16_kernel<<<nblk((int64_t)NH * NH, 256), 256, 0, mm->stream>>>(mm->p + OFF_W2, mm->W2b, (int64_t)NH * NH);
    to_bf16_kernel<<<nblk((int64_t)NOUT * NH, 256), 256, 0, mm->stream>>>(mm->p + OFF_W3, mm->W3b,
                                                                          (int64_t)NOUT * NH);
    return cudaGetLastError();
}

// the error flag as read into h_out[0]
int check_err(iblb_mlp *m)
{
    if (!*reinterpret_cast<const int *>(m->h_out))
        return IBLB_OK;
    MCK(cudaMemsetAsync(m->err, 0, sizeof(int), m->stream));
    return mfail(m, IBLB_E_TIMEOUT, "a bounded wait for the tensor-core MMAs gave up");
}

// *p holds at least n elements (its old contents are dropped when it grows)
template <typename T>
int grow(iblb_mlp *m, T **p, int64_t *cap, int64_t n)
{
    if (n <= *cap)
        return IBLB_OK;
    if (*p)
        MCK(cudaFree(*p));
    *p = nullptr;
    *cap = 0;
    MCK(cudaMalloc((void **)p, sizeof(T) * n));
    *cap = n;
    return IBLB_OK;
}

// x and y (may be null) to the device in FP32, through hx and hy, which stay
// as they are until the caller has synchronised the stream
int upload(iblb_mlp *m, const double *x, const double *y, int64_t S, std::vector<float> &hx, std::vector<float> &hy)
{
    if (S > m->data_cap) {
        int64_t cx = 0, cy = 0;
        m->data_cap = 0;
        int r = IBLB_OK;
        if (m->x)
            MCK(cudaFree(m->x));
        if (m->y)
            MCK(cudaFree(m->y));
        m->x = m->y = nullptr;
        if ((r = grow(m, &m->x, &cx, 3 * S)) || (r = grow(m, &m->y, &cy, (int64_t)NOUT * S)))
            return r;
        m->data_cap = S;
    }
    hx.resize(3 * S);
    hy.resize(y ? NOUT * S : 0);
    for (int64_t i = 0; i < 3 * S; ++i)
        hx[i] = (float)x[i];
    for (int64_t i = 0; i < (int64_t)hy.size(); ++i)
        hy[i] = (float)y[i];
    MCK(cudaMemcpyAsync(m->x, hx.data(), sizeof(float) * hx.size(), cudaMemcpyHostToDevice, m->stream));
    if (y)
        MCK(cudaMemcpyAsync(m->y, hy.data(), sizeof(float) * hy.size(), cudaMemcpyHostToDevice, m->stream));
    return IBLB_OK;
}

bool inputs_valid(const double *x, int64_t S)
{
    for (int64_t s = 0; s < S; ++s)
        if (!(x[3 * s + 2] > 0.0) || !std::isfinite(x[3 * s]) || !std::isfinite(x[3 * s + 1]))
            return false;
    return true;
}

uint64_t splitmix(uint64_t &s)
{
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

}  // namespace

extern "C" {

int64_t iblb_mlp_param_count(void) { return NPARAM; }

const char *iblb_mlp_last_error(const iblb_mlp *m) { return m ? m->msg.c_str() : g_mlp_error.c_str(); }

int iblb_mlp_create(const float *params, int64_t n_params, int max_batch, void *stream, iblb_mlp **out)
{
    iblb_mlp *m = nullptr;
    if (!params || !out || n_params != NPARAM || max_batch < 1 || max_batch > (1 << 20))
        return mfail(nullptr, IBLB_E_ARG,
                     "iblb_mlp_create: need " + std::to_string(NPARAM) + " parameters and 1 <= max_batch <= 2^20");
    for (int64_t i = 0; i < n_params; ++i)
        if (!std::isfinite(params[i]))
            return mfail(nullptr, IBLB_E_ARG, "iblb_mlp_create: non-finite parameter");
    m = new iblb_mlp();
    m->stream = (cudaStream_t)stream;
    m->max_batch = max_batch;
    const int64_t B = max_batch;
    // two passes: sizes, then the arrays' places in the slab (256-byte aligned)
    char *base = nullptr;
    int64_t at = 0;
    auto place = [&](auto **p, int64_t n) {
        if (base)
            *p = reinterpret_cast<std::remove_reference_t<decltype(*p)>>(base + at);
        at += (int64_t)((n * sizeof(**p) + 255) & ~(size_t)255);
    };
    auto place_all = [&]() {
        at = 0;
        for (float **q : {&m->p, &m->g, &m->m, &m->v})
            place(q, NPARAM);
        place(&m->W1b, (int64_t)NH * NH);
        place(&m->W2b, (int64_t)NH * NH);
        place(&m->W3b, (int64_t)NOUT * NH);
        place(&m->u, 3 * B);
        place(&m->err, HEAD);            // directly before yhat
        for (float **q : {&m->yhat, &m->dy, &m->sq})
            place(q, NOUT * B);
        for (float **q : {&m->d3, &m->d2, &m->d1})
            place(q, NH * B);
        for (__nv_bfloat16 **q : {&m->h1, &m->h2, &m->h3, &m->d3b, &m->d2b})
            place(q, NH * B);
        place(&m->dyb, NOUT * B);
    };
    static_assert(HEAD * sizeof(float) == 256, "the outputs follow the flag");
    place_all();
    cudaError_t e = cudaMalloc(&m->slab, (size_t)at);
    if (!e) {
        base = (char *)m->slab;
        place_all();
    }
    m->rows_out = std::min(max_batch, ROWS_OUT);
    if (!e) e = cudaMallocHost((void **)&m->h_out, sizeof(float) * (HEAD + (size_t)NOUT * m->rows_out));
    if (!e) e = cudaFuncSetAttribute(net_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, FWD_SMEM);
    if (!e) e = cudaFuncSetAttribute(net_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TRAIN_SMEM);
    if (!e) e = cudaFuncSetAttribute(update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * (UP_A + UP_B));
    if (!e) e = cudaMemcpyAsync(m->p, params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, m->stream);
    if (!e) e = cudaMemsetAsync(m->m, 0, sizeof(float) * NPARAM, m->stream);
    if (!e) e = cudaMemsetAsync(m->v, 0, sizeof(float) * NPARAM, m->stream);
    if (!e) e = cudaMemsetAsync(m->err, 0, sizeof(int), m->stream);
    if (!e) e = refresh_bf16(m);
    if (!e) e = cudaStreamSynchronize(m->stream);
    if (e) {
        std::string s = std::string("iblb_mlp_create: ") + cudaGetErrorString(e);
        iblb_mlp_destroy(m);
        return mfail(nullptr, e == cudaErrorMemoryAllocation ? IBLB_E_NOMEM : IBLB_E_CUDA, s);
    }
    *out = m;
    return IBLB_OK;
}

void iblb_mlp_destroy(iblb_mlp *m)
{
    if (!m)
        return;
    for (void *p : {m->slab, (void *)m->x, (void *)m->y, (void *)m->idx, (void *)m->loss})
        if (p)
            cudaFree(p);
    if (m->h_out)
        cudaFreeHost(m->h_out);
    delete m;
}

int iblb_mlp_get_params(iblb_mlp *m, float *out, int64_t n)
{
    if (!m || !out || n != NPARAM)
        return mfail(m, IBLB_E_ARG, "iblb_mlp_get_params: bad arguments");
    MCK(cudaMemcpyAsync(out, m->p, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, m->stream));
    MCK(cudaStreamSynchronize(m->stream));
    return IBLB_OK;
}

int iblb_selftest_mlp_give_up(iblb_mlp *m)
{
    if (!m)
        return mfail(m, IBLB_E_ARG, "iblb_selftest_mlp_give_up: null network");
    MCK(cudaMemsetAsync(m->err, 1, 1, m->stream));
    MCK(cudaStreamSynchronize(m->stream));
    return IBLB_OK;
}

int iblb_mlp_predict(iblb_mlp *m, const double *x, int S, double *y)
{
    if (!m || !x || !y || S < 1)
        return mfail(m, IBLB_E_ARG, "iblb_mlp_predict: bad arguments");
    if (!inputs_valid(x, S))
        return mfail(m, IBLB_E_ARG, "iblb_mlp_predict: inputs need finite theta_eq, R0 and lambda > 0");
    std::vector<float> hx, hy;
    int r = upload(m, x, nullptr, S, hx, hy);
    if (r)
        return r;
    for (int s0 = 0; s0 < S; s0 += m->max_batch) {
        const int n = std::min(m->max_batch, S - s0);
        MCK(forward(m, m->x + 3 * (int64_t)s0, n));
        for (int r0 = 0; r0 < n; r0 += m->rows_out) {
            // the flag with the first rows, further rows alone
            const int k = std::min(m->rows_out, n - r0);
            if (r0 == 0)
                MCK(cudaMemcpyAsync(m->h_out, m->err, sizeof(float) * (HEAD + NOUT * k), cudaMemcpyDeviceToHost,
                                    m->stream));
            else
                MCK(cudaMemcpyAsync(m->h_out + HEAD, m->yhat + (int64_t)NOUT * r0, sizeof(float) * NOUT * k,
                                    cudaMemcpyDeviceToHost, m->stream));
            MCK(cudaStreamSynchronize(m->stream));
            if (r0 == 0 && (r = check_err(m)))
                return r;
            const float *o = m->h_out + HEAD;
            for (int64_t i = 0; i < (int64_t)NOUT * k; ++i)
                y[(int64_t)NOUT * (s0 + r0) + i] = o[i];
        }
    }
    return IBLB_OK;
}

int iblb_mlp_grad(iblb_mlp *m, const double *x, const double *y, int S, double *grad, double *loss)
{
    if (!m || !x || !y || !grad || !loss || S < 1 || S > m->max_batch)
        return mfail(m, IBLB_E_ARG, "iblb_mlp_grad: bad arguments (1 <= S <= max_batch)");
    if (!inputs_valid(x, S))
        return mfail(m, IBLB_E_ARG, "iblb_mlp_grad: inputs need finite theta_eq, R0 and lambda > 0");
    std::vector<float> hx, hy;
    int r = upload(m, x, y, S, hx, hy);
    if (r)
        return r;
    if ((r = grow(m, &m->loss, &m->loss_cap, 1)))
        return r;
    MCK(train_step(m, m->x, m->y, nullptr, S, m->loss, 0.0f, 1.0f, 1.0f));
    std::vector<float> hg(NPARAM);
    MCK(cudaMemcpyAsync(m->h_out, m->err, sizeof(int), cudaMemcpyDeviceToHost, m->stream));
    MCK(cudaMemcpyAsync(hg.data(), m->g, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, m->stream));
    MCK(cudaMemcpyAsync(loss, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
    MCK(cudaStreamSynchronize(m->stream));
    if ((r = check_err(m)))
        return r;
    for (int64_t i = 0; i < NPARAM; ++i)
        grad[i] = hg[i];
    return IBLB_OK;
}

int iblb_mlp_train(iblb_mlp *m, const double *x, const double *y, int S, int epochs, int batch, double lr,
                   uint64_t seed, double *loss_per_epoch)
{
    if (!m || !x || !y || S < 1 || epochs < 0 || batch < 1 || batch > m->max_batch || !(lr > 0.0))
        return mfail(m, IBLB_E_ARG, "iblb_mlp_train: bad arguments (1 <= batch <= max_batch, lr > 0)");
    if (!inputs_valid(x, S))
        return mfail(m, IBLB_E_ARG, "iblb_mlp_train: inputs need finite theta_eq, R0 and lambda > 0");
    std::vector<float> hx, hy;
    int r = upload(m, x, y, S, hx, hy);
    if (r)
        return r;
    std::vector<int> perm(S), sent;
    for (int i = 0; i < S; ++i)
        perm[i] = i;
    uint64_t st = seed;
    auto shuffle = [&] {                       // Fisher-Yates shuffle of the sample order
        for (int i = S - 1; i > 0; --i) {
            const int j = (int)(splitmix(st) % (uint64_t)(i + 1));
            std::swap(perm[i], perm[j]);
        }
    };
    const int nb = S / batch;                  // full batches only
    if ((r = grow(m, &m->loss, &m->loss_cap, std::max(nb, 1))) || (r = grow(m, &m->idx, &m->idx_cap, S)))
        return r;
    std::vector<double> losses((size_t)std::max(nb, 1));
    if (epochs > 0)
        shuffle();
    for (int ep = 0; ep < epochs; ++ep) {
        // an epoch's order in one copy, so that its steps' kernels follow one
        // another without a gap; the next order is drawn while they run
        sent = perm;
        MCK(cudaMemcpyAsync(m->idx, sent.data(), sizeof(int) * S, cudaMemcpyHostToDevice, m->stream));
        for (int b = 0; b < nb; ++b) {
            m->t++;
            const float c1 = 1.0f - powf(BETA1, (float)m->t), c2 = 1.0f - powf(BETA2, (float)m->t);
            MCK(train_step(m, m->x, m->y, m->idx + (int64_t)b * batch, batch, m->loss + b, (float)lr, c1, c2));
        }
        MCK(cudaMemcpyAsync(m->h_out, m->err, sizeof(int), cudaMemcpyDeviceToHost, m->stream));
        if (ep + 1 < epochs)
            shuffle();
        if (nb)
            MCK(cudaMemcpyAsync(losses.data(), m->loss, sizeof(double) * nb, cudaMemcpyDeviceToHost, m->stream));
        MCK(cudaStreamSynchronize(m->stream));
        if ((r = check_err(m)))
            return r;
        double ep_loss = 0.0;
        for (int b = 0; b < nb; ++b)
            ep_loss += losses[b];
        if (loss_per_epoch)
            loss_per_epoch[ep] = nb ? ep_loss / nb : 0.0;
    }
    return IBLB_OK;
}

}  // extern "C"
