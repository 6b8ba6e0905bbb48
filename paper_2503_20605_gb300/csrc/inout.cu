// inout.cu -- in/out classification of lattice cells for the viscosity
// ratio (Sec. II A: tau = tau_in inside the closed interface, tau_out
// outside, re-identified every step by ray tracing).
//
// A vertical ray runs through every lattice column (X, Y).  One thread per
// face finds the columns inside the face's xy projection and records where
// the ray crosses it: the first layer Z above the crossing.  A cell is inside
// iff an odd number of crossings lies strictly below it; one warp per 32
// columns turns the crossings into one bit per cell, which the stream-collide
// kernel stages with its rows.  Points on a shared edge or vertex are
// assigned by a half-open rule (a symbolic shift of the point by (-e, -e^2))
// and each edge function is evaluated from its lower-numbered end point, so
// the two faces of an edge see exactly opposite values and the surface is
// watertight.
//
// The decisions are those of FP64 arithmetic with every product and sum
// individually rounded (no contraction).  They are taken in FP32 wherever
// FP32 is sure of them: on coordinates relative to the face (each node's
// integer part and FP32 fraction, from the force kernel) every edge function
// is within tol of its value, and a sign or a layer that tol leaves open is
// decided by the FP64 code (about one crossing in ten thousand).  FP64 issues
// at a fraction of FP32's rate here and bound this kernel.  Measured, with
// what clears, sorts or packs the crossings: 81 920 faces 26 -> 19 us, 428 800
// faces in 32 boxes 85 -> 32 us; and the stream-collide kernel, which walked
// each cell's column in FP64, 127 -> 111 us (256^2 x 128 BF16) and 171 -> 128
// us (32 boxes FP16).
#include "inout.cuh"

namespace iblb {

namespace {

__global__ void __launch_bounds__(128) face_cross_kernel(Arrays a)
{
    griddep_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < a.total_tri)
        face_cross(a, t);
}

__device__ __forceinline__ int find_drop_mask(const Drop *D, int n, int w)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (D[mid].mask_col0 <= w)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// 32 x 32 bit transpose across a warp: bit b of lane l <-> bit l of lane b
__device__ __forceinline__ uint32_t transpose32(uint32_t x)
{
    const int lane = threadIdx.x & 31;
    uint32_t m = 0x0000ffffu;
#pragma unroll
    for (int j = 16; j >= 1; j >>= 1) {
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
        x = (lane & j) ? ((x & ~m) | ((y & ~m) >> j)) : ((x & m) | ((y & m) << j));
        m ^= m << (j >> 1);
    }
    return x;
}

// One warp per 32 consecutive columns of a row y: lane x forms its column's
// inside bits, 32 layers at a time, and a bit transpose turns them into the
// rows' words.  The column's crossings are emptied for the next step.
__global__ void __launch_bounds__(256) mask_kernel(Arrays a)
{
    griddep_wait();
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= a.total_mask_cols)
        return;
    const int d = a.ndrops == 1 ? 0 : find_drop_mask(a.drops, a.ndrops, w);
    const Drop &D = a.drops[d];
    const int words = D.mask_pitch >> 2, k = w - D.mask_col0;
    const int y = k / words, wx = k - y * words, x = 32 * wx + lane;
    int cnt = 0;
    int t[MAXC];
    if (x < D.nx) {
        const int64_t col = D.col0 + x + (int64_t)D.nx * y;
        cnt = min(a.col_cnt[col], MAXC);
        if (cnt) {
            a.col_cnt[col] = 0;
#pragma unroll
            for (int q = 0; q < MAXC; ++q)
                t[q] = q < cnt ? a.col_t[col * MAXC + q] - D.walls : INT_MAX;
        }
    }
    // columns without a crossing now or in the step before: their words are 0
    const bool any = __any_sync(0xffffffffu, cnt != 0), had = a.mask_any[w] != 0;
    if (!any && !had)
        return;
    __syncwarp();
    if (lane == 0)
        a.mask_any[w] = any;
    uint32_t *out = reinterpret_cast<uint32_t *>(a.mask + D.mask0 + (int64_t)D.mask_pitch * y) + wx;
    for (int zb = 0; zb < D.nzf; zb += 32) {
        uint32_t m = 0;
        if (any) {
            if (cnt) {
#pragma unroll
                for (int q = 0; q < MAXC; ++q)
                    if (q < cnt)
                        m ^= t[q] <= zb ? 0xffffffffu : (t[q] - zb >= 32 ? 0u : 0xffffffffu << (t[q] - zb));
            }
            m = transpose32(m);
        }
        if (zb + lane < D.nzf)
            out[(int64_t)words * D.ny * (zb + lane)] = m;
    }
}

}  // namespace

cudaError_t launch_inout(const Arrays &a, cudaStream_t s, bool faces)
{
    if (a.total_tri <= 0 || a.total_mask_cols <= 0)
        return cudaSuccess;
    cudaError_t e = cudaSuccess;
    if (faces)
        e = launch_k(face_cross_kernel, dim3((a.total_tri + 127) / 128), dim3(128), 0, s, a.pdl != 0, a);
    if (e == cudaSuccess)
        e = launch_k(mask_kernel, dim3((a.total_mask_cols + 7) / 8), dim3(256), 0, s, a.pdl != 0, a);
    if (e != cudaSuccess)
        return e;
    return cudaGetLastError();
}

}  // namespace iblb
