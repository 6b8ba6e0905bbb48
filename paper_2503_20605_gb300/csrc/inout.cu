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
#include <climits>

#include "iblb_internal.h"

namespace iblb {

namespace {

__device__ __forceinline__ double orient_edge(const Arrays &a, int iu, int iv, double px, double py)
{
    const int lo = iu < iv ? iu : iv, hi = iu < iv ? iv : iu;
    const double ax = a.px[lo], ay = a.py[lo], bx = a.px[hi], by = a.py[hi];
    const double e = __dsub_rn(__dmul_rn(__dsub_rn(bx, ax), __dsub_rn(py, ay)),
                               __dmul_rn(__dsub_rn(by, ay), __dsub_rn(px, ax)));
    return iu < iv ? e : -e;
}

__device__ __forceinline__ bool edge_keeps(const Arrays &a, int iu, int iv, bool up)
{
    const int lo = iu < iv ? iu : iv, hi = iu < iv ? iv : iu;
    double dx = __dsub_rn(a.px[hi], a.px[lo]), dy = __dsub_rn(a.py[hi], a.py[lo]);
    if ((iu < iv) != up) {
        dx = -dx;
        dy = -dy;
    }
    return dy > 0.0 || (dy == 0.0 && dx < 0.0);
}

__device__ __forceinline__ double face_orient(const Arrays &a, int v0, int v1, int v2)
{
    int x = v0, y = v1, z = v2, t;
    bool even = true;
    if (x > y) { t = x; x = y; y = t; even = !even; }
    if (y > z) { t = y; y = z; z = t; even = !even; }
    if (x > y) { t = x; x = y; y = t; even = !even; }
    const double D = __dsub_rn(__dmul_rn(__dsub_rn(a.px[y], a.px[x]), __dsub_rn(a.py[z], a.py[x])),
                               __dmul_rn(__dsub_rn(a.py[y], a.py[x]), __dsub_rn(a.px[z], a.px[x])));
    return even ? D : -D;
}

// a crossing of droplet d's column (PX, PY) whose first layer above is Z
__device__ __forceinline__ void record(const Arrays &a, const Drop &D, int d, int PX, int PY, int Z)
{
    const int64_t col = D.col0 + wrapi(((PX % D.nx) + D.nx) % D.nx, D.nx) +
                        (int64_t)D.nx * (((PY % D.ny) + D.ny) % D.ny);
    const int slot = atomicAdd(&a.col_cnt[col], 1);
    if (slot < MAXC)
        a.col_t[col * MAXC + slot] = Z;
    else
        atomicOr(&a.status[4 * d], ST_COL_OVF);
}

// The face's crossings with columns X0 .. X1, Y0 .. Y1 (clipped to its
// projection) in FP64.
__device__ __noinline__ void cross_fp64(const Arrays &a, int t, int d, int X0, int X1, int Y0, int Y1)
{
    const Drop &D = a.drops[d];
    const int v0 = a.tri[3 * t], v1 = a.tri[3 * t + 1], v2 = a.tri[3 * t + 2];
    for (int k = 0; k < 3; ++k) {
        const int v = k == 0 ? v0 : (k == 1 ? v1 : v2);
        if (!(fabs(a.px[v]) < 1e8 && fabs(a.py[v]) < 1e8 && fabs(a.pz[v]) < 1e8))
            return;   // flagged by the force kernel
    }
    const double Dor = face_orient(a, v0, v1, v2);
    if (Dor == 0.0)
        return;
    const bool up = Dor > 0.0;
    const double xmin = fmin(a.px[v0], fmin(a.px[v1], a.px[v2]));
    const double xmax = fmax(a.px[v0], fmax(a.px[v1], a.px[v2]));
    const double ymin = fmin(a.py[v0], fmin(a.py[v1], a.py[v2]));
    const double ymax = fmax(a.py[v0], fmax(a.py[v1], a.py[v2]));
    const int PX0 = (int)ceil(xmin), PX1 = (int)floor(xmax);
    const int PY0 = (int)ceil(ymin), PY1 = (int)floor(ymax);
    if (PX1 - PX0 > D.nx || PY1 - PY0 > D.ny) {
        // a face wider than the box: the membrane has blown up
        atomicOr(&a.status[4 * d], ST_COL_OVF);
        return;
    }
    for (int PY = max(PY0, Y0); PY <= min(PY1, Y1); ++PY)
        for (int PX = max(PX0, X0); PX <= min(PX1, X1); ++PX) {
            const double px = (double)PX, py = (double)PY;
            const double e0 = orient_edge(a, v1, v2, px, py);
            const double e1 = orient_edge(a, v2, v0, px, py);
            const double e2 = orient_edge(a, v0, v1, px, py);
            const bool in0 = (up ? e0 > 0.0 : e0 < 0.0) || (e0 == 0.0 && edge_keeps(a, v1, v2, up));
            const bool in1 = (up ? e1 > 0.0 : e1 < 0.0) || (e1 == 0.0 && edge_keeps(a, v2, v0, up));
            const bool in2 = (up ? e2 > 0.0 : e2 < 0.0) || (e2 == 0.0 && edge_keeps(a, v0, v1, up));
            if (!(in0 && in1 && in2))
                continue;
            const double num = __dadd_rn(__dadd_rn(__dmul_rn(e0, a.pz[v0]), __dmul_rn(e1, a.pz[v1])),
                                         __dmul_rn(e2, a.pz[v2]));
            const double den = __dadd_rn(__dadd_rn(e0, e1), e2);
            const double zc = __ddiv_rn(num, den);
            // the first Z with zc < Z (never, for a crossing that is no number)
            const int Z = zc < 1e9 ? (zc > -1e9 ? (int)floor(zc) + 1 : -1000000000) : INT_MAX;
            record(a, D, d, PX, PY, Z);
        }
}

// Error bounds.  A relative coordinate c = integer part + fraction is within
// delta = 2^-24 (M + 1/2) of the FP64 position, M the face's largest |c| (the
// fraction is rounded to 2^-25, the sum to 2^-24 |c|).  With D above every
// difference of the face's x or y, a difference is within eta = 2 delta +
// 2^-24 D and an edge function, a difference of two products of two
// differences, within 4 D eta + 2^-22 D^2; tol is 1.5 times that, for the
// second-order terms and FP64's own rounding.  A crossing's height over
// corner 0 is a mean of the corners' (at most H apart) weighted by edge
// functions of one sign and sum den: it is within 3 delta + 2^-21 H +
// 5 H tol / den of its value; errz has room to spare.
__global__ void __launch_bounds__(128) face_cross_kernel(Arrays a)
{
    griddep_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.total_tri)
        return;
    const int d = a.ndrops == 1 ? 0 : a.face_drop[t];
    const Drop &D = a.drops[d];
    if (!D.vartau)
        return;
    const int v0 = a.tri[3 * t], v1 = a.tri[3 * t + 1], v2 = a.tri[3 * t + 2];
    const int4 i0 = a.ni[v0], i1 = a.ni[v1], i2 = a.ni[v2];
    const float4 f0 = a.nf[v0], f1 = a.nf[v1], f2 = a.nf[v2];
    const float x0 = f0.x, x1 = (float)(i1.x - i0.x) + f1.x, x2 = (float)(i2.x - i0.x) + f2.x;
    const float y0 = f0.y, y1 = (float)(i1.y - i0.y) + f1.y, y2 = (float)(i2.y - i0.y) + f2.y;
    const float z0 = f0.z, z1 = (float)(i1.z - i0.z) + f1.z, z2 = (float)(i2.z - i0.z) + f2.z;
    const float M = fmaxf(fmaxf(fmaxf(fabsf(x0), fabsf(x1)), fmaxf(fabsf(x2), fabsf(y0))),
                          fmaxf(fmaxf(fmaxf(fabsf(y1), fabsf(y2)), fmaxf(fabsf(z0), fabsf(z1))), fabsf(z2)));
    const float xlo = fminf(x0, fminf(x1, x2)), xhi = fmaxf(x0, fmaxf(x1, x2));
    const float ylo = fminf(y0, fminf(y1, y2)), yhi = fmaxf(y0, fmaxf(y1, y2));
    const float delta = 0x1p-24f * (M + 0.5f), Dm = fmaxf(xhi - xlo, yhi - ylo) + 0x1p-10f;
    const float tol = 1.5f * (4.0f * Dm * (2.0f * delta + 0x1p-24f * Dm) + 0x1p-22f * Dm * Dm);
    const float orient = (x1 - x0) * (y2 - y0) - (y1 - y0) * (x2 - x0);
    // a blown-up face, a node that is no number, or an open orientation
    if (!(M <= 64.0f) || (i0.w & i1.w & i2.w) == 0 || !(fabsf(orient) > tol)) {
        cross_fp64(a, t, d, INT_MIN, INT_MAX, INT_MIN, INT_MAX);
        return;
    }
    const float s = orient > 0.0f ? 1.0f : -1.0f;
    const float pad = 2.0f * delta;
    const int X0 = (int)ceilf(xlo - pad), X1 = (int)floorf(xhi + pad);
    const int Y0 = (int)ceilf(ylo - pad), Y1 = (int)floorf(yhi + pad);
    const float h1 = z1 - z0, h2 = z2 - z0, H = fmaxf(fabsf(h1), fabsf(h2));
    if (X1 - X0 > D.nx || Y1 - Y0 > D.ny) {
        cross_fp64(a, t, d, INT_MIN, INT_MAX, INT_MIN, INT_MAX);
        return;
    }
    for (int PY = Y0; PY <= Y1; ++PY)
        for (int PX = X0; PX <= X1; ++PX) {
            const float px = (float)PX, py = (float)PY;
            const float e0 = s * ((x2 - x1) * (py - y1) - (y2 - y1) * (px - x1));
            const float e1 = s * ((x0 - x2) * (py - y2) - (y0 - y2) * (px - x2));
            const float e2 = s * ((x1 - x0) * (py - y0) - (y1 - y0) * (px - x0));
            const float least = fminf(e0, fminf(e1, e2));
            if (least < -tol)
                continue;
            const float den = e0 + e1 + e2;
            const float z = z0 + (e1 * h1 + e2 * h2) / den;
            const float errz = 6.0f * delta + 0x1p-20f * H + 8.0f * H * tol / den;
            if (!(least > tol) || !(fabsf(z - rintf(z)) > errz)) {
                cross_fp64(a, t, d, i0.x + PX, i0.x + PX, i0.y + PY, i0.y + PY);
                continue;
            }
            record(a, D, d, i0.x + PX, i0.y + PY, i0.z + (int)floorf(z) + 1);
        }
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

cudaError_t launch_inout(const Arrays &a, cudaStream_t s)
{
    if (a.total_tri <= 0 || a.total_mask_cols <= 0)
        return cudaSuccess;
    cudaError_t e = launch_k(face_cross_kernel, dim3((a.total_tri + 127) / 128), dim3(128), 0, s, a.pdl != 0, a);
    if (e == cudaSuccess)
        e = launch_k(mask_kernel, dim3((a.total_mask_cols + 7) / 8), dim3(256), 0, s, a.pdl != 0, a);
    if (e != cudaSuccess)
        return e;
    return cudaGetLastError();
}

}  // namespace iblb
