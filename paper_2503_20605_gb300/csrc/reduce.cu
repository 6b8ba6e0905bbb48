// reduce.cu -- FP64 reductions over the membrane and the lattice:
//   * mesh volume V = (1/6) sum_t q_a . (q_b x q_c), area, node centroid,
//     z_min and z_max (the half-height l = (z_max - z_min)/2 of App. C, eq. ell);
//   * contact-radius protocols (i) and (ii) of Sec. III B;
//   * lattice mass sum_x sum_i f_i: each cell's 19 stored offsets are added
//     in FP32 (a few rounding errors of the offsets' size, about 1e-3 of a
//     cell's density) and the cells in FP64 in a fixed order and tree.
// Every reduction uses a fixed assignment of items to threads and a fixed
// shuffle tree, so results are bitwise reproducible and a droplet's values
// do not depend on the other droplets of a batch.
#include <math.h>

#include <algorithm>

#include "iblb_internal.h"
#include "reduce_util.cuh"

namespace iblb {

namespace {

constexpr int RB = 256;          // threads per reduction block

// Chunks of a mesh for the observation passes: enough for every SM to
// share the FP64 work (at least RED_MIN_FACES faces and RED_MIN_NODES nodes
// a chunk), at most RED_MAX_CHUNKS (the allocation-free scratch's size);
// the split depends on the mesh's size alone, so results are reproducible.
constexpr int RED_MIN_FACES = 64, RED_MIN_NODES = 32, RED_MAX_CHUNKS = 512;
__host__ __device__ int mesh_chunks(int nnodes, int ntri, int &fpc, int &npc)
{
    const int nf = (ntri + RED_MIN_FACES - 1) / RED_MIN_FACES, nn = (nnodes + RED_MIN_NODES - 1) / RED_MIN_NODES;
    int nc = nf > nn ? nf : nn;
    nc = nc < 1 ? 1 : (nc > RED_MAX_CHUNKS ? RED_MAX_CHUNKS : nc);
    fpc = (ntri + nc - 1) / nc;
    fpc = fpc < 1 ? 1 : fpc;
    npc = (nnodes + nc - 1) / nc;
    npc = npc < 1 ? 1 : npc;
    return nc;
}

// warps of a block that n items (one per thread, in order) reach
__device__ __forceinline__ int warps_of(int n) { return min(RB, n + 31) >> 5; }

// chunk k of a mesh: faces [k*fpc, ...) and nodes [k*npc, ...)
// -> 6V, area, sum x, sum y, sum z, z_min, z_max, clamped nodes
__device__ void pass1_chunk(const ObsMesh &m, int k, double *out)
{
    const int KIND[8] = {0, 0, 0, 0, 0, 1, 2, 0};
    double v[8] = {0.0, 0.0, 0.0, 0.0, 0.0, INFINITY, -INFINITY, 0.0};
    const int f1 = min(m.ntri, (k + 1) * m.fpc);
    for (int t = k * m.fpc + threadIdx.x; t < f1; t += RB) {
        const int ia = m.tri[3 * t] * m.stride, ib = m.tri[3 * t + 1] * m.stride, ic = m.tri[3 * t + 2] * m.stride;
        const double ax = m.qx[ia], ay = m.qy[ia], az = m.qz[ia];
        const double bx = m.qx[ib], by = m.qy[ib], bz = m.qz[ib];
        const double cx = m.qx[ic], cy = m.qy[ic], cz = m.qz[ic];
        v[0] += ax * (by * cz - bz * cy) + ay * (bz * cx - bx * cz) + az * (bx * cy - by * cx);
        const double e1x = bx - ax, e1y = by - ay, e1z = bz - az, e2x = cx - ax, e2y = cy - ay, e2z = cz - az;
        const double Nx = e1y * e2z - e1z * e2y, Ny = e1z * e2x - e1x * e2z, Nz = e1x * e2y - e1y * e2x;
        v[1] += 0.5 * sqrt(Nx * Nx + Ny * Ny + Nz * Nz);
    }
    const int n1 = min(m.nnodes, (k + 1) * m.npc);
    for (int j = k * m.npc + threadIdx.x; j < n1; j += RB) {
        const int ij = (m.node0 + j) * m.stride;
        if (m.clamped)
            v[7] += (double)m.clamped[m.node0 + j];
        v[2] += m.qx[ij];
        v[3] += m.qy[ij];
        const double z = m.qz[ij];
        v[4] += z;
        v[5] = fmin(v[5], z);
        v[6] = fmax(v[6], z);
    }
    block_reduce<8, RB>(v, KIND, warps_of(max(m.fpc, m.npc)));
    if (threadIdx.x == 0)
        for (int i = 0; i < 8; ++i)
            out[i] = v[i];
}

// Value v of nch groups of `width` partials, folded by one warp in a fixed
// order (chunk i goes to lane i % 32, lanes add their chunks in order, then a
// fixed shuffle tree): the sum, or the minimum / maximum.
__device__ __forceinline__ double fold(const double *part, int nch, int width, int v, int kind)
{
    const int lane = threadIdx.x & 31;
    double x = kind == 0 ? 0.0 : (kind == 1 ? INFINITY : -INFINITY);
    for (int i = lane; i < nch; i += 32) {
        const double p = __ldcg(part + (int64_t)width * i + v);
        x = kind == 0 ? x + p : (kind == 1 ? fmin(x, p) : fmax(x, p));
    }
    return kind == 0 ? warp_sum(x) : (kind == 1 ? warp_min(x) : warp_max(x));
}

// --- observation of meshes (blockIdx.y: which), used by iblb_observe, its
//     form for every droplet and the stateless entry points: three passes and
//     the result.  Each block of a pass folds what it needs of the previous
//     pass itself (two values, then three), so no launch of one warp stands
//     between the passes.  Measured per call: 20 480 faces and 128^3 cells
//     101 -> 67 us (the mass on a stream beside it), 64 droplets 3.4 -> 0.77
//     ms (one set of launches for all).  scratch of a mesh (doubles): NRED * nc partials of
//     pass 1, 4 * nc of pass 2, nc of pass 3.
struct ObsScratch {
    double *p1, *p2, *p3;
    __device__ ObsScratch(const ObsMesh &m)
    {
        p1 = m.scratch;
        p2 = p1 + (int64_t)NRED * m.nc;
        p3 = p2 + 4 * (int64_t)m.nc;
    }
};
// height of the cutting plane and the flatness limit of the contact-radius
// protocols (products and sums individually rounded)
__device__ __forceinline__ double cut_plane(const ObsMesh &m, double zcut) { return __dadd_rn(0.5, __dmul_rn(zcut, m.R0)); }

__global__ void __launch_bounds__(RB) pass1_kernel(const ObsMesh *table, ObsMesh one)
{
    griddep_wait();
    const ObsMesh m = table ? table[blockIdx.y] : one;
    if ((int)blockIdx.x >= m.nc)
        return;
    pass1_chunk(m, blockIdx.x, ObsScratch(m).p1 + (int64_t)NRED * blockIdx.x);
}

// protocol (i): edges (a < b) crossing z = zp: sum of crossing x, y and count;
// protocol (ii): lower-half faces with max |dz| < eps: area.
__global__ void __launch_bounds__(RB) pass2_kernel(const ObsMesh *table, ObsMesh one, double zcut, double eps_flat)
{
    griddep_wait();
    const ObsMesh m = table ? table[blockIdx.y] : one;
    const int k = blockIdx.x;
    if (k >= m.nc)
        return;
    const ObsScratch scr(m);
    __shared__ double zext[2];
    if (threadIdx.x < 64) {     // warps 0 and 1: z_min, z_max
        const int w = threadIdx.x >> 5;
        const double z = fold(scr.p1, m.nc, NRED, 5 + w, 1 + w);
        if ((threadIdx.x & 31) == 0)
            zext[w] = z;
    }
    __syncthreads();
    const int KIND[4] = {0, 0, 0, 0};
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    const double zmid = 0.5 * (zext[0] + zext[1]), zp = cut_plane(m, zcut), flat = eps_flat * m.R0;
    const int f1 = min(m.ntri, (k + 1) * m.fpc);
    for (int t = k * m.fpc + threadIdx.x; t < f1; t += RB) {
        int idx[3] = {m.tri[3 * t], m.tri[3 * t + 1], m.tri[3 * t + 2]};
        double zz[3];
        for (int e = 0; e < 3; ++e)
            zz[e] = m.qz[idx[e] * m.stride];
        for (int e = 0; e < 3; ++e) {
            const int ia = idx[e], ib = idx[(e + 1) % 3];
            if (ia > ib)
                continue;
            const double za = zz[e], zb = zz[(e + 1) % 3];
            if (!((za < zp && zb >= zp) || (zb < zp && za >= zp)))
                continue;
            const double s = (zp - za) / (zb - za);
            const double xa = m.qx[ia * m.stride], ya = m.qy[ia * m.stride];
            v[0] += xa + s * (m.qx[ib * m.stride] - xa);
            v[1] += ya + s * (m.qy[ib * m.stride] - ya);
            v[2] += 1.0;
        }
        if ((zz[0] + zz[1] + zz[2]) / 3.0 < zmid) {
            const double dz = fmax(fabs(zz[0] - zz[1]), fmax(fabs(zz[1] - zz[2]), fabs(zz[0] - zz[2])));
            if (dz < flat) {
                const int ia = idx[0] * m.stride, ib = idx[1] * m.stride, ic = idx[2] * m.stride;
                const double e1x = m.qx[ib] - m.qx[ia], e1y = m.qy[ib] - m.qy[ia], e1z = zz[1] - zz[0];
                const double e2x = m.qx[ic] - m.qx[ia], e2y = m.qy[ic] - m.qy[ia], e2z = zz[2] - zz[0];
                const double Nx = e1y * e2z - e1z * e2y, Ny = e1z * e2x - e1x * e2z, Nz = e1x * e2y - e1y * e2x;
                v[3] += 0.5 * sqrt(Nx * Nx + Ny * Ny + Nz * Nz);
            }
        }
    }
    block_reduce<4, RB>(v, KIND, warps_of(m.fpc));
    if (threadIdx.x == 0)
        for (int i = 0; i < 4; ++i)
            scr.p2[4 * k + i] = v[i];
}

// protocol (i) second pass: sum of distances of the crossings from their centre
__global__ void __launch_bounds__(RB) pass3_kernel(const ObsMesh *table, ObsMesh one, double zcut)
{
    griddep_wait();
    const ObsMesh m = table ? table[blockIdx.y] : one;
    const int k = blockIdx.x;
    if (k >= m.nc)
        return;
    const ObsScratch scr(m);
    __shared__ double sums[3];
    if (threadIdx.x < 96) {     // warps 0 .. 2: sum x, sum y, count of the crossings
        const double x = fold(scr.p2, m.nc, 4, threadIdx.x >> 5, 0);
        if ((threadIdx.x & 31) == 0)
            sums[threadIdx.x >> 5] = x;
    }
    __syncthreads();
    const int KIND[1] = {0};
    double v[1] = {0.0};
    const double cx = sums[2] > 0.0 ? sums[0] / sums[2] : 0.0, cy = sums[2] > 0.0 ? sums[1] / sums[2] : 0.0;
    const double zp = cut_plane(m, zcut);
    const int f1 = min(m.ntri, (k + 1) * m.fpc);
    for (int t = k * m.fpc + threadIdx.x; t < f1; t += RB)
        for (int e = 0; e < 3; ++e) {
            const int ia = m.tri[3 * t + e], ib = m.tri[3 * t + (e + 1) % 3];
            if (ia > ib)
                continue;
            const double za = m.qz[ia * m.stride], zb = m.qz[ib * m.stride];
            if (!((za < zp && zb >= zp) || (zb < zp && za >= zp)))
                continue;
            const double s = (zp - za) / (zb - za);
            const double xa = m.qx[ia * m.stride], ya = m.qy[ia * m.stride];
            const double px = xa + s * (m.qx[ib * m.stride] - xa) - cx;
            const double py = ya + s * (m.qy[ib * m.stride] - ya) - cy;
            v[0] += sqrt(px * px + py * py);
        }
    block_reduce<1, RB>(v, KIND, warps_of(m.fpc));
    if (threadIdx.x == 0)
        scr.p3[k] = v[0];
}

// The OBS_RAW results of mesh blockIdx.y: V, A, cx, cy, cz, zmin, zmax,
// clamped nodes, sum x, sum y, count of the crossings, flat area, sum of
// distances; with mass and status (of a context) the lattice mass, the
// droplet's status flags and droplet 0's.  One warp per value.
constexpr int FIN_THREADS = 32 * 13;
__global__ void __launch_bounds__(FIN_THREADS) obs_result_kernel(const ObsMesh *table, ObsMesh one, const double *mass,
                                                                 const int *status, int d0, double *out)
{
    griddep_wait();
    const ObsMesh m = table ? table[blockIdx.y] : one;
    double *o = out + (int64_t)OBS_RAW * blockIdx.y;
    const int w = threadIdx.x >> 5;
    if (m.nnodes) {
        const ObsScratch scr(m);
        double x;
        if (w < 8)
            x = fold(scr.p1, m.nc, NRED, w, w == 5 ? 1 : (w == 6 ? 2 : 0));
        else if (w < 12)
            x = fold(scr.p2, m.nc, 4, w - 8, 0);
        else
            x = fold(scr.p3, m.nc, 1, 0, 0);
        if (w == 0)
            x /= 6.0;
        else if (w >= 2 && w <= 4)
            x /= m.nnodes;
        if ((threadIdx.x & 31) == 0)
            o[w] = x;
    }
    if (threadIdx.x == 0 && mass) {
        const int d = d0 + blockIdx.y;
        o[13] = mass[d];
        o[14] = (double)status[4 * d];
        o[15] = (double)status[0];
    }
}

// ---- lattice mass: sum over cells of sum_i s_i (FP64), per droplet
template <typename S>
__device__ __forceinline__ float tof(S v);
template <> __device__ __forceinline__ float tof<float>(float v) { return v; }
template <> __device__ __forceinline__ float tof<__half>(__half v) { return __half2float(v); }
template <> __device__ __forceinline__ float tof<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

__device__ __forceinline__ int find_drop_mass(const Drop *D, int n, int b)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (D[mid].mass_block0 <= b)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// block b: cells [(b - mass_block0) MASS_CELLS_PER_BLOCK, ...) of its
// droplet, MASS_CELLS_PER_BLOCK / RB per thread (added in FP64 in a fixed
// order), then the fixed block tree: a quarter of the FP64 tree work per
// cell of one cell per thread.
template <typename S>
__global__ void __launch_bounds__(RB) mass_kernel(Arrays a, const S *f, int b0)
{
    griddep_wait();
    constexpr int CPT = MASS_CELLS_PER_BLOCK / RB;
    static_assert(CPT * RB == MASS_CELLS_PER_BLOCK, "whole cells per thread");
    const int KIND[1] = {0};
    const int b = b0 + blockIdx.x;
    const int d = find_drop_mass(a.drops, a.ndrops, b);
    const Drop &D = a.drops[d];
    const int64_t cb = (int64_t)(b - D.mass_block0) * MASS_CELLS_PER_BLOCK + threadIdx.x;
    float cell[CPT];
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
        const int64_t c = cb + (int64_t)u * RB;
        cell[u] = 0.0f;
        if (c < D.cells) {
            const int64_t row = c / D.nx;
            const S *p = f + (int64_t)Q * D.pcell0 + (c - row * D.nx) + (int64_t)D.pitch * row;
            for (int i = 0; i < Q; ++i)
                cell[u] += tof<S>(p[(int64_t)i * D.pcells]);
        }
    }
    double v[1] = {0.0};
#pragma unroll
    for (int u = 0; u < CPT; ++u)
        v[0] += (double)cell[u];
    block_reduce<1, RB>(v, KIND);
    if (threadIdx.x == 0)
        a.mass_part[b] = v[0];
}

// one block of RB threads per droplet: thread t adds partials t, t + RB, ...,
// then the fixed block tree
__global__ void __launch_bounds__(RB) mass_fold_kernel(Arrays a, double *out, int d0)
{
    griddep_wait();
    const int KIND[1] = {0};
    const int d = d0 + blockIdx.x;
    const Drop &D = a.drops[d];
    double v[1] = {0.0};
    for (int i = threadIdx.x; i < D.mass_nblocks; i += RB)
        v[0] += a.mass_part[D.mass_block0 + i];
    block_reduce<1, RB>(v, KIND);
    if (threadIdx.x == 0)
        out[d] = v[0] + (double)D.rho0 * (double)D.cells;
}

}  // namespace


// chunks and scratch size (doubles) of a mesh
void obs_mesh_plan(ObsMesh &m) { m.nc = mesh_chunks(m.nnodes, m.ntri, m.fpc, m.npc); }
int64_t observe_scratch_doubles(int n_nodes, int n_tri)
{
    int fpc = 0, npc = 0;
    return (int64_t)(NRED + 5) * mesh_chunks(n_nodes, n_tri, fpc, npc);
}

// meshes per launch: a grid has at most this many blocks in y
constexpr int OBS_GRID_Y = 65535;

// chained by programmatic dependent launch: each kernel waits for the
// previous one before reading its results
cudaError_t enqueue_observe(const ObsMesh *table, const ObsMesh *one, int n, int max_chunks, double zcut_frac,
                            double eps_flat, cudaStream_t s)
{
    const ObsMesh m = one ? *one : ObsMesh{};
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < n && e == cudaSuccess; i += OBS_GRID_Y) {
        const dim3 g(max_chunks, std::min(n - i, OBS_GRID_Y));
        const ObsMesh *t = table ? table + i : nullptr;
        if ((e = launch_k(pass1_kernel, g, dim3(RB), 0, s, true, t, m)) == cudaSuccess &&
            (e = launch_k(pass2_kernel, g, dim3(RB), 0, s, true, t, m, zcut_frac, eps_flat)) == cudaSuccess)
            e = launch_k(pass3_kernel, g, dim3(RB), 0, s, true, t, m, zcut_frac);
    }
    return e;
}
cudaError_t enqueue_observe_result(const ObsMesh *table, const ObsMesh *one, int n, const double *mass,
                                   const int *status, int d0, double *out, cudaStream_t s)
{
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < n && e == cudaSuccess; i += OBS_GRID_Y)
        e = launch_k(obs_result_kernel, dim3(1, std::min(n - i, OBS_GRID_Y)), dim3(FIN_THREADS), 0, s, true,
                     table ? table + i : nullptr, one ? *one : ObsMesh{}, mass, status, d0 + i,
                     out + (int64_t)OBS_RAW * i);
    return e;
}

// h_out: V, A, cx, cy, cz, zmin, zmax, theta(R0), theta(R_V), rc_cut,
// rc_flat, n_cut, chi_flat, clamped nodes
void finish_observe(const double *hv, double R0, double *h_out)
{
    const double V = hv[0], A = hv[1], zmin = hv[5], zmax = hv[6];
    const double ell = 0.5 * (zmax - zmin);
    const double RV = cbrt(3.0 * V / (4.0 * M_PI));
    auto theta = [](double l, double Rr) {
        const double l3 = l * l * l, R3 = Rr * Rr * Rr;
        if (l3 >= R3)
            return 180.0;
        return 2.0 * atan(sqrt(3.0 * l3 / (R3 - l3))) * 180.0 / M_PI;  // eq. angleh
    };
    h_out[0] = V;
    h_out[1] = A;
    h_out[2] = hv[2];
    h_out[3] = hv[3];
    h_out[4] = hv[4];
    h_out[5] = zmin;
    h_out[6] = zmax;
    h_out[7] = theta(ell, R0);
    h_out[8] = theta(ell, RV);
    h_out[9] = hv[10] > 0.0 ? hv[12] / hv[10] : 0.0;  // rc_cut
    h_out[10] = sqrt(hv[11] / M_PI);                  // rc_flat
    h_out[11] = hv[10];                               // n_cut
    h_out[12] = hv[11];                               // chi_flat
    h_out[13] = hv[7];                                // clamped nodes
}

cudaError_t launch_observe_view(const double *qx, const double *qy, const double *qz, int stride,
                                const int *tri, int ntri, int node0, int nnodes, double R0, double zcut_frac,
                                double eps_flat, double *scratch, double *h_out, cudaStream_t s)
{
    // the results follow the passes' scratch
    ObsMesh m{qx, qy, qz, stride, tri, ntri, node0, nnodes, 0, 0, 0, nullptr, R0, scratch};
    obs_mesh_plan(m);
    double *res = scratch + observe_scratch_doubles(nnodes, ntri), hv[OBS_RAW], t[14];
    cudaError_t e = enqueue_observe(nullptr, &m, 1, m.nc, zcut_frac, eps_flat, s);
    if (e == cudaSuccess)
        e = enqueue_observe_result(nullptr, &m, 1, nullptr, nullptr, 0, res, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(hv, res, sizeof(double) * OBS_RAW, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(s);
    if (e != cudaSuccess)
        return e;
    finish_observe(hv, R0, t);
    for (int i = 0; i < 13; ++i)   // the first 13 (no clamped count for a bare mesh)
        h_out[i] = t[i];
    return cudaSuccess;
}

cudaError_t preload_observe_kernels()
{
    // under lazy module loading a kernel's code reaches the device at its
    // first launch or at the first query of its attributes
    cudaFuncAttributes fa;
    const void *k[] = {(const void *)pass1_kernel, (const void *)pass2_kernel, (const void *)pass3_kernel,
                       (const void *)obs_result_kernel};
    for (const void *f : k) {
        cudaError_t e = cudaFuncGetAttributes(&fa, f);
        if (e != cudaSuccess)
            return e;
    }
    return cudaSuccess;
}

cudaError_t launch_mass(const Arrays &a, int storage, const void *f, double *d_out, int block0, int blocks, int d0,
                        int n, cudaStream_t s)
{
    const dim3 g(blocks), b(RB);
    cudaError_t e;
    switch (storage) {
    case 0: e = launch_k(mass_kernel<float>, g, b, 0, s, true, a, (const float *)f, block0); break;
    case 1: e = launch_k(mass_kernel<__half>, g, b, 0, s, true, a, (const __half *)f, block0); break;
    case 2: e = launch_k(mass_kernel<__nv_bfloat16>, g, b, 0, s, true, a, (const __nv_bfloat16 *)f, block0); break;
    default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess)
        return e;
    return launch_k(mass_fold_kernel, dim3(n), dim3(RB), 0, s, true, a, d_out, d0);
}

}  // namespace iblb
