// fields.cu -- conversion of one droplet's lattice state between the
// context's storage (offsets s_i = f_i - w_i rho0 in FP32 / FP16 / BF16) and
// FP64 arrays in the API layout, plus the derived fields returned to users:
// rho and U from the post-collision state (eq. hydro_var2 of the last step),
// the force density of the last step and the in/out flag of every cell.
#include "iblb_internal.h"

namespace iblb {

namespace {

__constant__ double kW[Q] = {1.0 / 3.0,  1.0 / 18.0, 1.0 / 18.0, 1.0 / 18.0, 1.0 / 18.0,
                             1.0 / 18.0, 1.0 / 18.0, 1.0 / 36.0, 1.0 / 36.0, 1.0 / 36.0,
                             1.0 / 36.0, 1.0 / 36.0, 1.0 / 36.0, 1.0 / 36.0, 1.0 / 36.0,
                             1.0 / 36.0, 1.0 / 36.0, 1.0 / 36.0, 1.0 / 36.0};

template <typename S> __device__ __forceinline__ double to_d(S v);
template <> __device__ __forceinline__ double to_d<float>(float v) { return (double)v; }
template <> __device__ __forceinline__ double to_d<__half>(__half v) { return (double)__half2float(v); }
template <> __device__ __forceinline__ double to_d<__nv_bfloat16>(__nv_bfloat16 v) { return (double)__bfloat162float(v); }
__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__half v) { return __half2float(v); }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename S> constexpr bool half_storage() { return false; }
template <> constexpr bool half_storage<__half>() { return true; }
template <typename S> __device__ __forceinline__ S from_d(double v);
template <> __device__ __forceinline__ float from_d<float>(double v) { return (float)v; }
template <> __device__ __forceinline__ __half from_d<__half>(double v) { return __double2half(v); }
template <> __device__ __forceinline__ __nv_bfloat16 from_d<__nv_bfloat16>(double v) { return __double2bfloat16(v); }

// storage index of population k of compact cell c (rows padded to the pitch)
__device__ __forceinline__ int64_t pop_index(const Drop &D, int k, int64_t c)
{
    const int64_t row = c / D.nx, x = c - row * D.nx;
    return (int64_t)Q * D.pcell0 + (int64_t)k * D.pcells + x + (int64_t)D.pitch * row;
}

template <typename S>
__global__ void export_pop_kernel(Arrays a, int d, const S *f, double *out)
{
    const Drop &D = a.drops[d];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Q * D.cells)
        return;
    const int k = (int)(i / D.cells);
    out[i] = kW[k] * (double)D.rho0 + to_d<S>(f[pop_index(D, k, i - k * D.cells)]);
}

template <typename S>
__global__ void import_pop_kernel(Arrays a, int d, S *f, const double *in)
{
    const Drop &D = a.drops[d];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Q * D.cells)
        return;
    const int k = (int)(i / D.cells);
    f[pop_index(D, k, i - k * D.cells)] = from_d<S>(in[i] - kW[k] * (double)D.rho0);
}

// offsets 0 everywhere (rest state f_i = w_i rho0), padding included
template <typename S>
__global__ void init_pop_kernel(Arrays a, S *f)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < Q * a.total_pcells)
        f[i] = from_d<S>(0.0);
}

__device__ __forceinline__ bool band_cell(const Arrays &a, const Drop &D, int64_t c, int *xyz)
{
    const int ci = (int)c;
    const int x = ci % D.nx, y = (ci / D.nx) % D.ny, z = ci / (D.nx * D.ny);
    xyz[0] = x;
    xyz[1] = y;
    xyz[2] = z;
    const int64_t t = D.tile0 + (x >> 2) + (int64_t)D.tx * ((y >> 2) + (int64_t)D.ty * (z >> 2));
    return a.tile_gen[t] == *a.gen;
}

// Sum and first moments of a cell's 19 offsets in FP64.  FP64 issues at a
// fraction of the other rates here, so nothing is multiplied by the
// directions' 0 and +-1.
__device__ __forceinline__ void moments(const double (&s)[Q], double &r, double (&j)[3])
{
#pragma unroll
    for (int k = 0; k < Q; ++k)
        r += s[k];
    j[0] = ((s[1] - s[2]) + (s[7] - s[8])) + ((s[9] - s[10]) + (s[15] - s[16])) + (s[17] - s[18]);
    j[1] = ((s[3] - s[4]) + (s[7] - s[8])) + ((s[10] - s[9]) + (s[11] - s[12])) + (s[13] - s[14]);
    j[2] = ((s[5] - s[6]) + (s[11] - s[12])) + ((s[14] - s[13]) + (s[15] - s[16])) + (s[18] - s[17]);
}

// Half offsets are multiples of 2^-24: below 4 in magnitude their sums fit a
// 32-bit integer and equal the FP64 sums exactly.
constexpr float HALF_UNITS = 16777216.0f, HALF_LIMIT = 4.0f;
__device__ __forceinline__ void moments_half(const float (&v)[Q], double &r, double (&j)[3])
{
    int n[Q], sum = 0;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        n[k] = __float2int_rn(v[k] * HALF_UNITS);
        sum += n[k];
    }
    r = fma((double)sum, 1.0 / 16777216.0, r);
    j[0] = (double)((n[1] - n[2]) + (n[7] - n[8]) + (n[9] - n[10]) + (n[15] - n[16]) + (n[17] - n[18]));
    j[1] = (double)((n[3] - n[4]) + (n[7] - n[8]) + (n[10] - n[9]) + (n[11] - n[12]) + (n[13] - n[14]));
    j[2] = (double)((n[5] - n[6]) + (n[11] - n[12]) + (n[14] - n[13]) + (n[15] - n[16]) + (n[18] - n[17]));
    for (int e = 0; e < 3; ++e)
        j[e] *= 1.0 / 16777216.0;
}

// A thread per cell, consecutive ones whatever the row's length: FP64 bounds the
// kernel, and an FP64 instruction costs a warp the same with 8 cells as with 32;
// the two integer divisions that find the row cost next to nothing.  Measured
// (ms, with the copy into kept host arrays), as it was with a buffer allocated
// for each call -> a block per 128 cells of a row -> this: 8 x 64 x 4000 FP32 1.38
// -> 2.32 -> 0.86, 24 x 100 x 900 BF16 1.44 -> 1.08 -> 0.90, 80^2 x 60 FP32 0.38 ->
// 0.20 -> 0.19, 128^3 FP16 1.40 -> 0.66 -> 0.66 (0.36 of it the copy).
constexpr int MACRO_THREADS = 128;
template <typename S>
__global__ void __launch_bounds__(MACRO_THREADS) macros_kernel(Arrays a, int d, const S *f, double *rho, double *u)
{
    const Drop &D = a.drops[d];
    const uint32_t c = blockIdx.x * MACRO_THREADS + threadIdx.x;      // (below 2^30 cells)
    if (c >= D.cells)
        return;
    const uint32_t r0 = c / (uint32_t)D.nx;
    const int x = (int)(c - r0 * (uint32_t)D.nx), row = (int)r0, z = row / D.ny, y = row - z * D.ny;
    const int64_t cell = x + (int64_t)D.pitch * row;
    const S *p = f + (int64_t)Q * D.pcell0 + cell;
    double r = D.rho0, j[3];
    float v[Q], most = 0.0f;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        v[k] = to_f(p[(int64_t)k * D.pcells]);
        most = fmaxf(most, fabsf(v[k]));
        most = v[k] == v[k] ? most : INFINITY;      // (fmaxf drops a NaN)
    }
    if (sizeof(S) == 2 && half_storage<S>() && most < HALF_LIMIT) {
        moments_half(v, r, j);
    } else {
        double s[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k)
            s[k] = (double)v[k];
        moments(s, r, j);
    }
    double F[3] = {D.bf[0], D.bf[1], D.bf[2]};
    const int64_t t = D.tile0 + (x >> 2) + (int64_t)D.tx * ((y >> 2) + (int64_t)D.ty * (z >> 2));
    if (a.tile_gen[t] == *a.gen)
        for (int e = 0; e < 3; ++e)
            F[e] += a.F[e * a.total_pcells + D.pcell0 + cell];
    rho[c] = r;
    // post-collision momentum = sum c_i f_i + F (BGK keeps rho U, Guo adds (1-1/2tau) F)
    // Divided, so that U is rounded once: products with 1 / rho are off by up to
    // one and a half units, and brought back to the rounded quotients by their
    // remainders cost more than the divisions (the call at 128^3 FP16: 0.47 ms
    // products, 0.66 divisions, 0.72 corrected products).
    for (int e = 0; e < 3; ++e)
        u[e * D.cells + c] = (j[e] - 0.5 * F[e]) / r;
}

__global__ void force_kernel(Arrays a, int d, double *F)
{
    const Drop &D = a.drops[d];
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= D.cells)
        return;
    int xyz[3];
    const bool band = band_cell(a, D, c, xyz);
    const int64_t g = pop_index(D, 0, c) - (int64_t)Q * D.pcell0 + D.pcell0;   // padded field index
    for (int e = 0; e < 3; ++e)
        F[e * D.cells + c] = (double)D.bf[e] + (band ? (double)a.F[e * a.total_pcells + g] : 0.0);
}

__global__ void inside_kernel(Arrays a, int d, uint8_t *inside)
{
    const Drop &D = a.drops[d];
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= D.cells)
        return;
    const int ci = (int)c;
    const int x = ci % D.nx, y = (ci / D.nx) % D.ny, z = ci / (D.nx * D.ny);
    int par = 0;
    if (D.vartau)
        par = (a.mask[D.mask0 + D.mask_pitch * (y + (int64_t)D.ny * z) + (x >> 3)] >> (x & 7)) & 1;
    inside[c] = (uint8_t)par;
}

inline unsigned blocks_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

cudaError_t launch_export_populations(const Arrays &a, int d, int storage, const void *f, double *out,
                                      int64_t cells, cudaStream_t s)
{
    const unsigned g = blocks_for(Q * cells, 256);
    switch (storage) {
    case 0: export_pop_kernel<float><<<g, 256, 0, s>>>(a, d, (const float *)f, out); break;
    case 1: export_pop_kernel<__half><<<g, 256, 0, s>>>(a, d, (const __half *)f, out); break;
    case 2: export_pop_kernel<__nv_bfloat16><<<g, 256, 0, s>>>(a, d, (const __nv_bfloat16 *)f, out); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_import_populations(const Arrays &a, int d, int storage, void *f, const double *in,
                                      int64_t cells, cudaStream_t s)
{
    const unsigned g = blocks_for(Q * cells, 256);
    switch (storage) {
    case 0: import_pop_kernel<float><<<g, 256, 0, s>>>(a, d, (float *)f, in); break;
    case 1: import_pop_kernel<__half><<<g, 256, 0, s>>>(a, d, (__half *)f, in); break;
    case 2: import_pop_kernel<__nv_bfloat16><<<g, 256, 0, s>>>(a, d, (__nv_bfloat16 *)f, in); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_init_populations(const Arrays &a, int storage, void *f, cudaStream_t s)
{
    const unsigned g = blocks_for(Q * a.total_pcells, 256);
    switch (storage) {
    case 0: init_pop_kernel<float><<<g, 256, 0, s>>>(a, (float *)f); break;
    case 1: init_pop_kernel<__half><<<g, 256, 0, s>>>(a, (__half *)f); break;
    case 2: init_pop_kernel<__nv_bfloat16><<<g, 256, 0, s>>>(a, (__nv_bfloat16 *)f); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_export_macros(const Arrays &a, const Drop &D, int d, int storage, const void *f, double *rho,
                                 double *u, cudaStream_t s)
{
    const unsigned g = blocks_for(D.cells, MACRO_THREADS);
    switch (storage) {
    case 0: macros_kernel<float><<<g, MACRO_THREADS, 0, s>>>(a, d, (const float *)f, rho, u); break;
    case 1: macros_kernel<__half><<<g, MACRO_THREADS, 0, s>>>(a, d, (const __half *)f, rho, u); break;
    case 2: macros_kernel<__nv_bfloat16><<<g, MACRO_THREADS, 0, s>>>(a, d, (const __nv_bfloat16 *)f, rho, u); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_export_force(const Arrays &a, int d, double *F, int64_t cells, cudaStream_t s)
{
    force_kernel<<<blocks_for(cells, 256), 256, 0, s>>>(a, d, F);
    return cudaGetLastError();
}

cudaError_t launch_export_inside(const Arrays &a, int d, uint8_t *inside, int64_t cells, cudaStream_t s)
{
    inside_kernel<<<blocks_for(cells, 256), 256, 0, s>>>(a, d, inside);
    return cudaGetLastError();
}

}  // namespace iblb
