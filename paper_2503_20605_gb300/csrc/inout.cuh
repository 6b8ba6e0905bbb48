// inout.cuh -- the in/out test's ray crossings of one face (see inout.cu), for
// its own kernel and for the spread kernel, whose blocks take the faces once
// their tiles are done.
#pragma once

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
__device__ __forceinline__ void face_cross(const Arrays &a, int t)
{
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

}  // namespace

}  // namespace iblb
