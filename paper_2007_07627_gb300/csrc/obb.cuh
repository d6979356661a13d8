// Oriented bounding box of a bucket of target points, and the float distance
// test the closest-point search runs against it. Host and device code: the
// kernels build and test the boxes with these functions, and a CPU test runs
// the same functions against exact FP64 distances.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#ifndef FRICP_HD
#define FRICP_HD __host__ __device__
#endif

namespace fricp {

// v rounded up to float.
FRICP_HD inline float f32_round_up(double v) {
#ifdef __CUDA_ARCH__
    return __double2float_ru(v);
#else
    float f = (float)v;
    if ((double)f < v) f = nextafterf(f, INFINITY);
    return f;
#endif
}

FRICP_HD inline float f32_rsqrt(float x) {
#ifdef __CUDA_ARCH__
    return rsqrtf(x);
#else
    return 1.0f / sqrtf(x);
#endif
}

// Eigenvectors of the symmetric 3x3 matrix A (cyclic Jacobi rotations, float):
// the columns of V. Only the tightness of the oriented boxes depends on them.
FRICP_HD inline void jacobi3f(float A[3][3], float V[3][3]) {
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) V[i][j] = i == j ? 1.0f : 0.0f;
    for (int sweep = 0; sweep < 8; ++sweep) {
        const float off = fabsf(A[0][1]) + fabsf(A[0][2]) + fabsf(A[1][2]);
        const float dia = fabsf(A[0][0]) + fabsf(A[1][1]) + fabsf(A[2][2]);
        if (!(off > 1e-7f * dia)) break;
        for (int p = 0; p < 2; ++p) {
            for (int q = p + 1; q < 3; ++q) {
                if (A[p][q] == 0.0f) continue;
                const float theta = (A[q][q] - A[p][p]) / (2.0f * A[p][q]);
                const float t = copysignf(1.0f, theta) / (fabsf(theta) + sqrtf(fmaf(theta, theta, 1.0f)));
                const float c = f32_rsqrt(fmaf(t, t, 1.0f)), sn = t * c;
                for (int k = 0; k < 3; ++k) {   // A <- A J (columns p, q)
                    const float akp = A[k][p], akq = A[k][q];
                    A[k][p] = c * akp - sn * akq;
                    A[k][q] = sn * akp + c * akq;
                }
                for (int k = 0; k < 3; ++k) {   // A <- J^T A (rows p, q)
                    const float apk = A[p][k], aqk = A[q][k];
                    A[p][k] = c * apk - sn * aqk;
                    A[q][k] = sn * apk + c * aqk;
                }
                for (int k = 0; k < 3; ++k) {   // V <- V J
                    const float vkp = V[k][p], vkq = V[k][q];
                    V[k][p] = c * vkp - sn * vkq;
                    V[k][q] = sn * vkp + c * vkq;
                }
            }
        }
    }
}

// Axes of an oriented box from the scatter matrix A (destroyed) of its points:
// their principal directions, made orthonormal in float (the coordinate axes when
// that set is not orthonormal to 1e-6; the float test, exact to 2e-7, takes 8e-7).
FRICP_HD inline void obb_axes(float A[3][3], float ax[3][3]) {
    float V[3][3];
    jacobi3f(A, V);
    float v0[3] = {V[0][0], V[1][0], V[2][0]}, v1[3] = {V[0][1], V[1][1], V[2][1]};
    const float i0 = 1.0f / sqrtf(fmaf(v0[2], v0[2], fmaf(v0[1], v0[1], v0[0] * v0[0])));
    for (int a = 0; a < 3; ++a) v0[a] *= i0;
    const float d01 = fmaf(v0[2], v1[2], fmaf(v0[1], v1[1], v0[0] * v1[0]));
    for (int a = 0; a < 3; ++a) v1[a] = fmaf(-d01, v0[a], v1[a]);
    const float i1 = 1.0f / sqrtf(fmaf(v1[2], v1[2], fmaf(v1[1], v1[1], v1[0] * v1[0])));
    for (int a = 0; a < 3; ++a) v1[a] *= i1;
    for (int a = 0; a < 3; ++a) {
        const int b = a == 2 ? 0 : a + 1, c = a == 0 ? 2 : a - 1;
        ax[0][a] = v0[a];
        ax[1][a] = v1[a];
        ax[2][a] = fmaf(v0[b], v1[c], -(v0[c] * v1[b]));
    }
    bool ortho = true;
    for (int a = 0; a < 3; ++a)
        for (int b = a; b < 3; ++b) {
            const float g = fmaf(ax[a][2], ax[b][2], fmaf(ax[a][1], ax[b][1], ax[a][0] * ax[b][0]));
            if (!(fabsf(g - (a == b ? 1.0f : 0.0f)) <= 8e-7f)) ortho = false;
        }
    if (!ortho)
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) ax[a][b] = a == b ? 1.0f : 0.0f;
}

// Half-extent h measured in float (each term of a point's extent is off by at most
// 5.2e-7 of the radius r, as in obb_eval), widened to cover that and the test's own
// rounding, rounded up.
FRICP_HD inline float obb_widen(float h, float r) {
    return f32_round_up((double)h * (1.0 + 2e-6) + 4e-6 * (double)r + 1e-37);
}

// Oriented box of the cnt >= 1 points p[0 .. cnt) (.w unused), written as
// out[0 .. 3] = (c, h0) (a0, h1) (a1, h2) (a2, r): axes along the points'
// principal directions (those float axes are what the box is exact for), the
// points' extents along them about a float centre c, and their radius r about it.
// All in float: the differences p - c are rounded relative to themselves, however
// far the points are from the origin. (With FP64 axes and extents, 64 cycles an
// instruction, the boxes of 500,000 points took 79 us, and 47 us of 100,000.)
FRICP_HD inline void obb_fit(const float4 *p, int cnt, float4 out[4]) {
    float c[3] = {p[0].x, p[0].y, p[0].z};
    float s[3] = {0.0f, 0.0f, 0.0f};
    for (int j = 1; j < cnt; ++j) {
        s[0] += p[j].x - c[0];
        s[1] += p[j].y - c[1];
        s[2] += p[j].z - c[2];
    }
    const float ic = 1.0f / (float)cnt;
    for (int a = 0; a < 3; ++a) c[a] = fmaf(s[a], ic, c[a]);
    float A[3][3] = {{0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f}};
    for (int j = 0; j < cnt; ++j) {
        const float d[3] = {p[j].x - c[0], p[j].y - c[1], p[j].z - c[2]};
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) A[a][b] = fmaf(d[a], d[b], A[a][b]);
    }
    float ax[3][3];
    obb_axes(A, ax);
    // extents about the mean, then about the float centre of the box
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int j = 0; j < cnt; ++j) {
        const float d[3] = {p[j].x - c[0], p[j].y - c[1], p[j].z - c[2]};
        for (int k = 0; k < 3; ++k) {
            const float u = fmaf(ax[k][2], d[2], fmaf(ax[k][1], d[1], ax[k][0] * d[0]));
            lo[k] = fminf(lo[k], u);
            hi[k] = fmaxf(hi[k], u);
        }
    }
    const float m[3] = {0.5f * (lo[0] + hi[0]), 0.5f * (lo[1] + hi[1]), 0.5f * (lo[2] + hi[2])};
    for (int a = 0; a < 3; ++a) c[a] += fmaf(m[2], ax[2][a], fmaf(m[1], ax[1][a], m[0] * ax[0][a]));
    float h[3] = {0.0f, 0.0f, 0.0f}, r2 = 0.0f;
    for (int j = 0; j < cnt; ++j) {
        const float d[3] = {p[j].x - c[0], p[j].y - c[1], p[j].z - c[2]};
        for (int k = 0; k < 3; ++k)
            h[k] = fmaxf(h[k], fabsf(fmaf(ax[k][2], d[2], fmaf(ax[k][1], d[1], ax[k][0] * d[0]))));
        r2 = fmaxf(r2, fmaf(d[2], d[2], fmaf(d[1], d[1], d[0] * d[0])));
    }
    const float r = sqrtf(r2) * (1.0f + 1e-6f);
    for (int k = 0; k < 3; ++k) h[k] = obb_widen(h[k], r);
    out[0] = make_float4(c[0], c[1], c[2], h[0]);
    out[1] = make_float4(ax[0][0], ax[0][1], ax[0][2], h[1]);
    out[2] = make_float4(ax[1][0], ax[1][1], ax[1][2], h[2]);
    out[3] = make_float4(ax[2][0], ax[2][1], ax[2][2], r);
}

// Oriented box of a patch of cnt >= 0 points, in the same form, by a team of nt
// threads: thread t takes points t, t + nt, ... and fold(v, k, max) leaves the sum
// (or maximum) of v[0 .. k) over the team in all of them. Axes of the points'
// scatter about c0 (the middle of their axis-aligned box), extents and radius about
// the middle of the extents, widened as obb_fit's. Nothing of a patch without points
// is used.
template <class Fold>
FRICP_HD inline void obb_fit_patch(const float4 *p, int cnt, const float c0[3], int t, int nt, Fold fold,
                                   float4 out[4]) {
    float c[3] = {c0[0], c0[1], c0[2]};
    float v[9] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    for (int k = t; k < cnt; k += nt) {
        const float d[3] = {p[k].x - c[0], p[k].y - c[1], p[k].z - c[2]};
        v[0] += d[0];
        v[1] += d[1];
        v[2] += d[2];
        v[3] = fmaf(d[0], d[0], v[3]);
        v[4] = fmaf(d[0], d[1], v[4]);
        v[5] = fmaf(d[0], d[2], v[5]);
        v[6] = fmaf(d[1], d[1], v[6]);
        v[7] = fmaf(d[1], d[2], v[7]);
        v[8] = fmaf(d[2], d[2], v[8]);
    }
    fold(v, 9, false);
    const float ic = 1.0f / fmaxf((float)cnt, 1.0f);
    const float xy = v[4] - v[0] * v[1] * ic, xz = v[5] - v[0] * v[2] * ic, yz = v[7] - v[1] * v[2] * ic;
    float A[3][3] = {{v[3] - v[0] * v[0] * ic, xy, xz}, {xy, v[6] - v[1] * v[1] * ic, yz},
                     {xz, yz, v[8] - v[2] * v[2] * ic}};
    float a[3][3];
    obb_axes(A, a);
    float e[6] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY, -INFINITY, -INFINITY};   // max u, max -u
    for (int k = t; k < cnt; k += nt) {
        const float d[3] = {p[k].x - c[0], p[k].y - c[1], p[k].z - c[2]};
        for (int r = 0; r < 3; ++r) {
            const float u = fmaf(a[r][2], d[2], fmaf(a[r][1], d[1], a[r][0] * d[0]));
            e[r] = fmaxf(e[r], u);
            e[3 + r] = fmaxf(e[3 + r], -u);
        }
    }
    fold(e, 6, true);
    if (cnt > 0) {   // the middle of the extents
        const float m[3] = {0.5f * (e[0] - e[3]), 0.5f * (e[1] - e[4]), 0.5f * (e[2] - e[5])};
        for (int r = 0; r < 3; ++r) c[r] += fmaf(m[2], a[2][r], fmaf(m[1], a[1][r], m[0] * a[0][r]));
    }
    float h[4] = {0.0f, 0.0f, 0.0f, 0.0f};   // half-extents and radius^2 about the float centre
    for (int k = t; k < cnt; k += nt) {
        const float d[3] = {p[k].x - c[0], p[k].y - c[1], p[k].z - c[2]};
        for (int r = 0; r < 3; ++r) h[r] = fmaxf(h[r], fabsf(fmaf(a[r][2], d[2], fmaf(a[r][1], d[1], a[r][0] * d[0]))));
        h[3] = fmaxf(h[3], fmaf(d[2], d[2], fmaf(d[1], d[1], d[0] * d[0])));
    }
    fold(h, 4, true);
    const float r = sqrtf(h[3]) * (1.0f + 1e-6f);
    for (int k = 0; k < 3; ++k) h[k] = obb_widen(h[k], r);
    out[0] = make_float4(c[0], c[1], c[2], h[0]);
    out[1] = make_float4(a[0][0], a[0][1], a[0][2], h[1]);
    out[2] = make_float4(a[1][0], a[1][1], a[1][2], h[2]);
    out[3] = make_float4(a[2][0], a[2][1], a[2][2], r);
}

// Squared distance from x = xh + xl to the box (c, h0) (a0, h1) (a1, h2) (a2, .),
// in float. Against the widening of obb_fit, the float rounding of
// u = A ((xh - c) + xl) (at most ~5.2e-7 of |x - c| per axis) leaves the result
// at most (1 + 8e-6) times the squared distance to the nearest of the box's
// points.
FRICP_HD inline float obb_eval(float4 c, float4 a0, float4 a1, float4 a2, const float xh[3], const float xl[3]) {
    const float dx = (xh[0] - c.x) + xl[0];
    const float dy = (xh[1] - c.y) + xl[1];
    const float dz = (xh[2] - c.z) + xl[2];
    const float e0 = fmaxf(fabsf(fmaf(a0.z, dz, fmaf(a0.y, dy, a0.x * dx))) - c.w, 0.0f);
    const float e1 = fmaxf(fabsf(fmaf(a1.z, dz, fmaf(a1.y, dy, a1.x * dx))) - a0.w, 0.0f);
    const float e2 = fmaxf(fabsf(fmaf(a2.z, dz, fmaf(a2.y, dy, a2.x * dx))) - a1.w, 0.0f);
    return fmaf(e2, e2, fmaf(e1, e1, e0 * e0));
}

}  // namespace fricp
