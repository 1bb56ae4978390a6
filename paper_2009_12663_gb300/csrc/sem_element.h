// Arithmetic of one spectral element and of one node's time step, shared by
// every time-step kernel (sem_step.cu, sem_resident.cu) so that all of them
// round alike: results do not depend on the kernel, the tile shape or the
// batching.  Internal to the gbfwi library.
#pragma once

#include <cuda_runtime.h>

namespace sem {

// D[i * 5 + k] = l_k'(xi_i) for the five GLL points -1, -sqrt(3/7), 0,
// sqrt(3/7), 1 (the three middle diagonal entries vanish), as literals: each
// product then takes its factor as an immediate operand.
__device__ __forceinline__ constexpr float D(int q)
{
    constexpr float t[25] = {-5.0f,        6.75650249f,  -2.66666667f, 1.41016418f,  -0.5f,
                             -1.24099025f, 0.0f,         1.74574312f,  -0.763762616f, 0.259009747f,
                             0.375f,       -1.33658458f, 0.0f,         1.33658458f,  -0.375f,
                             -0.259009747f, 0.763762616f, -1.74574312f, 0.0f,        1.24099025f,
                             0.5f,         -1.41016418f, 2.66666667f,  -6.75650249f, 5.0f};
    return t[q];
}

// the factor D[i][k] is zero and its product is left out
__device__ __forceinline__ constexpr bool dzero(int i, int k) { return i == k && i > 0 && i < 4; }

// GLL quadrature weight w_i w_j of local point (i, j)
__device__ __forceinline__ constexpr float weight(int i, int j)
{
    constexpr double w[5] = {1.0 / 10.0, 49.0 / 90.0, 32.0 / 45.0, 49.0 / 90.0, 1.0 / 10.0};
    return (float)(w[i] * w[j]);
}

// derivatives at local point (i, j) of the patch p (index j * 5 + i):
// gx = d/dxi, ge = d/deta of (ux, uz)
__device__ __forceinline__ void grad_at(const float2 (&p)[25], int i, int j, float2 &gx, float2 &ge)
{
    gx = ge = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        if (!dzero(i, k)) {
            gx.x = fmaf(D(i * 5 + k), p[j * 5 + k].x, gx.x);
            gx.y = fmaf(D(i * 5 + k), p[j * 5 + k].y, gx.y);
        }
        if (!dzero(j, k)) {
            ge.x = fmaf(D(j * 5 + k), p[k * 5 + i].x, ge.x);
            ge.y = fmaf(D(j * 5 + k), p[k * 5 + i].y, ge.y);
        }
    }
}

// Element nodal forces K u accumulated row by row of local points: the
// stresses of row j give the xi-part of the nodes of row j and the eta-part
// of every node, so one row of stresses is live at a time.  lmrow(j, lm)
// gives row j of (lambda, mu).  The quadrature weight multiplies the stresses:
// folded into the moduli it saves 75 products, but the second time differences
// of P2 and P4 magnify the roundings of the field (the map of a 100 x 25 mesh at
// 5 Hz moved by 3e-5 when only those roundings changed).
template <class LmRow>
__device__ __forceinline__ void element_force(const float2 (&p)[25], LmRow lmrow, float2 (&f)[25])
{
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        float2 lm[5];
        lmrow(j, lm);
        float txx[5], tzz[5], txz[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            float2 gx, ge;
            grad_at(p, i, j, gx, ge);
            const float l2m = fmaf(2.f, lm[i].y, lm[i].x);
            txx[i] = __fmul_rn(weight(i, j), fmaf(l2m, gx.x, __fmul_rn(lm[i].x, ge.y)));
            tzz[i] = __fmul_rn(weight(i, j), fmaf(lm[i].x, gx.x, __fmul_rn(l2m, ge.y)));
            txz[i] = __fmul_rn(weight(i, j), __fmul_rn(lm[i].y, __fadd_rn(ge.x, gx.y)));
        }
#pragma unroll
        for (int n = 0; n < 5; ++n)
#pragma unroll
            for (int m = 0; m < 5; ++m) {
                float fx, fz;
                if (j == 0) {
                    fx = __fmul_rn(D(n), txz[m]);
                    fz = __fmul_rn(D(n), tzz[m]);
                } else {
                    fx = f[n * 5 + m].x;
                    fz = f[n * 5 + m].y;
                    if (!dzero(j, n)) {
                        fx = fmaf(D(j * 5 + n), txz[m], fx);
                        fz = fmaf(D(j * 5 + n), tzz[m], fz);
                    }
                }
                if (n == j) {
#pragma unroll
                    for (int i = 0; i < 5; ++i)
                        if (!dzero(i, m)) {
                            fx = fmaf(D(i * 5 + m), txx[i], fx);
                            fz = fmaf(D(i * 5 + m), txz[i], fz);
                        }
                }
                f[n * 5 + m] = make_float2(fx, fz);
            }
    }
}

// Strain products of two fields at local point (i, j), without the
// quadrature weight (shared nodes carry equal weights, so it enters once,
// where the node sums are used): x = div A div B, y = 2 exx exx' + 2 ezz ezz' + gam gam'
__device__ __forceinline__ float2 strain_products(const float2 (&a)[25], const float2 (&b)[25], int i, int j)
{
    float2 ax, ae, bx, be;
    grad_at(a, i, j, ax, ae);
    grad_at(b, i, j, bx, be);
    const float da = __fadd_rn(ax.x, ae.y), db = __fadd_rn(bx.x, be.y);
    const float ga = __fadd_rn(ae.x, ax.y), gb = __fadd_rn(be.x, bx.y);
    const float y = fmaf(__fmul_rn(2.f, ax.x), bx.x, fmaf(__fmul_rn(2.f, ae.y), be.y, __fmul_rn(ga, gb)));
    return make_float2(__fmul_rn(da, db), y);
}

__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}

// acceleration of an interior node (k = K u - F, mi = 1 / M)
__device__ __forceinline__ float2 accel(float2 k, float mi) { return make_float2(__fmul_rn(-k.x, mi), __fmul_rn(-k.y, mi)); }

// acceleration of an absorbing-edge node: bd = (Cx, Cz, 1/(M + dt/2 Cx), 1/(M + dt/2 Cz))
__device__ __forceinline__ float2 accel_edge(float2 k, float2 v, float4 bd)
{
    return make_float2(__fmul_rn(-fmaf(bd.x, v.x, k.x), bd.z), __fmul_rn(-fmaf(bd.y, v.y, k.y), bd.w));
}

// a + b c, component by component
__device__ __forceinline__ float2 axpy2(float s, float2 b, float2 a)
{
    return make_float2(fmaf(s, b.x, a.x), fmaf(s, b.y, a.y));
}

// Stacey weights (w.x, w.y) of an edge node times the correlation of u with
// the mean of the two half-step velocities
__device__ __forceinline__ float edge_product(float2 w, float2 u, float2 v, float2 vn)
{
    const float vx = __fmul_rn(0.5f, __fadd_rn(v.x, vn.x)), vz = __fmul_rn(0.5f, __fadd_rn(v.y, vn.y));
    return fmaf(__fmul_rn(w.x, u.x), vx, __fmul_rn(__fmul_rn(w.y, u.y), vz));
}

// correlation u . a
__device__ __forceinline__ float dot2(float2 u, float2 a) { return fmaf(u.x, a.x, __fmul_rn(u.y, a.y)); }

}  // namespace sem
