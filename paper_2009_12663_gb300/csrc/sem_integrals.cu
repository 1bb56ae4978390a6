// Time integrals of the diagonal preconditioners P1..P4 (Eqs. 5-8, A21-A22)
// from stored levels (sm_103a), for meshes whose time loop is resident
// (sem_resident.cu).
//
// The preconditioner steps of sem_step.cu form the integrals beside the time
// step: every step a CTA loads its windows twice, sums twice over the elements
// through shared memory in four colour passes, and reads, adds to and writes
// four node maps; one step took 38 us at 81 x 21 elements and 5 shots, where
// the resident loop needs 4.5 us.  Here the passes only store their levels (the
// displacement, and one field's acceleration), and the integrals are sums over
// time at fixed nodes and elements: a thread keeps its sums in registers and
// streams through the levels (800 steps of those 5 shots: 0.61 ms for the strains
// and 0.02 ms for their assembly, 0.36 ms at the nodes, beside 7.0 ms for the
// two passes).  Bound by those reads (16 B a node, level and field) and, for the
// strains, by the few warps their registers allow: 14 chunks of time there; five took
// 0.85 ms.
//
// S0 = sum a . a (one field) or sum (second difference of u) . a, at nodes;
// S1..S3 = sums of [div div', exx exx' + ezz ezz', gam gam'] of the
// undivided time differences, at the elements' points, assembled to nodes
// once at the end.  A step's terms are rounded as in the preconditioner steps
// (differences of the stored levels, product, then the quadrature weight): where
// a field has only just arrived the terms are denormal numbers, whose sums are
// exact in any order, so both forms agree there too about what is zero.

#include <algorithm>

#include "gbfwi_internal.h"
#include "sem_element.h"
#include "size_rules.h"

using namespace sem;

namespace {

__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return make_float2(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y)); }

// differences of two levels over the element patch at node g: hi - lo
__device__ __forceinline__ void load_difference(const float2 *__restrict__ hi, const float2 *__restrict__ lo, int g, int pitch,
                                                float2 (&d)[25])
{
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const float4 *h = reinterpret_cast<const float4 *>(hi + g + j * pitch), *l = reinterpret_cast<const float4 *>(lo + g + j * pitch);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float4 A = __ldg(h + i), B = __ldg(l + i);
            d[j * 5 + 2 * i] = sub2(make_float2(A.x, A.y), make_float2(B.x, B.y));
            d[j * 5 + 2 * i + 1] = sub2(make_float2(A.z, A.w), make_float2(B.z, B.w));
        }
        d[j * 5 + 4] = sub2(__ldg(hi + g + j * pitch + 4), __ldg(lo + g + j * pitch + 4));
    }
}

// One thread an element, steps [chunk * steps, + steps) of blockIdx.y, shot
// blockIdx.z; esum [chunk][shot][75][elements].
// TWO: products of the differences of a and b (step j pairs a's levels j, j + 1
// with b's nt - j, nt - j + 1); otherwise squares of a's.  Chunks of time give
// a small mesh enough warps to cover the loads.
template <bool TWO>
__global__ void __launch_bounds__(128) strain_integral_kernel(const float2 *__restrict__ a, const float2 *__restrict__ b,
                                                              long long lev, long long NP, int pitch, int nex, int ne, int nt,
                                                              int steps, float *__restrict__ esum)
{
    const int e = blockIdx.x * 128 + threadIdx.x;
    if (e >= ne) return;
    const int ez = e / nex, g = 4 * ez * pitch + 4 * (e - ez * nex);
    a += blockIdx.z * NP;
    b += blockIdx.z * NP;
    const int j0 = blockIdx.y * steps, j1 = min(nt, j0 + steps);
    float s[75];
#pragma unroll
    for (int q = 0; q < 75; ++q) s[q] = 0.f;
#pragma unroll 1
    for (int j = j0; j < j1; ++j) {
        float2 pa[25], pb[25];
        load_difference(a + (j + 1) * lev, a + j * lev, g, pitch, pa);
        if (TWO) load_difference(b + (nt - j + 1) * lev, b + (nt - j) * lev, g, pitch, pb);
#pragma unroll
        for (int q = 0; q < 25; ++q) {
            float2 ax, ae, bx, be;
            grad_at(pa, q % 5, q / 5, ax, ae);
            if (TWO) {
                grad_at(pb, q % 5, q / 5, bx, be);
            } else {
                bx = ax;
                be = ae;
            }
            const float ww = weight(q % 5, q / 5);
            const float da = __fadd_rn(ax.x, ae.y), db = __fadd_rn(bx.x, be.y);
            const float ga = __fadd_rn(ae.x, ax.y), gb = __fadd_rn(be.x, bx.y);
            s[3 * q] = __fadd_rn(s[3 * q], __fmul_rn(ww, __fmul_rn(da, db)));
            s[3 * q + 1] = __fadd_rn(s[3 * q + 1], __fmul_rn(ww, fmaf(ax.x, bx.x, __fmul_rn(ae.y, be.y))));
            s[3 * q + 2] = __fadd_rn(s[3 * q + 2], __fmul_rn(ww, __fmul_rn(ga, gb)));
        }
    }
    float *o = esum + ((long long)blockIdx.y * gridDim.z + blockIdx.z) * 75 * ne + e;
#pragma unroll
    for (int q = 0; q < 75; ++q) o[(long long)q * ne] = s[q];
}

// node maps 1..3 of shot blockIdx.y: the element sums over time chunks and over
// the elements around the node
__global__ void strain_assemble_kernel(const float *__restrict__ esum, int chunks, int nshot, int nex, int nez, int nx, int nz,
                                       int pitch, long long NP, float *__restrict__ acc)
{
    const long long N = (long long)nx * nz;
    const int ne = nex * nez;
    acc += (long long)blockIdx.y * 4 * NP;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < N; q += (long long)gridDim.x * blockDim.x) {
        const int iz = (int)(q / nx), ix = (int)(q - (long long)iz * nx);
        float s[3] = {0.f, 0.f, 0.f};
        for (int r = 0; r < 4; ++r) {                    // elements (ex, ez), (ex-1, ez), (ex, ez-1), (ex-1, ez-1)
            const int ez = iz / 4 - (r >> 1), ex = ix / 4 - (r & 1), j = iz - 4 * ez, i = ix - 4 * ex;
            if (ez < 0 || ex < 0 || ez >= nez || ex >= nex || i > 4 || j > 4) continue;
            const float *o = esum + (long long)blockIdx.y * 75 * ne + (long long)3 * (j * 5 + i) * ne + ez * nex + ex;
            float t[3] = {0.f, 0.f, 0.f};
            for (int c = 0; c < chunks; ++c, o += (long long)nshot * 75 * ne)
#pragma unroll
                for (int k = 0; k < 3; ++k) t[k] += o[(long long)k * ne];
#pragma unroll
            for (int k = 0; k < 3; ++k) s[k] += t[k];
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) acc[(k + 1) * NP + (long long)iz * pitch + ix] = s[k];
    }
}

// node map 0 of shot blockIdx.y: a holds the acceleration that made the
// displacement level of its slot.  TWO: u's second difference at levels
// nt - j + 1, nt - j, nt - j - 1 times the acceleration of step j.
template <bool TWO>
__global__ void __launch_bounds__(128) mass_integral_kernel(const float2 *__restrict__ a, const float2 *__restrict__ u,
                                                            long long lev, long long NP, int nx, int nz, int pitch, int nt,
                                                            float *__restrict__ acc)
{
    const long long N = (long long)nx * nz;
    const long long q = blockIdx.x * 128LL + threadIdx.x;
    if (q >= N) return;
    const int iz = (int)(q / nx), ix = (int)(q - (long long)iz * nx);
    const long long g = blockIdx.y * NP + (long long)iz * pitch + ix;
    a += g + 2 * lev;                                    // step j: slot j + 2
    u += g;
    float2 p0, p1;
    if (TWO) {
        p0 = u[(nt + 1) * lev];
        p1 = u[nt * lev];
    }
    float s = 0.f;
    int j = 0;
    auto step = [&](float2 an, float2 p2) {
        if (TWO) {
            const float2 f = sub2(sub2(p0, p1), sub2(p1, p2));
            s = __fadd_rn(s, fmaf(f.x, an.x, __fmul_rn(f.y, an.y)));
            p0 = p1;
            p1 = p2;
        } else {
            s = __fadd_rn(s, fmaf(an.x, an.x, __fmul_rn(an.y, an.y)));
        }
    };
    constexpr int U = 8;                                 // steps whose loads are in flight together
    for (; j + U <= nt; j += U) {
        float2 an[U], un[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            an[i] = __ldg(a + (j + i) * lev);
            un[i] = TWO ? __ldg(u + (nt - 1 - j - i) * lev) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < U; ++i) step(an[i], un[i]);
    }
    for (; j < nt; ++j) step(a[j * lev], TWO ? u[(nt - 1 - j) * lev] : make_float2(0.f, 0.f));
    acc[blockIdx.y * 4 * NP + (long long)iz * pitch + ix] = s;
}

}  // namespace

size_t gb_integral_bytes(const gbfwi_mesh *m, int B)
{
    return sizes::integral_bytes((long long)m->d.nex * m->d.nez, m->d.nt, B);
}

int gb_time_integrals(const gbfwi_mesh *m, int B, const float2 *w, const float2 *a, const float2 *u, bool strains,
                      const DevBuf &esums, float *acc, cudaStream_t s)
{
    const int nt = m->d.nt, ne = m->d.nex * m->d.nez;
    if (strains && esums.bytes < gb_integral_bytes(m, B)) return GBFWI_EINVAL;
    float *esum = esums.as<float>();
    const long long NP = (long long)m->nz * m->pitch, N = (long long)m->nx * m->nz, lev = B * NP;
    const dim3 gm((unsigned)((N + 127) / 128), (unsigned)B);
    if (u)
        mass_integral_kernel<true><<<gm, 128, 0, s>>>(a, u, lev, NP, m->nx, m->nz, m->pitch, nt, acc);
    else
        mass_integral_kernel<false><<<gm, 128, 0, s>>>(a, a, lev, NP, m->nx, m->nz, m->pitch, nt, acc);
    GB_LAUNCHED();
    if (!strains) return GBFWI_OK;
    const int nc = sizes::strain_chunks(ne, nt), steps = (nt + nc - 1) / nc;
    const dim3 gs((unsigned)((ne + 127) / 128), (unsigned)nc, (unsigned)B);
    if (u)
        strain_integral_kernel<true><<<gs, 128, 0, s>>>(w, u, lev, NP, m->pitch, m->d.nex, ne, nt, steps, esum);
    else
        strain_integral_kernel<false><<<gs, 128, 0, s>>>(w, w, lev, NP, m->pitch, m->d.nex, ne, nt, steps, esum);
    GB_LAUNCHED();
    strain_assemble_kernel<<<dim3((unsigned)std::min<long long>((N + 255) / 256, 2048), (unsigned)B), 256, 0, s>>>(
        esum, nc, B, m->d.nex, m->d.nez, m->nx, m->nz, m->pitch, NP, acc);
    GB_LAUNCHED();
    return GBFWI_OK;
}
