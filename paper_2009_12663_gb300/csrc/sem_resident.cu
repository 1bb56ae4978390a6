// Whole time loops of the spectral-element scheme in one cooperative launch
// (sm_103a): forward passes, receiver-field passes and adjoint-gradient passes
// of meshes whose fields fit the SMs' shared memory.
//
// The step kernels of sem_step.cu read and write every field once per launch
// (44 B a node forward, 76 B adjoint, from L2) and start cold each step; a
// mesh of a few tiles leaves the GPU to launch latency (8 us forward, 23 us
// adjoint a step measured on 12 x 6 elements).  Here a CTA keeps its tile for
// all steps: the displacement window, the moduli, the velocity and
// the accumulators stay in shared memory or registers, and between steps a
// CTA only trades the node lines its neighbours need.  Measured a step: 3.9 to 4.4 us
// forward (40 x 20 elements, one CTA an SM), 5.7 us with two shots an SM,
// 5.6 us adjoint; the chain of a step is the exchange (1.5 us), the
// forces (1.6 us), the update (0.8 us) and the sends (0.4 us).
//
// Tile and threads.  A CTA owns TX x TZ elements (chosen at run time) of one
// shot and recomputes the element column to its left and the row above, one
// thread per element of that (TX+1) x (TZ+1) extended tile, as in sem_step.cu;
// ownership of nodes and the order of every sum are the same, so results are
// bitwise equal to the step kernels.
//
// Shared layout.  Window cell c = rz * E + cx (E = TX + 1; the trailing node
// column of row rz is cell E (TZ+2) + rz) holds the 4 x 4 nodes of an element;
// float4 plane (j & 3) * 2 + (i >> 1) holds nodes (i, i+1) of row j of every
// cell, so a warp's patch reads are contiguous 16-byte accesses: the loop is
// bound by shared-memory wavefronts and the FMA pipe together (72% and 61%
// of peak measured on the force loop alone).
//
// Correlations.  In the adjoint pass one more thread per owned element adds
// the step's strain and mass correlations from the forward level, beside the
// exchange and the next forces: on the element threads they took 138 ms of the
// gradient on 340 x 70 elements and 500 steps that takes 96 ms so (130 ms with
// the step kernels).
//
// Exchange.  Every node another tile's window holds is sent as two 64-bit
// words (component, step tag) with relaxed gpu-scope stores; the reader polls
// the words themselves, so there is no flag, fence or grid barrier: one store
// and one load latency a step.  Two slots by step parity suffice: a CTA sends
// level n + 2 only after it has received level n + 1 of all its neighbours,
// which they sent after reading its level n.  Waits are bounded; one that
// gives up sets the mesh's status word, which ends every other wait.

#include <algorithm>
#include <climits>

#include "gbfwi_internal.h"
#include "resident_plan.h"
#include "sem_element.h"
#include "sm100.h"

using namespace resident;
using namespace sem;

namespace {

template <int NT_, int MODE>
struct Shape {
    static constexpr bool ADJ = MODE == MODE_ADJ_G;
    static constexpr Limits L = limits_of(NT_);
    static constexpr int NT = NT_;                              // element threads
    static constexpr int PS = L.cells, NO = L.owned;
    static constexpr int NP = corr_threads(NT_, ADJ);           // correlation threads (adjoint)
    static constexpr int THREADS = NT + NP;
    static constexpr int WIN = window_f4(NT_);                  // float4 of one window
    static constexpr int MINB = blocks_per_sm(NT_, ADJ);
    static constexpr int F4 = head_f4(NT_, ADJ);                // float4 before the exchange inside the tile
};

struct Word2 { unsigned long long x, z; };

__device__ __forceinline__ void send_node(Word2 *p, float2 v, unsigned tag)
{
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(t | __float_as_uint(v.x)),
                 "l"(t | __float_as_uint(v.y))
                 : "memory");
}

__device__ __forceinline__ Word2 poll_node(const Word2 *p)
{
    Word2 w;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.z) : "l"(p) : "memory");
    return w;
}

__device__ __forceinline__ bool has_tag(const Word2 &w, unsigned tag)
{
    return (unsigned)(w.x >> 32) == tag && (unsigned)(w.z >> 32) == tag;
}

// accumulation without a round trip; an address is only ever added to by one
// thread, in step order
__device__ __forceinline__ void red_add(float *p, float v)
{
    asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}

__device__ __forceinline__ void copy4_async(float *dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// 32-byte global accesses (one whole sector: the four nodes of an element row)
// and an 8-byte load that stay where they are written
struct Row4 { float2 n[4]; };

__device__ __forceinline__ Row4 load_row(const float2 *p)
{
    Row4 r;
    asm volatile("ld.global.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r.n[0].x), "=f"(r.n[0].y), "=f"(r.n[1].x), "=f"(r.n[1].y), "=f"(r.n[2].x), "=f"(r.n[2].y),
                   "=f"(r.n[3].x), "=f"(r.n[3].y)
                 : "l"(p)
                 : "memory");
    return r;
}

__device__ __forceinline__ void store_row(float2 *p, float4 u, float4 v)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(u.x), "f"(u.y), "f"(u.z),
                 "f"(u.w), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

__device__ __forceinline__ float2 load2(const void *p)
{
    float2 v;
    asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// patch of the element with cells c0 (own), c1 (next column), c0d, c1d (one row down)
template <int PS>
__device__ __forceinline__ void load_cells(const float4 *w, int c0, int c1, int c0d, int c1d, float2 (&p)[25])
{
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int ca = j == 4 ? c0d : c0, cb = j == 4 ? c1d : c1;
        const float4 A = w[((j & 3) * 2) * PS + ca], B = w[((j & 3) * 2 + 1) * PS + ca];
        p[j * 5] = make_float2(A.x, A.y);
        p[j * 5 + 1] = make_float2(A.z, A.w);
        p[j * 5 + 2] = make_float2(B.x, B.y);
        p[j * 5 + 3] = make_float2(B.z, B.w);
        p[j * 5 + 4] = *reinterpret_cast<const float2 *>(w + ((j & 3) * 2) * PS + cb);
    }
}

// barriers: 4 and 2 the element threads (window complete, or a wait gave up;
// next window written); 1 shares published and, in the adjoint, the correlations
// of the step before done (they read the window that is written next); 3
// accelerations written (element threads arrive, correlation threads wait).  The
// correlations of a step so run beside the exchange and the next forces.
template <int NT_, int MODE>
__global__ void __launch_bounds__((Shape<NT_, MODE>::THREADS), (Shape<NT_, MODE>::MINB))
    sem_resident_kernel(const ResidentArgs a)
{
    using S = Shape<NT_, MODE>;
    constexpr int NT = S::NT, PS = S::PS, NO = S::NO, NA = S::THREADS, kMaxHalo = S::L.halo;
    constexpr bool ADJ = S::ADJ, ACC = MODE == MODE_RCV;
    extern __shared__ float4 rsm[];
    float4 *win0 = rsm;                                          // field window [8][PS], two in the adjoint
    float4 *lmw = win0 + (ADJ ? 2 : 1) * S::WIN;                 // moduli window [8][PS]
    float4 *smi = lmw + S::WIN;                                  // 1/M [4][NT]
    float4 *sac = smi + 4 * NT;                                  // adjoint: accelerations [8][NO]
    float4 *sst = sac + 8 * NO;                                  // strain sums [13][NO] (25 points, 2 each)
    float4 *sma = sst + 13 * NO;                                 // mass sums [4][NO]
    float2 *zc = reinterpret_cast<float2 *>(rsm + S::F4);        // exchange inside the tile [9][NT]
    float *tail = reinterpret_cast<float *>(zc + 9 * NT);
    const int TX = a.TX, TZ = a.TZ, E = TX + 1, R = TZ + 2;
    const Tail o = tail_of(ADJ, a.ntiles == 1, TX, TZ, a.edge_cap, a.grp_cap, a.ent_cap, a.rec_cap);
    float4 *sedge = reinterpret_cast<float4 *>(tail + o.edge);
    float4 *sev = reinterpret_cast<float4 *>(tail + o.ev);
    float2 *svx = reinterpret_cast<float2 *>(tail + o.vx);
    __shared__ int s_nhalo, s_nsend, s_bad;

    const int t = threadIdx.x, b = blockIdx.y, tile = blockIdx.x;
    const int bx = tile % a.ntx, bz = tile / a.ntx;
    const int ex0 = bx * TX, ez0 = bz * TZ;
    const int ix0 = 4 * ex0 - 4, iz0 = 4 * ez0 - 4;
    const int pitch = a.pitch;
    const long long fo = (long long)b * a.fstride;
    const bool right = bx + 1 < a.ntx, left = bx > 0, below = bz + 1 < a.ntz, above = bz > 0;
    const int nex = min(TX, a.nex - ex0), nez = min(TZ, a.nez - ez0);   // elements this tile owns
    // nodes this tile owns: [4 ex0, ixe) x [4 ez0, ize)
    const int ixe = right ? 4 * (ex0 + TX) : a.nx, ize = below ? 4 * (ez0 + TZ) : a.nz;

    // ---- windows of the first step, from the fields; nodes to receive and to send
    const int wnx = min(ix0 + 4 * E + 1, a.nx) - ix0, wnz = min(iz0 + 4 * (TZ + 1) + 1, a.nz) - iz0;
    auto cell_of = [&](int cx, int rz) { return cx < E ? rz * E + cx : E * R + rz; };
    auto slot_of = [&](int wx, int wz) {                          // float2 slot of window node (wx, wz)
        const int i = wx & 3, j = wz & 3;
        return ((j * 2 + (i >> 1)) * PS + cell_of(wx >> 2, wz >> 2)) * 2 + (i & 1);
    };
#pragma unroll 1
    for (int q = t; q < S::F4; q += NA) rsm[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t == 0) s_bad = 0;
    __syncthreads();
    float4 *first = ADJ ? win0 + (a.n0 & 1) * S::WIN : win0;
#pragma unroll 1
    for (int q = t; q < wnx * wnz; q += NA) {
        const int wz = q / wnx, wx = q - wz * wnx, ix = ix0 + wx, iz = iz0 + wz;
        if (ix < 0 || iz < 0) continue;
        const int g = iz * pitch + ix, sl = slot_of(wx, wz);
        reinterpret_cast<float2 *>(first)[sl] = a.u0[fo + g];
        reinterpret_cast<float2 *>(lmw)[sl] = __ldg(a.lm + g);
    }
    // nodes to receive (warp 0) and to send (warp 1) as lists in node order, so that
    // a warp's words lie together (in list order of arrival they took 32 lines each)
    int2 *hlist = reinterpret_cast<int2 *>(tail + o.recv), *slist = reinterpret_cast<int2 *>(tail + o.send);
    if (a.ntiles > 1 && t < 64) {
        const bool recv = t < 32;
        int count = 0;
#pragma unroll 1
        for (int q0 = 0; q0 < wnx * wnz; q0 += 32) {
            const int q = q0 + (t & 31), wz = q / wnx, wx = q - wz * wnx, ix = ix0 + wx, iz = iz0 + wz;
            const bool in = q < wnx * wnz && ix >= 0 && iz >= 0;
            const bool mine = ix >= 4 * ex0 && ix < ixe && iz >= 4 * ez0 && iz < ize;
            const bool edge = (right && ix >= ixe - 4) || (below && iz >= ize - 4) || (left && ix == 4 * ex0) ||
                              (above && iz == 4 * ez0);
            const bool take = in && (recv ? !mine : mine && edge);
            const unsigned m = __ballot_sync(0xffffffffu, take);
            const int at = count + __popc(m & ((1u << (t & 31)) - 1));
            if (take) {
                const int2 v = make_int2(iz * pitch + ix, slot_of(wx, wz));
                (recv ? hlist : slist)[at] = v;
            }
            count += __popc(m);
        }
        if ((t & 31) == 0) (recv ? s_nhalo : s_nsend) = count;
    } else if (a.ntiles == 1 && t == 0) {
        s_nhalo = s_nsend = 0;
    }
    __syncthreads();
    const int nhalo = s_nhalo, nsend = s_nsend;

    float *accb = ADJ ? a.acc + (long long)b * a.acc_shot_stride : nullptr;
    const long long cs = a.acc_comp_stride;
    const int hE = 4 * TZ + 1, wE = 4 * TX + 1;
    // absorbing edges.  A free surface has no damping: its nodes update like
    // interior ones (their Stacey factors would be (0, 0, 1/M, 1/M)).  Slots in
    // sedge: the left side, the right, the top, the bottom.
    const int offR = a.ntx == 1 ? hE : 0, offT = offR + hE, offB = offT + (a.ntz == 1 && !a.free_top ? wE : 0);
    const bool side_l = !left, side_r = !right, flat_t = !above && !a.free_top, flat_b = !below;
    const int rows = ize - 4 * ez0, cols = ixe - 4 * ex0;         // owned node rows and columns
    auto for_edges = [&](int t0, int nt, auto &&fn) {             // fn(slot, rx, rz) of every edge node, nodes spread over threads
#pragma unroll 1
        for (int q = t0; q < 2 * rows + 2 * cols; q += nt) {
            if (q < rows) {
                if (side_l) fn(q, 0, q);
            } else if (q < 2 * rows) {
                if (side_r) fn(offR + q - rows, cols - 1, q - rows);
            } else {
                const int rx = q - 2 * rows < cols ? q - 2 * rows : q - 2 * rows - cols;
                const bool top = q - 2 * rows < cols;
                if ((side_l && rx == 0) || (side_r && rx == cols - 1)) continue;   // corners belong to the sides
                if (top ? flat_t : flat_b) fn((top ? offT : offB) + rx, rx, top ? 0 : rows - 1);
            }
        }
    };
    for_edges(t, NA, [&](int sl, int rx, int rz) {
        sedge[sl] = __ldg(a.bnd + (4 * ez0 + rz) * pitch + 4 * ex0 + rx);
        if (ADJ) sev[sl] = make_float4(0.f, 0.f, 0.f, 0.f);
    });
    // ---- receivers the tile records
    const int rb = a.rec_tptr[tile], nr = a.seis ? a.rec_tptr[tile + 1] - rb : 0;
#pragma unroll 1
    for (int q = t; q < nr; q += NA) {
        const int r = a.rec_list[rb + q];
        const int2 e = a.rec_e[r];
        const int cx = e.x - ex0 + 1, rz = e.y - ez0 + 1;
        reinterpret_cast<int4 *>(tail + o.rec)[q] =
            make_int4(r, cell_of(cx, rz) | cell_of(cx + 1, rz) << 16, cell_of(cx, rz + 1) | cell_of(cx + 1, rz + 1) << 16, 0);
    }
#pragma unroll 1
    for (int q = t; q < 25 * nr; q += NA) tail[o.recw + q] = a.recw[a.rec_list[rb + q / 25] * 25 + q % 25];

    if (ADJ && t >= NT) {
        // =====================================================================
        // correlation threads: one owned element each, off the path of the field
        // =====================================================================
        const int oi = t - NT;
        const bool on = oi < nex * nez;
        const int ez = on ? oi / nex : 0, ex = on ? oi - ez * nex : 0;   // within the tile
        const int slot = ez * TX + ex;                            // per-element arrays
        const int cx = ex + 1, rz = ez + 1;
        const int c0 = cell_of(cx, rz), c1 = cell_of(cx + 1, rz), c0d = cell_of(cx, rz + 1), c1d = cell_of(cx + 1, rz + 1);
        const int g00 = 4 * (ez0 + ez) * pitch + 4 * (ex0 + ex);
        float4 *est = reinterpret_cast<float4 *>(a.eacc) + ((long long)b * a.nez * a.nex + (long long)(ez0 + ez) * a.nex + ex0 + ex) * 13;
        if (on) {
#pragma unroll
            for (int q = 0; q < 13; ++q) sst[q * NO + slot] = est[q];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                sma[j * NO + slot] = *reinterpret_cast<const float4 *>(accb + 2 * cs + g00 + j * pitch);
        }
        __syncthreads();
        bar_arrive(1, NA);                                        // nothing to wait for in the first step
#pragma unroll 1
        for (int n = a.n0; n < a.n1; ++n) {
            const float2 *hist = a.hist + (long long)(a.nt - n - a.hist_k0) * a.lev + fo;
            float2 u[25];
            if (on)
#pragma unroll
                for (int j = 0; j < 5; ++j) {
                    const float2 *r = hist + g00 + j * pitch;
                    const Row4 A = load_row(r);
#pragma unroll
                    for (int i = 0; i < 4; ++i) u[j * 5 + i] = A.n[i];
                    u[j * 5 + 4] = load2(r + 4);
                }
            bar_sync(3, NA);                                      // this step's update is done
            if (s_bad) return;
            if (on) {
                // mass correlation u_k . a (the node's mass factor enters once, in the chain rule)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 A = sac[(2 * j) * NO + slot], B = sac[(2 * j + 1) * NO + slot];
                    float4 m = sma[j * NO + slot];
                    m.x += dot2(u[j * 5], make_float2(A.x, A.y));
                    m.y += dot2(u[j * 5 + 1], make_float2(A.z, A.w));
                    m.z += dot2(u[j * 5 + 2], make_float2(B.x, B.y));
                    m.w += dot2(u[j * 5 + 3], make_float2(B.z, B.w));
                    sma[j * NO + slot] = m;
                }
                // bring the forward level of the step after next into L2 (each level lies in new
                // pages: the address translation alone takes microseconds, and loads issued
                // behind it wait too, so it is started where none follow for a while)
                if (n + 2 < a.n1)
#pragma unroll
                    for (int j = 0; j < 4; ++j) prefetch_l2(hist - 2 * a.lev + g00 + j * pitch);
                float2 p[25];
                load_cells<PS>(win0 + (n & 1) * S::WIN, c0, c1, c0d, c1d, p);
                float2 c[2];
#pragma unroll
                for (int q = 0; q < 25; ++q) {
                    c[q & 1] = strain_products(p, u, q % 5, q / 5);
                    if (q & 1) {
                        float4 s = sst[(q >> 1) * NO + slot];
                        sst[(q >> 1) * NO + slot] = make_float4(s.x + c[0].x, s.y + c[0].y, s.z + c[1].x, s.w + c[1].y);
                    }
                }
                float2 &s = *reinterpret_cast<float2 *>(&sst[12 * NO + slot]);
                s = add2(s, c[0]);
            }
            // absorbing edges: the two Stacey terms, and the mass term of the extra lines.
            // Side edges: normal x, tangential z with weight wz; top and bottom the other way
            for_edges(t - NT, S::NP, [&](int sl, int rx, int rz_) {
                const int ix = 4 * ex0 + rx, iz = 4 * ez0 + rz_, g = iz * pitch + ix;
                const bool side = (side_l && rx == 0) || (side_r && rx == cols - 1);
                const bool flat = (flat_t && rz_ == 0) || (flat_b && rz_ == rows - 1);
                const float wz = side ? __ldg(a.wzs + iz) : 0.f, wx = flat ? __ldg(a.wxs + ix) : 0.f;
                const float2 uk = load2(hist + g);
                const float4 va = sev[sl];
                red_add(accb + 3 * cs + g, fmaf(__fmul_rn(wz, uk.x), va.x, __fmul_rn(__fmul_rn(wx, uk.y), va.y)));
                red_add(accb + 4 * cs + g, fmaf(__fmul_rn(wx, uk.x), va.x, __fmul_rn(__fmul_rn(wz, uk.y), va.y)));
                if (ix == a.nx - 1 || iz == a.nz - 1) red_add(accb + 2 * cs + g, dot2(uk, make_float2(va.z, va.w)));
            });
            if (n + 1 < a.n1) bar_arrive(1, NA);
        }
        if (on) {
#pragma unroll
            for (int q = 0; q < 13; ++q) est[q] = sst[q * NO + slot];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                *reinterpret_cast<float4 *>(accb + 2 * cs + g00 + j * pitch) = sma[j * NO + slot];
        }
        return;
    }

    // =========================================================================
    // element threads
    // =========================================================================
    const int elz = t / E, elx = t - elz * E;
    const int ex = ex0 - 1 + elx, ez = ez0 - 1 + elz;
    const bool evalid = elz <= TZ && ex >= 0 && ez >= 0 && ex < a.nex && ez < a.nez;
    const bool owns = evalid && elx >= 1 && elz >= 1;
    const int c0 = elz <= TZ ? t : 0;
    const int c1 = elx < TX ? c0 + 1 : E * R + min(elz, TZ);
    const int c0d = c0 + E, c1d = elx < TX ? c0d + 1 : c1 + 1;
    const int oi = (elz - 1) * TX + elx - 1;                     // per-element arrays
    const int g00 = 4 * ez * pitch + 4 * ex;                     // node (0, 0)
    // slots of node (0, 0) on the left side / the absorbing top, or negative
    const int eL = ex == 0 ? 4 * (elz - 1) : -64, eT = ez == 0 && !a.free_top ? offT + 4 * (elx - 1) : -64;
    auto lmrow = [&](int j, float2(&lm)[5]) {
        const int ca = j == 4 ? c0d : c0, cb = j == 4 ? c1d : c1;
        const float4 A = lmw[((j & 3) * 2) * PS + ca], B = lmw[((j & 3) * 2 + 1) * PS + ca];
        lm[0] = make_float2(A.x, A.y);
        lm[1] = make_float2(A.z, A.w);
        lm[2] = make_float2(B.x, B.y);
        lm[3] = make_float2(B.z, B.w);
        lm[4] = *reinterpret_cast<const float2 *>(lmw + ((j & 3) * 2) * PS + cb);
    };
    // the extra node lines of the mesh's last column and row, all on absorbing
    // edges: column nodes q < ncol at (4 nex, q), then row nodes at (q - ncol, 4 nez)
    const int ncol = right ? 0 : rows, nextra = ncol + (below ? 0 : 4 * nex);

    // ---- per-element state
    float2 *vhb = a.vh + fo;
    float4 vr[8];                                                 // half-step velocity
    if (owns)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long g = g00 + j * pitch;
            vr[2 * j] = *reinterpret_cast<const float4 *>(vhb + g);
            vr[2 * j + 1] = *reinterpret_cast<const float4 *>(vhb + g + 2);
            smi[j * NT + t] = *reinterpret_cast<const float4 *>(a.minv + g);
        }
#pragma unroll 1
    for (int q = t; q < nextra; q += NT)
        svx[q] = vhb[q < ncol ? (4 * ez0 + q) * pitch + a.nx - 1 : (a.nz - 1) * pitch + 4 * ex0 + q - ncol];
    // ---- injections of the tile: entries, groups (nodes), and the nodes of this
    // thread that receive one, as a mask and the first group
    const int src_id = a.shot_map ? a.shot_map[b] : b;
    const int *gp = a.gptr + (a.per_shot_groups ? (long long)src_id * (a.ntiles + 1) : 0);
    const int gb = gp[tile], ng = gp[tile + 1] - gb;
    const int eb = ng > 0 ? a.groups[gb].begin : 0, ne = ng > 0 ? a.groups[gb + ng - 1].end - eb : 0;
    const int4 *sent = reinterpret_cast<const int4 *>(tail + o.ent);
    float2 *sinj = reinterpret_cast<float2 *>(tail + o.inj);
    float *ssig = tail + o.sig;
    unsigned imask = 0;
    int ibase = 0;
#pragma unroll 1
    for (int g = ng - 1; g >= 0; --g) {
        const int node = a.groups[gb + g].node;
        if (node >> 5 == t) {
            imask |= 1u << (node & 31);
            ibase = g;
        }
    }
#pragma unroll 1
    for (int g = t; g <= ng; g += NT) reinterpret_cast<int *>(tail + o.grp)[g] = g < ng ? a.groups[gb + g].begin - eb : ne;
#pragma unroll 1
    for (int e = t; e < ne; e += NT) {
        const InjEntry I = a.entries[eb + e];
        reinterpret_cast<int4 *>(tail + o.ent)[e] = make_int4(I.cx * a.sig_chan_stride, I.cz * a.sig_chan_stride,
                                                              __float_as_int(I.wx), __float_as_int(I.wz));
    }
    // places of the extra nodes: this element's share in zc and the left or upper
    // neighbour's (or -1), the window slot, the edge slot and 1 + the injection group
    int4 *sxi = reinterpret_cast<int4 *>(tail + o.xi);
#pragma unroll 1
    for (int q = t; q < nextra; q += NT) {
        const bool col = q < ncol;
        const int rx = col ? 4 * nex : q - ncol, rz = col ? q : 4 * nez;      // owned node (rx, rz)
        const int qx = col ? nex : rx / 4 + 1, qz = col ? min(rz / 4, nez - 1) + 1 : nez;
        const int te = qz * E + qx, i = rx - 4 * (qx - 1), j = rz - 4 * (qz - 1);   // its element and local node
        const int other = i == 4 ? (j == 0 ? 4 * NT + te - E : -1) : (i == 0 ? 4 * NT + te - 1 : -1);
        int grp = 0;
#pragma unroll 1
        for (int g = 0; g < ng; ++g)
            if (a.groups[gb + g].node == te * 32 + j * 5 + i) grp = g + 1;
        const int sl = col ? offR + rz : (side_l && rx == 0) ? rz : offB + rx;
        sxi[q] = make_int4((i == 4 ? j : 5 + i) * NT + te, other, slot_of(rx + 4, rz + 4), sl | grp << 16);
    }
    const float *sig = a.sig + (long long)src_id * a.sig_shot_stride;
    Word2 *xch = reinterpret_cast<Word2 *>(a.xch) + (long long)b * a.xstride;
    __syncthreads();

    // signals of step n into their half of ssig (asynchronous)
    auto fetch_signals = [&](int n) {
        const int ts = ADJ || (ACC && a.reverse) ? a.nt - 1 - n : n + 1;
#pragma unroll 1
        for (int e = t; e < ne; e += NT) {
            const int4 I = sent[e];
            float *d = ssig + (n & 1) * 2 * a.ent_cap + 2 * e;
            copy4_async(d, sig + I.x + ts);
            copy4_async(d + 1, sig + I.y + ts);
        }
    };
    fetch_signals(a.n0);
    // the owned nodes of level k from window w to the level's field
    auto store_level = [&](int k, const float4 *w) {
        float2 *ob = a.out + (long long)(a.out_ring ? k % 3 : k - a.out_k0) * a.lev + fo;
        if (owns)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                store_row(ob + g00 + j * pitch, w[(2 * j) * PS + c0], w[(2 * j + 1) * PS + c0]);
#pragma unroll 1
        for (int q = t; q < nextra; q += NT) {
            const int rx = q < ncol ? 4 * nex : q - ncol, rz = q < ncol ? q : 4 * nez;
            ob[(4 * ez0 + rz) * pitch + 4 * ex0 + rx] = reinterpret_cast<const float2 *>(w)[sxi[q].z];
        }
        // the next level lies in new pages: have their translation ready
        if (!a.out_ring && t < 2 && k <= a.n1) prefetch_l2(ob + a.lev + (t ? ize - 1 : 4 * ez0) * pitch + 4 * ex0);
    };
    const float dt = a.dt;
#pragma unroll 1
    for (int n = a.n0; n < a.n1; ++n) {
        const int par = n & 1;
        float4 *win = ADJ ? win0 + par * S::WIN : win0;            // level n + 1
        float4 *nxt = ADJ ? win0 + (par ^ 1) * S::WIN : win0;      // level n + 2
        // ---- halo of the current level
        bool bad = false;
        if (n > a.n0) {
            const unsigned tag = (unsigned)(n - a.n0);
            const Word2 *src = xch + (long long)par * a.xslot;
            Word2 w[kMaxHalo];
#pragma unroll
            for (int h = 0; h < kMaxHalo; ++h)
                if (t + h * NT < nhalo) w[h] = poll_node(src + hlist[t + h * NT].x);
            if (n + 1 >= a.out_from) store_level(n + 1, win);     // while the words are under way
#pragma unroll
            for (int h = 0; h < kMaxHalo; ++h)
                if (t + h * NT < nhalo) {
                    const int2 at = hlist[t + h * NT];
                    if (!has_tag(w[h], tag)) {
                        const long long t0 = clock64();
                        int spin = 0;
                        while (!bad) {
                            w[h] = poll_node(src + at.x);
                            if (has_tag(w[h], tag)) break;
                            if ((++spin & 255) == 0 && *reinterpret_cast<volatile int *>(a.status)) bad = true;
                            if (clock64() - t0 > sm100::kWaitCycles) bad = true;
                        }
                    }
                    reinterpret_cast<float2 *>(win)[at.y] =
                        make_float2(__uint_as_float((unsigned)w[h].x), __uint_as_float((unsigned)w[h].z));
                }
        }
        if (ne > 0) asm volatile("cp.async.wait_all;" ::: "memory");
        if (bad) s_bad = 1;
        bar_sync(4, NT);
        if (s_bad) {                                              // a wait gave up: flag it and leave
            if (t == 0) atomicExch(a.status, 1);
            if (ADJ) bar_arrive(3, NA);
            return;
        }
        // ---- injected forces of this step, records
        if (ng > 0) {
            if (n + 1 < a.n1) fetch_signals(n + 1);
            const int *grp = reinterpret_cast<const int *>(tail + o.grp);
#pragma unroll 1
            for (int g = t; g < ng; g += NT) {
                float fx = 0.f, fz = 0.f;
#pragma unroll 1
                for (int q = grp[g]; q < grp[g + 1]; ++q) {
                    const int4 I = sent[q];
                    const float *d = ssig + par * 2 * a.ent_cap + 2 * q;
                    fx = fmaf(__int_as_float(I.z), d[0], fx);
                    fz = fmaf(__int_as_float(I.w), d[1], fz);
                }
                sinj[g] = make_float2(-fx * a.sig_scale, -fz * a.sig_scale);
            }
        }
#pragma unroll 1
        for (int q = t; q < 2 * nr; q += NT) {
            const int4 I = reinterpret_cast<const int4 *>(tail + o.rec)[q >> 1];
            const float *wt = tail + o.recw + 25 * (q >> 1);
            const float *w = reinterpret_cast<const float *>(win) + (q & 1);
            float v[25], s = 0.f;
#pragma unroll
            for (int k = 0; k < 25; ++k) {
                const int i = k % 5, j = k / 5, cc = j < 4 ? I.y : I.z, cell = i < 4 ? cc & 0xffff : cc >> 16;
                v[k] = w[(((j & 3) * 2 + ((i & 3) >> 1)) * PS + cell) * 4 + (i & 1) * 2];
            }
#pragma unroll
            for (int k = 0; k < 25; ++k) s = fmaf(wt[k], v[k], s);
            a.seis[(long long)b * a.seis_shot_stride + (long long)(I.x * 2 + (q & 1)) * a.nt + n] = s;
        }
        // ---- element forces; the i = 4 column and the j = 4 row are published
        float2 f[16];
        if (evalid) {
            float2 p[25], fe[25];
            load_cells<PS>(win, c0, c1, c0d, c1d, p);
            element_force(p, lmrow, fe);
#pragma unroll
            for (int j = 0; j < 5; ++j) zc[j * NT + t] = fe[j * 5 + 4];
#pragma unroll
            for (int i = 0; i < 4; ++i) zc[(5 + i) * NT + t] = fe[20 + i];
#pragma unroll
            for (int q = 0; q < 16; ++q) f[q] = fe[q / 4 * 5 + q % 4];
        } else {
#pragma unroll
            for (int q = 0; q < 9; ++q) zc[q * NT + t] = make_float2(0.f, 0.f);
        }
        bar_sync(1, NA);                                          // shares published, window read
        // the accelerations of this step, in the slot of the level they make
        float2 *ab = ACC ? a.aout + (long long)(n + 2 - a.out_k0) * a.lev + fo : nullptr;
        // ---- Newmark update of the owned nodes
        if (owns) {
            // the shares of the elements to the left, above and diagonal
            f[0] = add2(add2(f[0], zc[t - 1]), add2(zc[5 * NT + t - E], zc[4 * NT + t - E - 1]));
#pragma unroll
            for (int j = 1; j < 4; ++j) f[4 * j] = add2(f[4 * j], zc[j * NT + t - 1]);
#pragma unroll
            for (int i = 1; i < 4; ++i) f[i] = add2(f[i], zc[(5 + i) * NT + t - E]);
            if (ng > 0)
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const int k = q / 4 * 5 + q % 4;
                    if (imask >> k & 1) f[q] = add2(f[q], sinj[ibase + __popc(imask & ((1u << k) - 1))]);
                }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 m4 = smi[j * NT + t];
                const float mi[4] = {m4.x, m4.y, m4.z, m4.w};
                float4 ar[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 v = vr[2 * j + h], u = win[(2 * j + h) * PS + c0];
                    float4 ac, vn, un;
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int i = 2 * h + e;
                        const float2 v2 = e ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
                        const float2 u2 = e ? make_float2(u.z, u.w) : make_float2(u.x, u.y);
                        float2 a2;
                        int sl = -1;
                        if (i == 0 || j == 0) {                   // possible edge nodes
                            sl = i == 0 ? (j == 0 && eL < 0 ? eT : eL + j) : eT + i;
                            float4 bd = make_float4(0.f, 0.f, mi[i], mi[i]);
                            if (sl >= 0) bd = sedge[sl];
                            a2 = accel_edge(f[4 * j + i], v2, bd);
                        } else {
                            a2 = accel(f[4 * j + i], mi[i]);
                        }
                        const float2 n2 = axpy2(dt, a2, v2), w2 = axpy2(dt, n2, u2);
                        if (ADJ && (i == 0 || j == 0) && sl >= 0)
                            sev[sl] = make_float4(0.5f * (v2.x + n2.x), 0.5f * (v2.y + n2.y), a2.x, a2.y);
                        if (e) {
                            ac.z = a2.x; ac.w = a2.y; vn.z = n2.x; vn.w = n2.y; un.z = w2.x; un.w = w2.y;
                        } else {
                            ac.x = a2.x; ac.y = a2.y; vn.x = n2.x; vn.y = n2.y; un.x = w2.x; un.y = w2.y;
                        }
                    }
                    vr[2 * j + h] = vn;
                    nxt[(2 * j + h) * PS + c0] = un;
                    if (ADJ) sac[(2 * j + h) * NO + oi] = ac;
                    ar[h] = ac;
                }
                if (ACC) store_row(ab + g00 + j * pitch, ar[0], ar[1]);
            }
        }
        // ---- and of the extra lines, one node a thread
#pragma unroll 1
        for (int q = t; q < nextra; q += NT) {
            const int4 X = sxi[q];
            float2 k = zc[X.x];
            if (X.y >= 0) k = add2(k, zc[X.y]);
            if (X.w >> 16) k = add2(k, sinj[(X.w >> 16) - 1]);
            const int sl = X.w & 0xffff;
            const float2 v = svx[q], a2 = accel_edge(k, v, sedge[sl]);
            const float2 n2 = axpy2(dt, a2, v), un = axpy2(dt, n2, reinterpret_cast<float2 *>(win)[X.z]);
            if (ADJ) sev[sl] = make_float4(0.5f * (v.x + n2.x), 0.5f * (v.y + n2.y), a2.x, a2.y);
            svx[q] = n2;
            reinterpret_cast<float2 *>(nxt)[X.z] = un;
            if (ACC) ab[q < ncol ? (4 * ez0 + q) * pitch + a.nx - 1 : (a.nz - 1) * pitch + 4 * ex0 + q - ncol] = a2;
        }
        if (a.ntiles > 1) {
            // ---- the node lines the neighbours need
            bar_sync(2, NT);
            Word2 *xo = xch + (long long)(par ^ 1) * a.xslot;
            const unsigned tag = (unsigned)(n + 1 - a.n0);
#pragma unroll
            for (int h = 0; h < kMaxHalo; ++h)
                if (t + h * NT < nsend) {
                    const int2 at = slist[t + h * NT];
                    send_node(xo + at.x, reinterpret_cast<const float2 *>(nxt)[at.y], tag);
                }
        }
        // the correlation threads start after the sends: their traffic on the shared-memory
        // pipe would hold the words back
        if (ADJ) bar_arrive(3, NA);
    }
    if (a.n1 + 1 >= a.out_from) store_level(a.n1 + 1, ADJ ? win0 + (a.n1 & 1) * S::WIN : win0);
    // ---- state of the last step
    if (owns)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long g = g00 + j * pitch;
            *reinterpret_cast<float4 *>(vhb + g) = vr[2 * j];
            *reinterpret_cast<float4 *>(vhb + g + 2) = vr[2 * j + 1];
        }
#pragma unroll 1
    for (int q = t; q < nextra; q += NT)
        vhb[q < ncol ? (4 * ez0 + q) * pitch + a.nx - 1 : (a.nz - 1) * pitch + 4 * ex0 + q - ncol] = svx[q];
}

// node sums of the strain correlations from the elements' own sums, in the
// order [(ex, ez) + (ex-1, ez)] + [(ex, ez-1) + (ex-1, ez-1)]: acc components 0, 1
__global__ void assemble_strain_kernel(const float *__restrict__ eacc, int nex, int nez, int nx, int nz, int pitch,
                                       float *__restrict__ acc, long long acc_shot_stride, long long cs)
{
    const long long N = (long long)nx * nz;
    const float *e = eacc + (long long)blockIdx.y * nex * nez * 52;
    float *out = acc + (long long)blockIdx.y * acc_shot_stride;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < N; q += (long long)gridDim.x * blockDim.x) {
        const int iz = (int)(q / nx), ix = (int)(q - (long long)iz * nx);
        float2 row[2];
        for (int r = 0; r < 2; ++r) {                             // element rows iz / 4, then the one above
            const int ez = iz / 4 - r, j = iz - 4 * ez;
            float2 s = make_float2(0.f, 0.f);
            for (int c = 0; c < 2; ++c) {
                const int ex = ix / 4 - c, i = ix - 4 * ex;
                if (ez < 0 || ex < 0 || ez >= nez || ex >= nex || i > 4 || j > 4) continue;
                s = add2(s, *reinterpret_cast<const float2 *>(e + ((long long)ez * nex + ex) * 52 + 2 * (j * 5 + i)));
            }
            row[r] = s;
        }
        const float2 s = add2(row[0], row[1]);
        out[(long long)iz * pitch + ix] = s.x;
        out[cs + (long long)iz * pitch + ix] = s.y;
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// choice of the tile and launch
// ---------------------------------------------------------------------------

namespace {

using Kernel = void (*)(const ResidentArgs);

struct Variant { int NT, MODE, threads; Kernel fn; };

template <int NT, int MODE>
constexpr Variant variant()
{
    return {NT, MODE, Shape<NT, MODE>::THREADS, sem_resident_kernel<NT, MODE>};
}

const Variant kVariants[] = {variant<64, MODE_FWD>(),   variant<128, MODE_FWD>(),   variant<192, MODE_FWD>(),
                             variant<64, MODE_RCV>(),   variant<128, MODE_RCV>(),   variant<192, MODE_RCV>(),
                             variant<64, MODE_ADJ_G>(), variant<128, MODE_ADJ_G>(), variant<192, MODE_ADJ_G>()};

const Variant *find_variant(int NT, int mode)
{
    for (const Variant &v : kVariants)
        if (v.NT == NT && v.MODE == mode) return &v;
    return nullptr;
}

// the kernel that runs a mode (MODE_RCV's also stores the accelerations)
int kernel_mode(int mode) { return mode == MODE_FWD_PC ? MODE_RCV : mode; }

// resident CTAs of a variant on the current device (0: none)
int slots_of(const Variant &v, size_t smem, int *nsm)
{
    int dev = 0, occ = 0, coop = 0, most = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || !coop ||
        smem > (size_t)most - 64 || gb_allow_smem((const void *)v.fn) != GBFWI_OK ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, v.fn, v.threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return occ * *nsm;
}

}  // namespace

// Plan of the resident loop for `shots` shots in `mode` (best_tile).  null: the
// mesh does not fit (the step kernels of sem_step.cu run), or the lists of the tile
// could not be allocated this time (asked again by the next call).
const ResidentPlan *gb_resident_plan(gbfwi_mesh *m, int mode, int shots)
{
    if (mode == MODE_ADJ_PC) return nullptr;
    const auto known = m->plans.find({mode, shots});
    if (known != m->plans.end()) return known->second.NT ? &known->second : nullptr;
    const bool adj = kernel_mode(mode) == MODE_ADJ_G, fwd = mode == MODE_FWD || mode == MODE_FWD_PC;
    auto slots = [&](int NT, size_t smem, int &nsm) {
        const Variant *v = find_variant(NT, kernel_mode(mode));
        return v ? slots_of(*v, smem, &nsm) : 0;
    };
    // with the injection and record lists of the tile shape: shots that fit one launch
    auto with_lists = [&](const Tile &t) {
        const ListSizes &n = gb_list_sizes(m, t.TX, t.TZ);
        ResidentPlan p;
        p.NT = t.NT; p.TX = t.TX; p.TZ = t.TZ; p.ntx = t.ntx; p.ntz = t.ntz;
        p.grp_cap = fwd ? n.src_groups : n.rec_groups;
        p.ent_cap = fwd ? n.src_entries : n.rec_entries;
        p.rec_cap = fwd ? n.recorded : 0;
        p.smem = smem_bytes(t.NT, adj, t.TX, t.TZ, t.ntx, t.ntz, m->d.free_surface_top, p.grp_cap, p.ent_cap, p.rec_cap);
        int nsm = 0;
        p.per_launch = p.grp_cap < 32767 ? std::min(slots(t.NT, p.smem, nsm) / (t.ntx * t.ntz), 60000) : 0;
        return p;
    };
    const Tile best = best_tile(m->d.nex, m->d.nez, m->d.free_surface_top, adj, shots, slots,
                                [&](const Tile &t) { return with_lists(t).per_launch >= 1; });
    ResidentPlan p;
    if (best.NT) {
        TileLists &lists = m->plan_lists[{best.TX, best.TZ}];
        if (!lists.built && gb_build_lists(m, best.TX, best.TZ, true, lists) != GBFWI_OK) return nullptr;
        p = with_lists(best);
        p.lists = &lists;
    }
    const ResidentPlan &kept = m->plans[{mode, shots}] = p;
    return kept.NT ? &kept : nullptr;
}

int gb_launch_resident(const ResidentPlan &p, int mode, ResidentArgs a, int nshots, DevBuf &xch, cudaStream_t s)
{
    const Variant *v = find_variant(p.NT, kernel_mode(mode));
    if (!v || a.pitch % 4 != 0 || a.fstride % 4 != 0 || a.lev % 4 != 0 || a.acc_comp_stride % 4 != 0 ||
        a.acc_shot_stride % 4 != 0 || ((uintptr_t)a.aout & 31) || ((uintptr_t)a.u0 & 15) || ((uintptr_t)a.out & 31) || ((uintptr_t)a.vh & 15) ||
        ((uintptr_t)a.minv & 15) || ((uintptr_t)a.acc & 15) || ((uintptr_t)a.hist & 31) || ((uintptr_t)a.eacc & 15) || !a.status)
        return GBFWI_EINVAL;
    if (xch.bytes < gb_resident_exchange(p, nshots, a.fstride)) return GBFWI_EINVAL;
    a.TX = p.TX; a.TZ = p.TZ; a.ntx = p.ntx; a.ntz = p.ntz;
    a.ntiles = p.ntx * p.ntz;
    a.edge_cap = edge_cap(p.TX, p.TZ, p.ntx, p.ntz, a.free_top);
    a.grp_cap = p.grp_cap; a.ent_cap = p.ent_cap; a.rec_cap = p.rec_cap;
    const size_t smem = p.smem;
    GB_TRY(gb_allow_smem((const void *)v->fn));
    const ResidentArgs all = a;
    for (int s0 = 0; s0 < nshots; s0 += p.per_launch) {
        const int B = std::min(p.per_launch, nshots - s0);
        a = all;
        a.u0 += s0 * a.fstride;
        a.vh += s0 * a.fstride;
        a.out += s0 * a.fstride;
        if (a.aout) a.aout += s0 * a.fstride;
        if (a.hist) a.hist += s0 * a.fstride;
        if (a.acc) a.acc += s0 * a.acc_shot_stride;
        if (a.eacc) a.eacc += (long long)s0 * a.nex * a.nez * 52;
        if (a.seis) a.seis += s0 * a.seis_shot_stride;
        if (a.shot_map) a.shot_map += s0;
        else a.sig += s0 * a.sig_shot_stride;
        a.xstride = a.fstride;
        a.xslot = B * a.fstride;
        a.xch = xch.p;
        if (a.ntiles > 1) GB_CUDA(cudaMemsetAsync(xch.p, 0, 32 * (size_t)a.xslot, s));
        void *args[] = {&a};
        GB_CUDA(cudaLaunchCooperativeKernel((const void *)v->fn, dim3(a.ntiles, B), dim3(v->threads), args, smem, s));
        GB_LAUNCHED();
    }
    return GBFWI_OK;
}

int gb_assemble_strain(const gbfwi_mesh *m, const float *eacc, int B, float *acc, long long acc_shot_stride, long long cs,
                       cudaStream_t s)
{
    const long long N = (long long)m->nx * m->nz;
    assemble_strain_kernel<<<dim3((unsigned)std::min<long long>((N + 255) / 256, 2048), B), 256, 0, s>>>(
        eacc, m->d.nex, m->d.nez, m->nx, m->nz, m->pitch, acc, acc_shot_stride, cs);
    GB_LAUNCHED();
    return GBFWI_OK;
}

size_t gb_resident_exchange(const ResidentPlan &p, int nshots, long long NP)
{
    return exchange_bytes(p.ntx * p.ntz, nshots, p.per_launch, NP);
}
