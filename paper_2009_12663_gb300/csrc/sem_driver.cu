// Simulation driver of the gbfwi library: forward runs, misfit + adjoint
// gradient, and the diagonal preconditioners, as sequences of step launches
// (sem_step.cu) plus a few small kernels.
//
// Time indexing (records s_n = P u_n, n = 1..nt; sources F_n = f stf(t_n)):
//   forward launch n (n = 0..nt-1) reads u_{n+1}, vh_n, uses F_{n+1}, records
//   s_{n+1} and writes u_{n+2}, vh_{n+1};
//   adjoint launch j (j = 0..nt-1) is the same recurrence for w (w_0 = w_1 =
//   0) driven by F_{j+1} = P^T r_{nt-j} / dt; w_{j+1} is the Lagrange
//   multiplier lam_k with k = nt - j, which is correlated with u_k:
//     g = -dt^2 sum_k u_k^T [dM/dm a^w + dC/dm v^w + dK/dm w]
//   (the discrete gradient of Eqs. A16-A18 after summation by parts in time).
//
// Storage: fields are [slot][shot][nz][pitch] float2.  The forward history is
// either kept whole (nt + 2 slots) or as snapshots every C steps with the
// segment recomputed into C + 2 slots during the backward pass.

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <functional>
#include <string>
#include <vector>

#include "gbfwi_internal.h"
#include "size_rules.h"

namespace {

struct Ctx {
    gbfwi_mesh *m;
    TileLists *L;
    int tile;
    int B;                 // shots in this batch
    cudaStream_t s;
    const int *d_shots;    // [B] source ids
    long long NP;          // nz * pitch
    bool resident = false; // run each range of steps as one resident launch
};

// time levels of a field: level k at slot k - k0, or k % 3 of a ring
struct Levels {
    float2 *base = nullptr;
    long long lev = 0;         // B * NP
    int k0 = 0;
    bool ring = false;
    float2 *at(int k) const { return base + (long long)(ring ? k % 3 : k - k0) * lev; }
};

void base_args(StepArgs &a, const Ctx &c)
{
    std::memset(&a, 0, sizeof(a));
    gbfwi_mesh *m = c.m;
    a.nex = m->d.nex; a.nez = m->d.nez; a.nx = m->nx; a.nz = m->nz; a.pitch = m->pitch;
    a.dt = (float)m->d.dt;
    a.fstride = c.NP;
    a.hstride = c.NP;
    a.lm = m->d_lm.as<float2>();
    a.minv = m->d_minv.as<float>();
    a.bnd = m->d_bnd.as<float4>();
    a.bw = m->d_bw.as<float4>();
    a.wxs = m->d_wx.as<float>();
    a.wzs = m->d_wz.as<float>();
    a.ntiles = c.L->ntx * c.L->ntz;
    a.rec_tptr = c.L->rec_tptr.as<int>();
    a.rec_list = c.L->rec_list.as<int>();
    a.recw = m->d_recw.as<float>();
    a.rec_e = m->d_rec_e.as<int2>();
    a.nt = m->d.nt;
    a.seis_shot_stride = (long long)m->nrec * 2 * m->d.nt;
    a.status = m->w_status.as<int>();
}

// resident arguments shared by both directions
void resident_args(ResidentArgs &r, const StepArgs &a, const Ctx &c, int n0, int n1, const Levels &f, int out_from)
{
    std::memset(&r, 0, sizeof(r));
    r.nex = a.nex; r.nez = a.nez; r.nx = a.nx; r.nz = a.nz; r.pitch = a.pitch; r.nt = a.nt;
    r.dt = a.dt;
    r.n0 = n0; r.n1 = n1;
    r.fstride = c.NP;
    r.lev = f.lev;
    r.u0 = f.at(n0 + 1);
    r.vh = a.vh;
    r.out = f.base;
    r.out_from = out_from; r.out_ring = f.ring; r.out_k0 = f.k0;
    r.lm = a.lm; r.minv = a.minv; r.bnd = a.bnd; r.wxs = a.wxs; r.wzs = a.wzs;
    r.free_top = c.m->d.free_surface_top;
    r.per_shot_groups = a.per_shot_groups;
    r.sig = a.sig; r.sig_shot_stride = a.sig_shot_stride; r.sig_chan_stride = a.sig_chan_stride;
    r.sig_scale = a.sig_scale;
    r.shot_map = a.shot_map;
    r.recw = a.recw; r.rec_e = a.rec_e;
    r.seis = a.seis; r.seis_shot_stride = a.seis_shot_stride;
    r.acc = a.acc; r.acc_shot_stride = a.acc_shot_stride; r.acc_comp_stride = a.acc_comp_stride;
    r.status = a.status;
}

int run_resident(const Ctx &c, int mode, ResidentArgs &r)
{
    const ResidentPlan *p = gb_resident_plan(c.m, mode, c.B);
    if (!p) return GBFWI_EINVAL;
    const bool fwd = mode == MODE_FWD || mode == MODE_FWD_PC;
    r.gptr = (fwd ? p->lists->src_gptr : p->lists->rec_gptr).as<int>();
    r.groups = (fwd ? p->lists->src_groups : p->lists->rec_groups).as<InjGroup>();
    r.entries = (fwd ? p->lists->src_entries : p->lists->rec_entries).as<InjEntry>();
    r.rec_tptr = p->lists->rec_tptr.as<int>();
    r.rec_list = p->lists->rec_list.as<int>();
    return gb_launch_resident(*p, mode, r, c.B, c.m->w_xch, c.s);
}

constexpr int kNoLevel = INT_MAX;

// forward launches n in [n0, n1); `need`: first level that is read later
int fwd_range(const Ctx &c, int mode, int n0, int n1, const Levels &f, int need, float2 *vh, float *seis, float *acc,
              long long acc_shot_stride, long long acc_comp_stride, float2 *aout = nullptr)
{
    StepArgs a;
    base_args(a, c);
    a.vh = vh;
    a.gptr = c.L->src_gptr.as<int>();
    a.groups = c.L->src_groups.as<InjGroup>();
    a.entries = c.L->src_entries.as<InjEntry>();
    a.per_shot_groups = 1;
    a.sig = c.m->d_stf.as<float>();
    a.sig_shot_stride = c.m->d.nt + 1;
    a.sig_chan_stride = 0;
    a.sig_scale = 1.0f;
    a.shot_map = c.d_shots;
    a.seis = seis;
    a.acc = acc;
    a.acc_shot_stride = acc_shot_stride;
    a.acc_comp_stride = acc_comp_stride;
    if (c.resident) {
        ResidentArgs r;
        resident_args(r, a, c, n0, n1, f, need);
        r.aout = aout;
        return run_resident(c, mode, r);
    }
    for (int n = n0; n < n1; ++n) {
        a.ucur = f.at(n + 1);
        a.unext = f.at(n + 2);
        a.uold = f.at(n);
        a.tsig = n + 1;
        a.trec = n;
        GB_TRY(gb_launch_step(mode, c.tile, a, c.B, c.s));
    }
    return GBFWI_OK;
}

// adjoint launches j in [j0, j1); the adjoint field cycles through the ring w.
// MODE_RCV (resident): the field alone, all levels to w and their accelerations to aout
int adj_range(const Ctx &c, int mode, int j0, int j1, const Levels &w, float2 *wh, const Levels &hist,
              const float *sig, float *acc, long long acc_shot_stride, long long acc_comp_stride, float2 *aout = nullptr)
{
    const int nt = c.m->d.nt;
    StepArgs a;
    base_args(a, c);
    a.vh = wh;
    a.gptr = c.L->rec_gptr.as<int>();
    a.groups = c.L->rec_groups.as<InjGroup>();
    a.entries = c.L->rec_entries.as<InjEntry>();
    a.per_shot_groups = 0;
    a.sig = sig;
    a.sig_shot_stride = (long long)2 * c.m->nrec * nt;
    a.sig_chan_stride = nt;
    a.sig_scale = (float)(1.0 / c.m->d.dt);
    a.shot_map = nullptr;
    a.acc = acc;
    a.acc_shot_stride = acc_shot_stride;
    a.acc_comp_stride = acc_comp_stride;
    if (c.resident && mode == MODE_RCV) {
        ResidentArgs r;
        resident_args(r, a, c, j0, j1, w, 0);
        r.reverse = 1;
        r.aout = aout;
        return run_resident(c, mode, r);
    }
    if (c.resident && mode == MODE_ADJ_G) {
        ResidentArgs r;
        if (hist.lev != w.lev) return GBFWI_EINVAL;            // the kernel has one stride for both
        resident_args(r, a, c, j0, j1, w, j1 < nt ? j1 : kNoLevel);
        r.hist = hist.base;
        r.hist_k0 = hist.k0;
        r.eacc = c.m->w_eacc.as<float>();
        return run_resident(c, mode, r);
    }
    for (int j = j0; j < j1; ++j) {
        int k = nt - j;
        a.ucur = w.at(j + 1);
        a.unext = w.at(j + 2);
        a.uold = w.at(j);
        if (mode == MODE_ADJ_G) {
            a.h0 = hist.at(k);
        } else {
            a.h0 = hist.at(k + 1);
            a.h1 = hist.at(k);
            a.h2 = hist.at(k - 1);
        }
        a.tsig = nt - 1 - j;
        GB_TRY(gb_launch_step(mode, c.tile, a, c.B, c.s));
    }
    return GBFWI_OK;
}

}  // namespace

int gb_take_status(gbfwi_mesh *m)
{
    int st = 0;
    GB_CUDA(cudaMemcpy(&st, m->w_status.p, sizeof(int), cudaMemcpyDeviceToHost));
    if (st) {
        GB_CUDA(cudaMemset(m->w_status.p, 0, sizeof(int)));
        return GBFWI_ETIMEOUT;
    }
    return GBFWI_OK;
}

namespace {

// ------------------------------------------------------------------ kernels

// r = s - d in place, per-shot partial sums of r^2: grid (kMisfitBlocks, B)
constexpr int kMisfitBlocks = 64;

__global__ void residual_kernel(float *__restrict__ syn, const float *__restrict__ obs, long long per_shot,
                                double *__restrict__ partial, int *__restrict__ flag)
{
    const int shot = blockIdx.y;
    float *s = syn + (long long)shot * per_shot;
    const float *d = obs + (long long)shot * per_shot;
    double acc = 0.0;
    int bad = 0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < per_shot;
         q += (long long)gridDim.x * blockDim.x) {
        float r = s[q] - d[q];
        if (!isfinite(r)) bad = 1;
        s[q] = r;
        acc += (double)r * (double)r;
    }
    __shared__ double red[256];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[shot * kMisfitBlocks + blockIdx.x] = red[0];
    if (bad) atomicOr(flag, 1);
}

// total += 1/2 dt sum_b partial[s][b], shot by shot in order, so the result
// does not depend on how the shots were batched
__global__ void misfit_finish(const double *__restrict__ partial, int nshot, double half_dt,
                              double *__restrict__ total)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double t = *total;
        for (int sh = 0; sh < nshot; ++sh) {
            double s = 0.0;
            for (int b = 0; b < kMisfitBlocks; ++b) s += partial[sh * kMisfitBlocks + b];
            t += half_dt * s;
        }
        *total = t;
    }
}

__global__ void finite_check(const float *__restrict__ x, long long n, int *__restrict__ flag)
{
    int bad = 0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n;
         q += (long long)gridDim.x * blockDim.x)
        if (!isfinite(x[q])) bad = 1;
    if (bad) atomicOr(flag, 1);
}

// total[c][g] += sum_b acc[b][c][g]  (fixed order over b)
__global__ void acc_reduce(const float *__restrict__ acc, int B, int ncomp, long long NP,
                           float *__restrict__ total)
{
    long long n = (long long)ncomp * NP;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n;
         q += (long long)gridDim.x * blockDim.x) {
        float s = total[q];
        for (int b = 0; b < B; ++b) s += acc[(long long)b * n + q];
        total[q] = s;
    }
}

// gradient chain rule: (g_lambda, g_mu, sum u.a^w, g_Zp, g_Zs) -> (rho, vp, vs), times -dt^2;
// dM_g/drho_g = W_g = wx[ix] wz[iz]
__global__ void chain_kernel(const float *__restrict__ tot, const float *__restrict__ model,
                             const float *__restrict__ wx, const float *__restrict__ wz, int nx, int nz,
                             int pitch, float mdt2, float *__restrict__ grad)
{
    long long NP = (long long)nz * pitch, N = (long long)nz * nx;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < N;
         q += (long long)gridDim.x * blockDim.x) {
        int iz = (int)(q / nx), ix = (int)(q - (long long)iz * nx);
        long long g = (long long)iz * pitch + ix;
        const double w1[4] = {0.1, 49.0 / 90.0, 32.0 / 45.0, 49.0 / 90.0};
        const float ww = (float)(w1[ix & 3] * w1[iz & 3]);    // quadrature weight of the strain correlations
        float gl = ww * tot[g], gm = ww * tot[NP + g], gp = tot[3 * NP + g], gs = tot[4 * NP + g];
        float gM = wx[ix] * wz[iz] * tot[2 * NP + g];
        float r = model[g], p = model[NP + g], s = model[2 * NP + g];
        float grho = gl * (p * p - 2.f * s * s) + gm * s * s + gM + gp * p + gs * s;
        float gvp = gl * (2.f * r * p) + gp * r;
        float gvs = gl * (-4.f * r * s) + gm * (2.f * r * s) + gs * r;
        grad[q] = mdt2 * grho;
        grad[N + q] = mdt2 * gvp;
        grad[2 * N + q] = mdt2 * gvs;
    }
}

// Preconditioner maps from the time integrals (Eqs. 5-8, A21-A22):
//   H_rho = W |f0 S0|, H_a = 8 rho^2 vp^2 |f1 S1|,
//   H_b = 16 rho^2 vs^2 |f1 S2| + 4 rho^2 vs^2 |f1 S3|
// kind 1/2 replicate H_rho.  Output [3][nz][nx].
__global__ void precond_finish(const float *__restrict__ tot, const float *__restrict__ model,
                               const float *__restrict__ wx, const float *__restrict__ wz, int nx, int nz,
                               int pitch, int kind, float f0, float f1, float *__restrict__ H)
{
    long long NP = (long long)nz * pitch, N = (long long)nz * nx;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < N;
         q += (long long)gridDim.x * blockDim.x) {
        int iz = (int)(q / nx), ix = (int)(q - (long long)iz * nx);
        long long g = (long long)iz * pitch + ix;
        float hr = wx[ix] * wz[iz] * fabsf(f0 * tot[g]);
        float ha = hr, hb = hr;
        if (kind >= 3) {
            float r = model[g], p = model[NP + g], s = model[2 * NP + g];
            float r2 = r * r;
            ha = 8.f * r2 * p * p * fabsf(f1 * tot[NP + g]);
            hb = 16.f * r2 * s * s * fabsf(f1 * tot[2 * NP + g]) + 4.f * r2 * s * s * fabsf(f1 * tot[3 * NP + g]);
        }
        H[q] = hr;
        H[N + q] = ha;
        H[2 * N + q] = hb;
    }
}

// Separable Gaussian smoothing along one axis of [3][nz][nx]:
// out(i) = sum_j G(c_i - c_j) w_j f(j) / sum_j G(c_i - c_j) w_j over |c_i - c_j| <= 5 sigma
// A weight serves every node that shares it: along x a thread keeps one ix and
// takes kSmoothRows rows of the three maps; along z a block keeps one iz, forms
// its weights once in shared memory (chunks of kSmoothTaps) and spreads over ix.
// Bound by the exponentials before (one per node, map and tap: 68 and 88 us along
// x and z at 1361 x 281 nodes, 80 taps), by the loads of f from L1 now (38 and 31 us).
constexpr int kSmoothRows = 4, kSmoothTaps = 256;

__global__ void __launch_bounds__(128) smooth_x_kernel(const float *__restrict__ in, float *__restrict__ out, int nx, int nz,
                                                       const float *__restrict__ coord, const float *__restrict__ wts,
                                                       const int2 *__restrict__ range, float inv2s2, int row0)
{
    const int ix = blockIdx.x * blockDim.x + threadIdx.x, iz0 = row0 + blockIdx.y * kSmoothRows;
    if (ix >= nx) return;
    const long long N = (long long)nx * nz;
    const int rows = min(kSmoothRows, nz - iz0);
    const int2 rg = range[ix];
    const float ci = coord[ix];
    float num[3][kSmoothRows], den = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int r = 0; r < kSmoothRows; ++r) num[c][r] = 0.f;
    const float *base = in + (long long)iz0 * nx;
    for (int jj = rg.x; jj <= rg.y; ++jj) {
        const float d = ci - coord[jj];
        const float gw = __expf(-d * d * inv2s2) * wts[jj];
        den += gw;
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int r = 0; r < kSmoothRows; ++r)
                if (r < rows) num[c][r] = fmaf(gw, base[c * N + (long long)r * nx + jj], num[c][r]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int r = 0; r < kSmoothRows; ++r)
            if (r < rows) out[c * N + (long long)(iz0 + r) * nx + ix] = num[c][r] / den;
}

__global__ void __launch_bounds__(128) smooth_z_kernel(const float *__restrict__ in, float *__restrict__ out, int nx, int nz,
                                                       const float *__restrict__ coord, const float *__restrict__ wts,
                                                       const int2 *__restrict__ range, float inv2s2)
{
    __shared__ float sg[kSmoothTaps];
    const int ix = blockIdx.x * blockDim.x + threadIdx.x;
    const long long N = (long long)nx * nz;
    for (int iz = blockIdx.y; iz < nz; iz += gridDim.y) {
        const int2 rg = range[iz];
        const float ci = coord[iz];
        float num[3] = {0.f, 0.f, 0.f}, den = 0.f;
        for (int j0 = rg.x; j0 <= rg.y; j0 += kSmoothTaps) {
            const int m = min(kSmoothTaps, rg.y - j0 + 1);
            __syncthreads();
            for (int q = threadIdx.x; q < m; q += blockDim.x) {
                const float d = ci - coord[j0 + q];
                sg[q] = __expf(-d * d * inv2s2) * wts[j0 + q];
            }
            __syncthreads();
            if (ix < nx)
                for (int q = 0; q < m; ++q) {
                    const float gw = sg[q];
                    const float *f = in + (long long)(j0 + q) * nx + ix;
                    den += gw;
#pragma unroll
                    for (int c = 0; c < 3; ++c) num[c] = fmaf(gw, f[c * N], num[c]);
                }
        }
        if (ix < nx)
#pragma unroll
            for (int c = 0; c < 3; ++c) out[c * N + (long long)iz * nx + ix] = num[c] / den;
    }
}

// radix select of rank k over n floats, 8 bits per pass, the three maps at once
// (map blockIdx.y / blockIdx.x); state [3][4] = {prefix, mask, rank, -}
__device__ __forceinline__ unsigned fkey(float f)
{
    unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__global__ void radix_hist(const float *__restrict__ x, long long n, const unsigned *__restrict__ state,
                           int shift, unsigned *__restrict__ hist)
{
    __shared__ unsigned h[256];
    for (int t = threadIdx.x; t < 256; t += blockDim.x) h[t] = 0;
    __syncthreads();
    x += blockIdx.y * n;
    state += blockIdx.y * 4;
    hist += blockIdx.y * 256;
    unsigned prefix = state[0], mask = state[1];
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n;
         q += (long long)gridDim.x * blockDim.x) {
        unsigned k = fkey(x[q]);
        if ((k & mask) == prefix) atomicAdd(&h[(k >> shift) & 0xFFu], 1u);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 256; t += blockDim.x)
        if (h[t]) atomicAdd(&hist[t], h[t]);
}

// the bin holding the rank, by a prefix sum over the 256 bins (one thread each:
// a single thread's walk over them took 10 to 15 us a map and pass, the three
// maps together 3 us here)
__global__ void __launch_bounds__(256) radix_pick(unsigned *__restrict__ state, unsigned *__restrict__ hist, int shift,
                                                  float *__restrict__ result)
{
    __shared__ unsigned wsum[8];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    state += blockIdx.x * 4;
    hist += blockIdx.x * 256;
    const unsigned rank = state[2], prefix = state[0], h = hist[t];
    unsigned inc = h;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    for (int q = 0; q < w; ++q) inc += wsum[q];
    hist[t] = 0;
    if (inc > rank && inc - h <= rank) {
        const unsigned p = prefix | (unsigned)t << shift;
        state[0] = p;
        state[1] |= 0xFFu << shift;
        state[2] = rank - (inc - h);
        if (shift == 0) result[blockIdx.x] = __uint_as_float((p & 0x80000000u) ? (p & 0x7FFFFFFFu) : ~p);
    }
}

__global__ void radix_init(unsigned *__restrict__ state, unsigned *__restrict__ hist, unsigned rank)
{
    for (int t = threadIdx.x; t < 768; t += blockDim.x) hist[t] = 0;
    if (threadIdx.x < 12) state[threadIdx.x] = threadIdx.x % 4 == 2 ? rank : 0u;
}

__global__ void b0_kernel(const float *__restrict__ S, const float *__restrict__ med, long long N, float damp,
                          float *__restrict__ B0)
{
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < 3 * N;
         q += (long long)gridDim.x * blockDim.x) {
        int c = (int)(q / N);
        B0[q] = 1.f / (S[q] + damp * med[c]);
    }
}

// ------------------------------------------------------------------ helpers

int grid_for(long long n) { return (int)std::min<long long>(std::max<long long>((n + 255) / 256, 1), 152 * 8); }

struct Staged {
    const void *dptr = nullptr;
};

int stage_in(DevBuf &buf, const void *user, size_t bytes, cudaStream_t s, const void **dptr)
{
    if (gb_is_device_ptr(user)) { *dptr = user; return GBFWI_OK; }
    GB_TRY(buf.ensure(bytes));
    GB_CUDA(cudaMemcpyAsync(buf.p, user, bytes, cudaMemcpyHostToDevice, s));
    *dptr = buf.p;
    return GBFWI_OK;
}

int check_shots(const gbfwi_mesh *m, const int *shot_ids, int nshot)
{
    if (nshot < 1 || !shot_ids) return GBFWI_EINVAL;
    for (int i = 0; i < nshot; ++i)
        if (shot_ids[i] < 0 || shot_ids[i] >= (int)m->src.size()) return GBFWI_EINVAL;
    return GBFWI_OK;
}

// Shots taken `most` at a time, and whether batches of that size and the last one
// run as resident loops.  The last batch has plans of its own: it may take more shots in one
// launch than the others (the exchange buffer is sized for both), or none at all
// where its tile does not hold the receivers' lists (the step kernels serve it).
struct Batches {
    int most = 0, last = 0;
    bool resident_most = false, resident_last = false;
    bool resident(int B) const { return B == most ? resident_most : resident_last; }
};

// ... for passes in all of `modes`; reserves the exchange (before any work is queued)
int plan_batches(gbfwi_mesh *m, std::initializer_list<int> modes, int nshot, int most, long long NP, Batches &b)
{
    b = Batches{most, sizes::last_batch(nshot, most)};
    auto resident = [&](int B) {
        return std::all_of(modes.begin(), modes.end(), [&](int mode) { return gb_resident_plan(m, mode, B) != nullptr; });
    };
    b.resident_most = resident(most);
    b.resident_last = b.resident_most && resident(b.last);
    for (int B : {most, b.last})
        if (b.resident(B))
            for (int mode : modes) GB_TRY(m->w_xch.ensure(gb_resident_exchange(*gb_resident_plan(m, mode, B), B, NP)));
    return GBFWI_OK;
}

// Most shots a call takes together beyond what its schedule asks for in one launch
// (blockIdx.y counts the shots of a batch)
constexpr long long kMostShots = 65535;

// Shots of a batch where the resident loop takes it, and where it does not (`resident`
// false: it is not asked).  A call prefers more shots at once than its schedule asks for;
// where their buffers do not fit the memory that is left, it goes back to the schedule's
// number, and to the step kernels.
struct Choice { int most, stepped; bool resident; };

// gives back the buffers that grow with a batch (a cudaFree waits for work that uses them)
void release_batch_buffers(gbfwi_mesh *m)
{
    for (DevBuf *b : {&m->w_hist, &m->w_snap, &m->w_vh, &m->w_adj, &m->w_wh, &m->w_seis, &m->w_lacc, &m->w_pc, &m->w_eacc, &m->w_xch})
        b->release();
    for (gbfwi_mesh::Lane *l : m->lanes)
        for (DevBuf *b : {&l->hist, &l->snap, &l->vh, &l->adj, &l->wh, &l->seis, &l->acc}) b->release();
}

// reserve(batches) for the first of the choices whose buffers fit; passes in `modes` are those
// the resident loop would run
template <class Reserve>
int reserve_batches(gbfwi_mesh *m, std::initializer_list<int> modes, int nshot, const std::vector<Choice> &choices, Batches &b,
                    Reserve reserve)
{
    const long long NP = (long long)m->nz * m->pitch;
    return sizes::first_that_fits(choices, GBFWI_ENOMEM, [&](const Choice &c) -> int {
        b = Batches();
        if (c.resident && modes.size()) GB_TRY(plan_batches(m, modes, nshot, c.most, NP, b));
        if (!b.resident_most) b = Batches{c.stepped, sizes::last_batch(nshot, c.stepped)};
        return reserve(b);
    }, [&] { release_batch_buffers(m); });
}

// Forward runs that keep no history: the resident loop takes as many shots as fit
// the SMs at once (three levels and a velocity each), the step kernels the
// schedule's.  seis_shot: values of a shot's records that the mesh keeps (0: the caller
// does); fixed(): the buffers that do not grow with the batch
template <class Fixed>
int reserve_forward(gbfwi_mesh *m, int nshot, size_t seis_shot, Batches &b, Fixed fixed)
{
    const ResidentPlan *p = gb_resident_plan(m, MODE_FWD, nshot);
    const long long NP = (long long)m->nz * m->pitch;
    const int scheduled = std::min(nshot, m->sch.shots_per_launch);
    const int preferred = p ? std::min(nshot, std::max(p->per_launch, scheduled)) : scheduled;
    const std::vector<Choice> choices = {{preferred, scheduled, p != nullptr}, {scheduled, scheduled, true}, {scheduled, scheduled, false}};
    return reserve_batches(m, {MODE_FWD}, nshot, choices, b, [&](const Batches &c) -> int {
        GB_TRY(fixed());
        GB_TRY(m->w_hist.ensure((size_t)3 * c.most * NP * sizeof(float2)));
        GB_TRY(m->w_vh.ensure((size_t)c.most * NP * sizeof(float2)));
        return seis_shot ? m->w_seis.ensure(seis_shot * c.most * sizeof(float)) : GBFWI_OK;
    });
}

}  // namespace

// ---------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------

extern "C" int gbfwi_forward(gbfwi_mesh *m, const int *shot_ids, int nshot, float *seis, void *stream)
{
    if (!m || !seis) return GBFWI_EINVAL;
    GB_TRY(gb_check_local(seis));
    GB_TRY(check_shots(m, shot_ids, nshot));
    if (!m->have_model) return GBFWI_ENOMODEL;
    cudaStream_t s = (cudaStream_t)stream;
    const int tile = m->sch.tile;
    GB_TRY(gb_build_tile_lists(m, tile));
    const int nt = m->d.nt;
    const long long NP = (long long)m->nz * m->pitch;
    const size_t seis_shot = (size_t)m->nrec * 2 * nt;
    const bool dev_out = gb_is_device_ptr(seis);
    Batches batches;
    GB_TRY(reserve_forward(m, nshot, dev_out ? 0 : seis_shot, batches,
                           [&] { return m->w_shots.ensure((size_t)nshot * sizeof(int)); }));
    const int Bmax = batches.most;
    GB_CUDA(cudaMemcpyAsync(m->w_shots.p, shot_ids, nshot * sizeof(int), cudaMemcpyHostToDevice, s));
    for (int i0 = 0; i0 < nshot; i0 += Bmax) {
        int B = std::min(Bmax, nshot - i0);
        Ctx c{m, &m->lists[tile], tile, B, s, m->w_shots.as<int>() + i0, NP, batches.resident(B)};
        const Levels ring{m->w_hist.as<float2>(), (long long)B * NP, 0, true};
        GB_CUDA(cudaMemsetAsync(ring.base, 0, 3 * ring.lev * sizeof(float2), s));
        GB_CUDA(cudaMemsetAsync(m->w_vh.p, 0, ring.lev * sizeof(float2), s));
        float *out = dev_out ? seis + seis_shot * i0 : m->w_seis.as<float>();
        GB_TRY(fwd_range(c, MODE_FWD, 0, nt, ring, kNoLevel, m->w_vh.as<float2>(), out, nullptr, 0, 0));
        if (!dev_out)
            GB_CUDA(cudaMemcpyAsync(seis + seis_shot * i0, out, seis_shot * B * sizeof(float),
                                    cudaMemcpyDeviceToHost, s));
    }
    if (!dev_out) {
        GB_CUDA(cudaStreamSynchronize(s));
        GB_TRY(gb_take_status(m));
    }
    return GBFWI_OK;
}

// ---------------------------------------------------------------------------
// misfit only
// ---------------------------------------------------------------------------

extern "C" int gbfwi_misfit(gbfwi_mesh *m, const int *shot_ids, int nshot, const float *d_obs, double *misfit,
                            void *stream)
{
    if (!m || !d_obs || !misfit) return GBFWI_EINVAL;
    GB_TRY(gb_check_local(d_obs, misfit));
    GB_TRY(check_shots(m, shot_ids, nshot));
    if (!m->have_model) return GBFWI_ENOMODEL;
    cudaStream_t s = (cudaStream_t)stream;
    const int tile = m->sch.tile;
    GB_TRY(gb_build_tile_lists(m, tile));
    const int nt = m->d.nt;
    const long long NP = (long long)m->nz * m->pitch;
    const size_t seis_shot = (size_t)m->nrec * 2 * nt;
    const int npart = kMisfitBlocks * nshot;
    Batches batches;
    GB_TRY(reserve_forward(m, nshot, seis_shot, batches, [&]() -> int {
        GB_TRY(m->w_shots.ensure((size_t)nshot * sizeof(int)));
        GB_TRY(m->w_red.ensure((size_t)(npart + 8) * sizeof(double) + 4096));
        GB_TRY(m->w_flag.ensure(16));
        return gb_is_device_ptr(d_obs) ? GBFWI_OK : m->w_obs.ensure(seis_shot * nshot * sizeof(float));
    }));
    const int Bmax = batches.most;
    const void *obs_d = nullptr;
    GB_TRY(stage_in(m->w_obs, d_obs, seis_shot * nshot * sizeof(float), s, &obs_d));
    double *partial = m->w_red.as<double>();
    double *mis_d = partial + npart;
    int *flag = m->w_flag.as<int>();
    GB_CUDA(cudaMemcpyAsync(m->w_shots.p, shot_ids, nshot * sizeof(int), cudaMemcpyHostToDevice, s));
    GB_CUDA(cudaMemsetAsync(mis_d, 0, sizeof(double), s));
    GB_CUDA(cudaMemsetAsync(flag, 0, 16, s));
    for (int i0 = 0; i0 < nshot; i0 += Bmax) {
        int B = std::min(Bmax, nshot - i0);
        Ctx c{m, &m->lists[tile], tile, B, s, m->w_shots.as<int>() + i0, NP, batches.resident(B)};
        const Levels ring{m->w_hist.as<float2>(), (long long)B * NP, 0, true};
        GB_CUDA(cudaMemsetAsync(ring.base, 0, 3 * ring.lev * sizeof(float2), s));
        GB_CUDA(cudaMemsetAsync(m->w_vh.p, 0, ring.lev * sizeof(float2), s));
        float *seis_d = m->w_seis.as<float>();
        GB_TRY(fwd_range(c, MODE_FWD, 0, nt, ring, kNoLevel, m->w_vh.as<float2>(), seis_d, nullptr, 0, 0));
        residual_kernel<<<dim3(kMisfitBlocks, B), 256, 0, s>>>(seis_d, (const float *)obs_d + seis_shot * i0,
                                                              (long long)seis_shot, partial, flag);
        GB_LAUNCHED();
        misfit_finish<<<1, 32, 0, s>>>(partial, B, 0.5 * m->d.dt, mis_d);
        GB_LAUNCHED();
    }
    double mis_h = 0;
    int flag_h = 0;
    GB_CUDA(cudaMemcpyAsync(&mis_h, mis_d, sizeof(double), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaMemcpyAsync(&flag_h, flag, sizeof(int), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    GB_TRY(gb_take_status(m));
    if (flag_h || !std::isfinite(mis_h)) return gb_nonfinite("misfit");
    *misfit = mis_h;
    return GBFWI_OK;
}

// ---------------------------------------------------------------------------
// forward pass with history (full) or snapshots (checkpointed) for one batch
// ---------------------------------------------------------------------------

namespace {

// buffers for the largest batch; a batch of B shots lays its levels out B * NP apart
struct BatchHist {
    float2 *full = nullptr;    // ckpt == 0: nt + 2 levels
    float2 *ring = nullptr;    // ckpt > 0: 3-slot ring for the forward pass
    float2 *seg = nullptr;     // ckpt > 0: C + 2 slots
    float2 *snap = nullptr;    // ckpt > 0: [nseg][3][B][NP]: u_{sC}, u_{sC+1}, vh_{sC}
    float2 *vh_rec = nullptr;  // recompute velocity
    float2 *vh = nullptr;      // forward half-step velocity
    float2 *wring = nullptr;   // adjoint field, 3 levels
    float2 *wh = nullptr;      // adjoint half-step velocity
    int C = 0, nseg = 0;
};

// Bytes of forward levels a gradient may keep beyond what its schedule asks
// for, to run more shots at once on meshes too small to fill the GPU.
constexpr long long kSmallHistory = 1LL << 30;

// Bytes of levels the preconditioner maps may keep to form their integrals from
// (sem_integrals.cu).
constexpr long long kMapHistory = 6LL << 30;

// the work buffers of one concurrent lane
struct LaneRef {
    DevBuf *hist, *snap, *vh, *adj, *wh, *seis, *batch, *acc;
    cudaStream_t st;
};

LaneRef lane0(gbfwi_mesh *m, cudaStream_t s)
{
    return LaneRef{&m->w_hist, &m->w_snap, &m->w_vh, &m->w_adj, &m->w_wh, &m->w_seis, &m->w_batch, &m->w_lacc, s};
}

int alloc_hist(gbfwi_mesh *m, const LaneRef &L, int B, int ckpt, long long NP, BatchHist &h, bool adjoint)
{
    const int nt = m->d.nt;
    long long lev = (long long)B * NP;
    if (ckpt <= 0 || ckpt >= nt) {
        GB_TRY(L.hist->ensure((size_t)(nt + 2) * lev * sizeof(float2)));
        h.full = L.hist->as<float2>();
        h.C = 0;
    } else {
        h.C = ckpt;
        h.nseg = (nt + ckpt - 1) / ckpt;
        size_t ring = 3, seg = (size_t)ckpt + 2, snap = (size_t)h.nseg * 3, vrec = 1;
        GB_TRY(L.hist->ensure((ring + seg + vrec) * lev * sizeof(float2)));
        GB_TRY(L.snap->ensure(snap * lev * sizeof(float2)));
        h.ring = L.hist->as<float2>();
        h.seg = h.ring + ring * lev;
        h.vh_rec = h.seg + seg * lev;
        h.snap = L.snap->as<float2>();
    }
    GB_TRY(L.vh->ensure(lev * sizeof(float2)));
    h.vh = L.vh->as<float2>();
    if (adjoint) {
        GB_TRY(L.adj->ensure(3 * lev * sizeof(float2)));
        GB_TRY(L.wh->ensure(lev * sizeof(float2)));
        h.wring = L.adj->as<float2>();
        h.wh = L.wh->as<float2>();
    }
    return GBFWI_OK;
}

// forward over all launches, recording into seis (device, [B][nrec][2][nt])
int forward_pass(const Ctx &c, BatchHist &h, float *seis)
{
    gbfwi_mesh *m = c.m;
    const int nt = m->d.nt;
    const long long lev = (long long)c.B * c.NP;
    float2 *vh = h.vh;
    GB_CUDA(cudaMemsetAsync(vh, 0, lev * sizeof(float2), c.s));
    if (h.C == 0) {
        GB_CUDA(cudaMemsetAsync(h.full, 0, 2 * lev * sizeof(float2), c.s));
        return fwd_range(c, MODE_FWD, 0, nt, Levels{h.full, lev, 0, false}, 0, vh, seis, nullptr, 0, 0);
    }
    GB_CUDA(cudaMemsetAsync(h.ring, 0, 3 * lev * sizeof(float2), c.s));
    const Levels ring{h.ring, lev, 0, true};
    for (int sg = 0; sg < h.nseg; ++sg) {
        int n0 = sg * h.C, n1 = std::min(nt, n0 + h.C);
        float2 *sp = h.snap + (long long)sg * 3 * lev;
        GB_CUDA(cudaMemcpyAsync(sp, ring.at(n0), lev * sizeof(float2), cudaMemcpyDeviceToDevice, c.s));
        GB_CUDA(cudaMemcpyAsync(sp + lev, ring.at(n0 + 1), lev * sizeof(float2), cudaMemcpyDeviceToDevice, c.s));
        GB_CUDA(cudaMemcpyAsync(sp + 2 * lev, vh, lev * sizeof(float2), cudaMemcpyDeviceToDevice, c.s));
        GB_TRY(fwd_range(c, MODE_FWD, n0, n1, ring, n1 < nt ? n1 : kNoLevel, vh, seis, nullptr, 0, 0));
    }
    return GBFWI_OK;
}

// adjoint over all launches; segments recomputed when checkpointed
int adjoint_pass(const Ctx &c, BatchHist &h, int mode, const float *sig, float *acc, long long acc_shot_stride,
                 long long acc_comp_stride)
{
    gbfwi_mesh *m = c.m;
    const int nt = m->d.nt;
    const long long lev = (long long)c.B * c.NP;
    const Levels wring{h.wring, lev, 0, true};
    float2 *wh = h.wh;
    GB_CUDA(cudaMemsetAsync(h.wring, 0, 3 * lev * sizeof(float2), c.s));
    GB_CUDA(cudaMemsetAsync(wh, 0, lev * sizeof(float2), c.s));
    if (h.C == 0) {
        return adj_range(c, mode, 0, nt, wring, wh, Levels{h.full, lev, 0, false}, sig, acc, acc_shot_stride, acc_comp_stride);
    }
    for (int sg = h.nseg - 1; sg >= 0; --sg) {
        int n0 = sg * h.C, n1 = std::min(nt, n0 + h.C);
        float2 *sp = h.snap + (long long)sg * 3 * lev;
        const Levels seg{h.seg, lev, n0, false};
        GB_CUDA(cudaMemcpyAsync(seg.at(n0), sp, lev * sizeof(float2), cudaMemcpyDeviceToDevice, c.s));
        GB_CUDA(cudaMemcpyAsync(seg.at(n0 + 1), sp + lev, lev * sizeof(float2), cudaMemcpyDeviceToDevice, c.s));
        GB_CUDA(cudaMemcpyAsync(h.vh_rec, sp + 2 * lev, lev * sizeof(float2), cudaMemcpyDeviceToDevice, c.s));
        GB_TRY(fwd_range(c, MODE_FWD, n0, n1, seg, 0, h.vh_rec, nullptr, nullptr, 0, 0));
        // adjoint launches whose correlation level k lies in [n0 + 1, n1]
        int j0 = nt - n1, j1 = nt - n0;
        GB_TRY(adj_range(c, mode, j0, j1, wring, wh, seg, sig, acc, acc_shot_stride, acc_comp_stride));
    }
    return GBFWI_OK;
}

// Run body() on the caller's stream s, or, with graphs enabled, replay a CUDA
// graph of it captured once on a private stream (the caller's stream may be
// the legacy default stream, which cannot be captured).
int run_pass(gbfwi_mesh *m, bool replay, const std::string &key, cudaStream_t s, const std::function<int(cudaStream_t)> &body)
{
    if (!replay || !m->sch.use_graph) return body(s);
    for (auto &g : m->graphs)
        if (g.key == key) {
            GB_CUDA(cudaGraphLaunch(g.exec, s));
            gb_note_launches(g.kernels);
            return GBFWI_OK;
        }
    if (!m->cap_stream) GB_CUDA(cudaStreamCreateWithFlags(&m->cap_stream, cudaStreamNonBlocking));
    // the capture stream must not run ahead of work already queued on s
    cudaEvent_t ready;
    GB_CUDA(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
    GB_CUDA(cudaEventRecord(ready, s));
    GB_CUDA(cudaStreamWaitEvent(m->cap_stream, ready, 0));
    GB_CUDA(cudaEventDestroy(ready));
    GB_CUDA(cudaStreamSynchronize(m->cap_stream));
    const long long before = gb_launches_so_far();
    GB_CUDA(cudaStreamBeginCapture(m->cap_stream, cudaStreamCaptureModeThreadLocal));
    int rc = body(m->cap_stream);
    cudaGraph_t graph = nullptr;
    cudaError_t ce = cudaStreamEndCapture(m->cap_stream, &graph);
    // launches recorded during capture did not run: count them at replay
    const long long kernels = gb_launches_so_far() - before;
    gb_note_launches(-kernels);
    if (rc != GBFWI_OK || ce != cudaSuccess) {
        if (graph) cudaGraphDestroy(graph);
        if (rc == GBFWI_OK) {
            gb_set_last_cuda_error(ce, "cudaStreamEndCapture", __FILE__, __LINE__);
            rc = GBFWI_ECUDA;
        }
        return rc;
    }
    cudaGraphExec_t exec = nullptr;
    ce = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (ce != cudaSuccess) {
        gb_set_last_cuda_error(ce, "cudaGraphInstantiate", __FILE__, __LINE__);
        return GBFWI_ECUDA;
    }
    if (m->graphs.size() >= 16) {          // bounded cache
        cudaGraphExecDestroy(m->graphs.front().exec);
        m->graphs.erase(m->graphs.begin());
    }
    m->graphs.push_back({key, exec, kernels});
    GB_CUDA(cudaGraphLaunch(exec, s));
    gb_note_launches(kernels);
    return GBFWI_OK;
}

std::string pass_key(const char *what, const gbfwi_mesh *m, int B, int ckpt, std::initializer_list<const void *> ptrs)
{
    std::string k = what;
    k += "|" + std::to_string(m->sch.tile) + "|" + std::to_string(B) + "|" + std::to_string(ckpt);
    for (const void *p : ptrs) k += "|" + std::to_string((uintptr_t)p);
    return k;
}

}  // namespace

// ---------------------------------------------------------------------------
// misfit + gradient
// ---------------------------------------------------------------------------

extern "C" int gbfwi_adjoint_gradient(gbfwi_mesh *m, const int *shot_ids, int nshot, const float *d_obs,
                                      double *misfit, float *grad, int ckpt_every, void *stream)
{
    if (!m || !d_obs || !misfit || !grad) return GBFWI_EINVAL;
    GB_TRY(gb_check_local(d_obs, misfit, grad));
    GB_TRY(check_shots(m, shot_ids, nshot));
    if (!m->have_model) return GBFWI_ENOMODEL;
    cudaStream_t s = (cudaStream_t)stream;
    const int tile = m->sch.tile;
    GB_TRY(gb_build_tile_lists(m, tile));
    const int nt = m->d.nt;
    const int ckpt = ckpt_every >= 0 ? ckpt_every : m->sch.ckpt_every;
    const long long NP = (long long)m->nz * m->pitch;
    const long long N = (long long)m->nz * m->nx;
    const size_t seis_shot = (size_t)m->nrec * 2 * nt;
    // Resident loops: one lane whose batch holds the shots the schedule keeps in
    // flight (shots per launch x streams), or more while their histories stay small
    const bool full = ckpt <= 0 || ckpt >= nt;
    const long long levels = full ? nt + 2 : 3LL * ((nt + ckpt - 1) / ckpt) + ckpt + 6;
    const long long small = kSmallHistory / (levels * NP * (long long)sizeof(float2));
    const int stepped = std::min(m->sch.shots_per_launch, nshot);
    const int scheduled = (int)std::min<long long>({nshot, (long long)m->sch.shots_per_launch * m->sch.streams, kMostShots});
    const int preferred = (int)std::min<long long>({nshot, std::max<long long>(scheduled, small), kMostShots});
    const size_t eacc_shot = (size_t)m->d.nex * m->d.nez * 52 * sizeof(float);
    // per-shot accumulators and misfit partials, reduced once in shot order at
    // the end: the result does not depend on batching or lanes
    const int npart = kMisfitBlocks * nshot;
    const bool dev_grad = gb_is_device_ptr(grad);
    auto fixed_buffers = [&]() -> int {
        GB_TRY(m->w_acc.ensure((size_t)nshot * 5 * NP * sizeof(float)));
        GB_TRY(m->w_grad.ensure((size_t)5 * NP * sizeof(float)));
        GB_TRY(m->w_shots.ensure((size_t)nshot * sizeof(int)));
        GB_TRY(m->w_red.ensure((size_t)(npart + 8) * sizeof(double) + 4096));
        GB_TRY(m->w_flag.ensure(16));
        if (!dev_grad) GB_TRY(m->w_tmp.ensure((size_t)3 * N * sizeof(float)));
        return gb_is_device_ptr(d_obs) ? GBFWI_OK : m->w_obs.ensure(seis_shot * nshot * sizeof(float));
    };
    // lanes: 0 = the mesh's own buffers on the caller's stream, 1.. = extra streams
    int nbatch = 0, L = 0;
    std::vector<LaneRef> lanes;
    std::vector<BatchHist> hs;
    Batches batches;
    const std::vector<Choice> choices = {{preferred, stepped, true}, {scheduled, stepped, true}, {stepped, stepped, false}};
    GB_TRY(reserve_batches(m, {MODE_FWD, MODE_ADJ_G}, nshot, choices, batches, [&](const Batches &b) -> int {
        GB_TRY(fixed_buffers());
        nbatch = (nshot + b.most - 1) / b.most;
        L = b.resident_most ? 1 : std::max(1, std::min(m->sch.streams, nbatch));
        if (b.resident_most) GB_TRY(m->w_eacc.ensure(eacc_shot * b.most));
        while ((int)m->lanes.size() < L - 1) m->lanes.push_back(new gbfwi_mesh::Lane());
        lanes.assign(1, lane0(m, s));
        for (int l = 1; l < L; ++l) {
            gbfwi_mesh::Lane *ln = m->lanes[l - 1];
            if (!ln->st) GB_CUDA(cudaStreamCreateWithFlags(&ln->st, cudaStreamNonBlocking));
            lanes.push_back(
                LaneRef{&ln->hist, &ln->snap, &ln->vh, &ln->adj, &ln->wh, &ln->seis, &ln->batch, &ln->acc, ln->st});
        }
        hs.assign(L, BatchHist());
        for (int l = 0; l < L; ++l) {
            GB_TRY(alloc_hist(m, lanes[l], b.most, ckpt, NP, hs[l], true));
            GB_TRY(lanes[l].seis->ensure(seis_shot * b.most * sizeof(float)));
            GB_TRY(lanes[l].batch->ensure((size_t)b.most * sizeof(int)));
            GB_TRY(lanes[l].acc->ensure((size_t)b.most * 5 * NP * sizeof(float)));
        }
        return GBFWI_OK;
    }));
    const int Bmax = batches.most;
    const void *obs_d = nullptr;
    GB_TRY(stage_in(m->w_obs, d_obs, seis_shot * nshot * sizeof(float), s, &obs_d));
    float *grad_d = dev_grad ? grad : m->w_tmp.as<float>();
    double *partial = m->w_red.as<double>();
    double *mis_d = partial + npart;
    int *flag = m->w_flag.as<int>();
    float *acc_all = m->w_acc.as<float>();
    GB_CUDA(cudaMemcpyAsync(m->w_shots.p, shot_ids, nshot * sizeof(int), cudaMemcpyHostToDevice, s));
    GB_CUDA(cudaMemsetAsync(mis_d, 0, sizeof(double), s));
    GB_CUDA(cudaMemsetAsync(flag, 0, 16, s));
    float *tot = m->w_grad.as<float>();
    GB_CUDA(cudaMemsetAsync(tot, 0, 5 * NP * sizeof(float), s));
    m->timed_valid = false;
    if (m->timing) {
        while ((int)m->ev.size() < 4 * nbatch + 2 * L) {
            cudaEvent_t e;
            GB_CUDA(cudaEventCreate(&e));
            m->ev.push_back(e);
        }
        m->fwd_launches = m->adj_launches = 0;
    }
    GB_TRY(gb_prepare_step(MODE_FWD, tile));
    GB_TRY(gb_prepare_step(MODE_ADJ_G, tile));
    // fork the lanes off the caller's stream
    std::vector<cudaEvent_t> sync_ev(L);
    for (int l = 0; l < L; ++l) GB_CUDA(cudaEventCreateWithFlags(&sync_ev[l], cudaEventDisableTiming));
    GB_CUDA(cudaEventRecord(sync_ev[0], s));
    for (int l = 1; l < L; ++l) GB_CUDA(cudaStreamWaitEvent(lanes[l].st, sync_ev[0], 0));

    int rc = GBFWI_OK;
    for (int i0 = 0, bi = 0; i0 < nshot && rc == GBFWI_OK; i0 += Bmax, ++bi) {
        const int l = bi % L;
        const LaneRef &lr = lanes[l];
        BatchHist &h = hs[l];
        cudaStream_t ls = lr.st;
        const int B = std::min(Bmax, nshot - i0);
        const bool resident = batches.resident(B);
        auto step = [&]() -> int {
            auto mark = [&](int i) -> int {
                if (m->timing) GB_CUDA(cudaEventRecord(m->ev[i], ls));
                return GBFWI_OK;
            };
            // this batch's source ids at a fixed address, so captured passes replay for every batch
            GB_CUDA(cudaMemcpyAsync(lr.batch->p, m->w_shots.as<int>() + i0, B * sizeof(int),
                                    cudaMemcpyDeviceToDevice, ls));
            Ctx c{m, &m->lists[tile], tile, B, ls, lr.batch->as<int>(), NP, resident};
            float *seis_d = lr.seis->as<float>();
            float *acc = lr.acc->as<float>();
            const std::string kf = pass_key("fwd", m, B, h.C, {lr.hist->p, lr.vh->p, lr.seis->p, lr.snap->p,
                                                               lr.batch->p});
            const std::string ka = pass_key("adj", m, B, h.C, {lr.hist->p, lr.seis->p, lr.snap->p, lr.adj->p,
                                                               lr.wh->p, lr.acc->p});
            GB_TRY(mark(4 * bi));
            GB_TRY(run_pass(m, !resident, kf, ls, [&](cudaStream_t cs) {
                Ctx cc = c;
                cc.s = cs;
                return forward_pass(cc, h, seis_d);
            }));
            GB_TRY(mark(4 * bi + 1));
            // residual r = s - d (in place), per-shot partial sums of r^2
            residual_kernel<<<dim3(kMisfitBlocks, B), 256, 0, ls>>>(seis_d, (const float *)obs_d + seis_shot * i0,
                                                                   (long long)seis_shot,
                                                                   partial + (long long)kMisfitBlocks * i0, flag);
            GB_LAUNCHED();
            GB_TRY(mark(4 * bi + 2));
            GB_TRY(run_pass(m, !resident, ka, ls, [&](cudaStream_t cs) -> int {
                Ctx cc = c;
                cc.s = cs;
                GB_CUDA(cudaMemsetAsync(acc, 0, (size_t)B * 5 * NP * sizeof(float), cs));
                if (resident) GB_CUDA(cudaMemsetAsync(m->w_eacc.p, 0, eacc_shot * B, cs));
                GB_TRY(adjoint_pass(cc, h, MODE_ADJ_G, seis_d, acc, 5 * NP, NP));
                return resident ? gb_assemble_strain(m, m->w_eacc.as<float>(), B, acc, 5 * NP, NP, cs) : GBFWI_OK;
            }));
            GB_TRY(mark(4 * bi + 3));
            GB_CUDA(cudaMemcpyAsync(acc_all + (long long)i0 * 5 * NP, acc, (size_t)B * 5 * NP * sizeof(float),
                                    cudaMemcpyDeviceToDevice, ls));
            m->fwd_launches += nt;
            m->adj_launches += (h.C == 0) ? nt : 2LL * nt;
            return GBFWI_OK;
        };
        rc = step();
    }
    // join the lanes back into the caller's stream (also after an error)
    for (int l = 1; l < L; ++l) {
        cudaEventRecord(sync_ev[l], lanes[l].st);
        cudaStreamWaitEvent(s, sync_ev[l], 0);
    }
    for (int l = 0; l < L; ++l) cudaEventDestroy(sync_ev[l]);
    if (rc != GBFWI_OK) return rc;
    misfit_finish<<<1, 32, 0, s>>>(partial, nshot, 0.5 * m->d.dt, mis_d);
    GB_LAUNCHED();
    acc_reduce<<<grid_for(5 * NP), 256, 0, s>>>(acc_all, nshot, 5, NP, tot);
    GB_LAUNCHED();
    const float dt = (float)m->d.dt;
    chain_kernel<<<grid_for(N), 256, 0, s>>>(tot, m->d_model.as<float>(), m->d_wx.as<float>(), m->d_wz.as<float>(),
                                             m->nx, m->nz, m->pitch, -dt * dt, grad_d);
    GB_LAUNCHED();
    finite_check<<<grid_for(3 * N), 256, 0, s>>>(grad_d, 3 * N, flag);
    GB_LAUNCHED();
    double mis_h = 0;
    int flag_h = 0;
    GB_CUDA(cudaMemcpyAsync(&mis_h, mis_d, sizeof(double), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaMemcpyAsync(&flag_h, flag, sizeof(int), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    GB_TRY(gb_take_status(m));
    if (m->timing) {
        double fm = 0, am = 0;
        for (int bi = 0; bi < nbatch; ++bi) {
            float a = 0, b = 0;
            GB_CUDA(cudaEventElapsedTime(&a, m->ev[4 * bi], m->ev[4 * bi + 1]));
            GB_CUDA(cudaEventElapsedTime(&b, m->ev[4 * bi + 2], m->ev[4 * bi + 3]));
            fm += a;
            am += b;
        }
        m->fwd_ms = fm;
        m->adj_ms = am;
        m->timed_valid = true;
    }
    if (flag_h || !std::isfinite(mis_h)) return gb_nonfinite("misfit");
    if (!dev_grad) {
        GB_CUDA(cudaMemcpyAsync(grad, grad_d, 3 * N * sizeof(float), cudaMemcpyDeviceToHost, s));
        GB_CUDA(cudaStreamSynchronize(s));
    }
    *misfit = mis_h;
    return GBFWI_OK;
}

// ---------------------------------------------------------------------------
// preconditioners P1..P4, smoothing, damping, inversion
// ---------------------------------------------------------------------------

// B0 = 1 / (S(H) + damp * median(S(H))) per parameter from the raw map Hd
// [3][N] (device); S1, S2 scratch [3][N].  Writes B0 (device or host).
static int b0_from_map(gbfwi_mesh *m, const float *Hd, float *S1, float *S2, double sigma, double damp, float *B0,
                       cudaStream_t s)
{
    const long long N = (long long)m->nx * m->nz;
    // smoothing tables (node coordinates and weights along each axis, 5-sigma
    // index ranges), in one upload
    const int nx = m->nx, nz = m->nz;
    std::vector<int2> tab(2 * (size_t)(nx + nz));       // (coordinate, weight) as bits, then the ranges
    for (int ax = 0, o = 0; ax < 2; o += ax == 0 ? nx : 0, ++ax) {
        const int n = ax == 0 ? nx : nz;
        const std::vector<double> X = gb_axis(m, ax == 0 ? m->d.nex : m->d.nez);
        const std::vector<double> &w = ax == 0 ? m->wx1 : m->wz1;
        float *c = reinterpret_cast<float *>(tab.data()) + 2 * o;
        for (int i = 0; i < n; ++i) {
            c[i] = (float)X[i];
            c[n + i] = (float)w[i];
        }
        for (int i = 0, lo = 0, hi = 0; i < n; ++i) {
            while (c[i] - c[lo] > 5.0 * sigma) ++lo;
            hi = std::max(hi, i);
            while (hi < n - 1 && c[hi + 1] - c[i] <= 5.0 * sigma) ++hi;
            tab[nx + nz + o + i] = make_int2(lo, hi);
        }
    }
    GB_TRY(m->w_stage.ensure(tab.size() * sizeof(int2) + 64));
    GB_CUDA(cudaMemcpyAsync(m->w_stage.p, tab.data(), tab.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
    const float *dcx = m->w_stage.as<float>(), *dcz = dcx + 2 * nx;
    const int2 *drx = m->w_stage.as<int2>() + nx + nz, *drz = drx + nx;
    float inv2s2 = (float)(1.0 / (2.0 * sigma * sigma));
    const unsigned gx = (unsigned)((nx + 127) / 128);
    for (int z0 = 0; z0 < nz; z0 += 65535 * kSmoothRows) {
        const unsigned gy = (unsigned)std::min((nz - z0 + kSmoothRows - 1) / kSmoothRows, 65535);
        smooth_x_kernel<<<dim3(gx, gy), 128, 0, s>>>(Hd, S1, nx, nz, dcx, dcx + nx, drx, inv2s2, z0);
        GB_LAUNCHED();
    }
    smooth_z_kernel<<<dim3(gx, (unsigned)std::min(nz, 65535)), 128, 0, s>>>(S1, S2, nx, nz, dcz, dcz + nz, drz, inv2s2);
    GB_LAUNCHED();
    // medians of the smoothed maps (rank (N-1)/2)
    GB_TRY(m->w_red.ensure((1024 + 8) * sizeof(double) + 4096));
    unsigned *rstate = (unsigned *)(m->w_red.as<char>() + (1024 + 8) * sizeof(double));   // radix-select state
    unsigned *rhist = rstate + 12;
    float *med = (float *)(rhist + 768);
    radix_init<<<1, 256, 0, s>>>(rstate, rhist, (unsigned)((N - 1) / 2));
    GB_LAUNCHED();
    for (int shift = 24; shift >= 0; shift -= 8) {
        radix_hist<<<dim3((unsigned)std::min<long long>(grid_for(N), 304), 3), 256, 0, s>>>(S2, N, rstate, shift, rhist);
        GB_LAUNCHED();
        radix_pick<<<3, 256, 0, s>>>(rstate, rhist, shift, med);
        GB_LAUNCHED();
    }
    const bool dev_b0 = gb_is_device_ptr(B0);
    float *B0d = dev_b0 ? B0 : S1;   // S1 is free after the second pass
    b0_kernel<<<grid_for(3 * N), 256, 0, s>>>(S2, med, N, (float)damp, B0d);
    GB_LAUNCHED();
    if (!dev_b0) GB_CUDA(cudaMemcpyAsync(B0, B0d, 3 * N * sizeof(float), cudaMemcpyDeviceToHost, s));
    return GBFWI_OK;
}

// Shots a resident map run takes at once (0: the preconditioner steps run). Both
// passes keep their levels, so the batches are smaller than the steps' of Bold
// shots; a step costs about 5.3 us a launch resident, and 8 us forward (receiver maps) and
// 36 to 51 us a wave of 304 CTAs otherwise.  P4 measured from levels and by steps, 24 shots in one
// batch of steps: 40 x 20 elements, 300 steps: 3.8 and 13 ms; 81 x 21: 5.1 and 24 ms; 160 x 60, 200 steps
// (batches of 8 from levels): 19 and 82 ms; 340 x 70, 600 steps (one by one): 183 and 577 ms.  The steps
// win where few shots of a long run on a small mesh fit the memory for levels and
// the schedule lets many run together (40 x 20, 16000 steps, 24 shots a launch: 3.27 and 0.69 s; one a launch:
// 3.27 and 14.9 s).  Where both are close the rule loses 12% at most (81 x 21, 6000 steps, four streams).
static int map_batch(gbfwi_mesh *m, int nshot, bool receiver, int tile, int Bold, long long NP)
{
    const long long shot = (receiver ? 3 : 2) * (m->d.nt + 2LL) * NP * (long long)sizeof(float2);
    int B = (int)std::min<long long>({nshot, kMapHistory / shot, kMostShots});
    if (B < 1 || !gb_resident_plan(m, MODE_FWD, B)) return 0;
    B = (nshot + (nshot + B - 1) / B - 1) / ((nshot + B - 1) / B);      // equal batches
    const int fwd = receiver ? MODE_FWD : MODE_FWD_PC, rcv = receiver ? MODE_RCV : fwd, last = sizes::last_batch(nshot, B);
    const ResidentPlan *f = gb_resident_plan(m, fwd, B), *r = gb_resident_plan(m, rcv, B);
    if (!f || !r || !gb_resident_plan(m, fwd, last) || !gb_resident_plan(m, rcv, last)) return 0;
    const TileShape &t = kTiles[tile];
    const long long ctas = (long long)((m->d.nex + t.tx - 1) / t.tx) * ((m->d.nez + t.tz - 1) / t.tz) * Bold;
    const double launches = (B + f->per_launch - 1) / f->per_launch + (receiver ? (B + r->per_launch - 1) / r->per_launch : 0);
    const double here = (double)((nshot + B - 1) / B) * 5.3 * launches;
    const double steps = (double)((nshot + Bold - 1) / Bold) * ((receiver ? 8.0 : 0.0) + 38.0 * (double)((ctas + 303) / 304));
    return here < steps ? B : 0;
}

// buffers of resident_maps
static int reserve_maps(gbfwi_mesh *m, int nshot, int Bmax, bool receiver, bool strains)
{
    const long long NP = (long long)m->nz * m->pitch;
    const size_t levels = (size_t)(m->d.nt + 2) * Bmax * NP * sizeof(float2);
    Batches b;
    GB_TRY(receiver ? plan_batches(m, {MODE_FWD, MODE_RCV}, nshot, Bmax, NP, b) : plan_batches(m, {MODE_FWD_PC}, nshot, Bmax, NP, b));
    GB_TRY(m->w_hist.ensure(levels));
    GB_TRY(m->w_snap.ensure(levels));
    if (receiver) GB_TRY(m->w_adj.ensure(levels));
    if (receiver) GB_TRY(m->w_seis.ensure((size_t)m->nrec * 2 * m->d.nt * Bmax * sizeof(float)));
    if (strains) GB_TRY(m->w_eacc.ensure(gb_integral_bytes(m, Bmax)));
    GB_TRY(m->w_pc.ensure((size_t)Bmax * 4 * NP * sizeof(float)));
    return m->w_vh.ensure((size_t)Bmax * NP * sizeof(float2));
}

// the integrals of every shot (summed into tot) from stored levels
static int resident_maps(gbfwi_mesh *m, int nshot, int Bmax, int kind, int tile, float *tot, long long NP, cudaStream_t s)
{
    const int nt = m->d.nt;
    const bool receiver = kind == 2 || kind == 4, strains = kind >= 3;
    const int fwd = receiver ? MODE_FWD : MODE_FWD_PC;
    float *acc = m->w_pc.as<float>();
    float2 *vh = m->w_vh.as<float2>();
    for (int i0 = 0; i0 < nshot; i0 += Bmax) {
        const int B = std::min(Bmax, nshot - i0);
        const long long lev = B * NP;
        const Ctx c{m, &m->lists[tile], tile, B, s, m->w_shots.as<int>() + i0, NP, true};
        const Levels u{m->w_hist.as<float2>(), lev, 0, false};
        float2 *acc_levels = m->w_snap.as<float2>();
        const Levels w{m->w_adj.as<float2>(), lev, 0, false};
        auto at_rest = [&](const Levels &f) -> int {
            GB_CUDA(cudaMemsetAsync(f.base, 0, 2 * lev * sizeof(float2), s));
            GB_CUDA(cudaMemsetAsync(vh, 0, lev * sizeof(float2), s));
            return GBFWI_OK;
        };
        GB_TRY(at_rest(u));
        GB_CUDA(cudaMemsetAsync(acc, 0, (size_t)B * 4 * NP * sizeof(float), s));
        float *seis = m->w_seis.as<float>();
        GB_TRY(fwd_range(c, fwd, 0, nt, u, 0, vh, receiver ? seis : nullptr, nullptr, 0, 0, receiver ? nullptr : acc_levels));
        if (receiver) {
            GB_TRY(at_rest(w));
            GB_TRY(adj_range(c, MODE_RCV, 0, nt, w, vh, u, seis, nullptr, 0, 0, acc_levels));
        }
        GB_TRY(gb_time_integrals(m, B, receiver ? w.base : u.base, acc_levels, receiver ? u.base : nullptr, strains,
                                 m->w_eacc, acc, s));
        acc_reduce<<<grid_for(4 * NP), 256, 0, s>>>(acc, B, 4, NP, tot);
        GB_LAUNCHED();
    }
    return GBFWI_OK;
}

extern "C" int gbfwi_precond_diag(gbfwi_mesh *m, const int *shot_ids, int nshot, int kind, double sigma,
                                  double damp, float *H, float *B0, void *stream)
{
    if (!m || !B0 || kind < 1 || kind > 4 || !(sigma > 0) || !(damp >= 0)) return GBFWI_EINVAL;
    GB_TRY(gb_check_local(H, B0));
    GB_TRY(check_shots(m, shot_ids, nshot));
    if (!m->have_model) return GBFWI_ENOMODEL;
    cudaStream_t s = (cudaStream_t)stream;
    const int tile = m->sch.tile;
    GB_TRY(gb_build_tile_lists(m, tile));
    const int nt = m->d.nt;
    const long long NP = (long long)m->nz * m->pitch;
    const long long N = (long long)m->nz * m->nx;
    // shots in one launch: what the schedule keeps in flight (shots per launch x
    // streams), or more while their levels and maps stay small
    const bool receiver = kind == 2 || kind == 4;
    const int ck = m->sch.ckpt_every;
    const long long levels = !receiver ? 4 : ck <= 0 || ck >= nt ? nt + 6 : 3LL * ((nt + ck - 1) / ck) + ck + 10;
    const long long small = kSmallHistory / ((levels + 2) * NP * (long long)sizeof(float2));
    const int scheduled = std::min(m->sch.shots_per_launch, nshot);
    const int preferred =
        (int)std::min<long long>({nshot, std::max<long long>((long long)m->sch.shots_per_launch * m->sch.streams, small), kMostShots});
    const size_t seis_shot = (size_t)m->nrec * 2 * nt;
    const double dt = m->d.dt;

    const int Bmap = map_batch(m, nshot, receiver, tile, preferred, NP);
    auto fixed_buffers = [&]() -> int {
        GB_TRY(m->w_grad.ensure((size_t)5 * NP * sizeof(float)));
        GB_TRY(m->w_tmp.ensure((size_t)9 * N * sizeof(float) + 4096));
        return m->w_shots.ensure((size_t)nshot * sizeof(int));
    };
    // the maps from stored levels where their buffers fit, else the preconditioner steps
    BatchHist h;
    Batches batches;
    int rc = fixed_buffers();
    if (!rc && Bmap) rc = reserve_maps(m, nshot, Bmap, receiver, kind >= 3);
    const bool from_levels = Bmap && rc == GBFWI_OK;
    if (!from_levels) {
        if (rc && rc != GBFWI_ENOMEM) return rc;
        if (rc) release_batch_buffers(m);
        const auto steps = [&](const Batches &b) -> int {
            GB_TRY(fixed_buffers());
            GB_TRY(m->w_vh.ensure((size_t)b.most * NP * sizeof(float2)));
            GB_TRY(m->w_pc.ensure((size_t)b.most * 4 * NP * sizeof(float)));
            if (!receiver) return m->w_hist.ensure((size_t)3 * b.most * NP * sizeof(float2));
            GB_TRY(alloc_hist(m, lane0(m, s), b.most, ck, NP, h, true));
            return m->w_seis.ensure(seis_shot * b.most * sizeof(float));
        };
        const std::vector<Choice> choices = {{preferred, preferred, receiver}, {scheduled, scheduled, receiver}, {scheduled, scheduled, false}};
        GB_TRY(reserve_batches(m, {MODE_FWD}, nshot, choices, batches, steps));
    }
    GB_CUDA(cudaMemcpyAsync(m->w_shots.p, shot_ids, nshot * sizeof(int), cudaMemcpyHostToDevice, s));
    float *tot = m->w_grad.as<float>();
    GB_CUDA(cudaMemsetAsync(tot, 0, 4 * NP * sizeof(float), s));
    if (from_levels) GB_TRY(resident_maps(m, nshot, Bmap, kind, tile, tot, NP, s));
    const int Bmax = batches.most;
    for (int i0 = 0; i0 < nshot && !from_levels; i0 += Bmax) {
        int B = std::min(Bmax, nshot - i0);
        Ctx c{m, &m->lists[tile], tile, B, s, m->w_shots.as<int>() + i0, NP, batches.resident(B)};
        float *acc = m->w_pc.as<float>();
        GB_CUDA(cudaMemsetAsync(acc, 0, (size_t)B * 4 * NP * sizeof(float), s));
        long long blev = (long long)B * NP;
        if (!receiver) {
            const Levels ring{m->w_hist.as<float2>(), blev, 0, true};
            GB_CUDA(cudaMemsetAsync(ring.base, 0, 3 * blev * sizeof(float2), s));
            GB_CUDA(cudaMemsetAsync(m->w_vh.p, 0, blev * sizeof(float2), s));
            GB_TRY(fwd_range(c, MODE_FWD_PC, 0, nt, ring, 0, m->w_vh.as<float2>(), nullptr, acc, 4 * NP, NP));
        } else {
            // receiver wavefield: adjoint recurrence driven by the synthetic data s(m0)
            float *seis_d = m->w_seis.as<float>();
            GB_TRY(forward_pass(c, h, seis_d));
            GB_TRY(adjoint_pass(c, h, MODE_ADJ_PC, seis_d, acc, 4 * NP, NP));
        }
        acc_reduce<<<grid_for(4 * NP), 256, 0, s>>>(acc, B, 4, NP, tot);
        GB_LAUNCHED();
    }
    // time-integral factors: forward mode S0 = sum a.a (x dt), S1..3 = sum of
    // products of undivided differences (x 1/dt); receiver mode S0 = sum of
    // (second difference) . a (x 1/dt)
    float f0 = (kind == 1 || kind == 3) ? (float)dt : (float)(1.0 / dt);
    float f1 = (float)(1.0 / dt);
    float *Hd = m->w_tmp.as<float>();
    float *S1 = Hd + 3 * N, *S2 = Hd + 6 * N;
    precond_finish<<<grid_for(N), 256, 0, s>>>(tot, m->d_model.as<float>(), m->d_wx.as<float>(),
                                               m->d_wz.as<float>(), m->nx, m->nz, m->pitch, kind, f0, f1, Hd);
    GB_LAUNCHED();

    GB_TRY(b0_from_map(m, Hd, S1, S2, sigma, damp, B0, s));
    if (H) {
        if (gb_is_device_ptr(H))
            GB_CUDA(cudaMemcpyAsync(H, Hd, 3 * N * sizeof(float), cudaMemcpyDeviceToDevice, s));
        else
            GB_CUDA(cudaMemcpyAsync(H, Hd, 3 * N * sizeof(float), cudaMemcpyDeviceToHost, s));
    }
    GB_CUDA(cudaStreamSynchronize(s));
    GB_TRY(gb_take_status(m));
    return GBFWI_OK;
}

extern "C" int gbfwi_precond_from_hessian(gbfwi_mesh *m, const float *H, double sigma, double damp, float *B0,
                                          void *stream)
{
    if (!m || !H || !B0 || !(sigma > 0) || !(damp >= 0)) return GBFWI_EINVAL;
    GB_TRY(gb_check_local(H, B0));
    cudaStream_t s = (cudaStream_t)stream;
    const long long N = (long long)m->nx * m->nz;
    GB_TRY(m->w_tmp.ensure((size_t)9 * N * sizeof(float) + 4096));
    float *Hd = m->w_tmp.as<float>();
    float *S1 = Hd + 3 * N, *S2 = Hd + 6 * N;
    GB_CUDA(cudaMemcpyAsync(Hd, H, 3 * N * sizeof(float), cudaMemcpyDefault, s));
    GB_TRY(b0_from_map(m, Hd, S1, S2, sigma, damp, B0, s));
    GB_CUDA(cudaStreamSynchronize(s));
    return GBFWI_OK;
}
