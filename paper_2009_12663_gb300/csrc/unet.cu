// Learned diagonal preconditioner: a U-Net in bfloat16 that predicts the
// logarithm of the diagonal pseudo-Hessian (the P-maps of Eqs. 5-8) from
// the model and the acquisition, with its training (backward pass, mean
// squared loss, Adam) and inference on sm_103a.  The paper has no learned
// component; the network is the standard U-Net of Ronneberger, Fischer &
// Brox (2015): per level two 3x3 convolutions with ReLU, 2x2 average
// pooling down, nearest 2x upsampling up, skip connections concatenated
// after the upsampled features, a 1x1 output convolution.
//
// Every convolution is a dense contraction and runs on the tensor cores as
// one BF16 GEMM with FP32 accumulation (mma.sync m16n8k16, fed by ldmatrix):
//   forward        Y[co][p]   = W[co][kk] X[kk][p]          (+ bias, ReLU, -> bf16)
//   weight grad    dW[co][kk] += G[co][p] X^T[p][kk]        (split over p, splits summed in order)
//   input grad     dX[c][p]   = sum_tap (sum_co W[co][c, tap] G[co][p - tap])
// with kk = c*9 + ky*3 + kx and X[kk][y*W + x] = x[c][y+ky-1][x+kx-1] (zero
// outside).  The column matrix X is never written: the kernels gather its
// 8-pixel chunks from the activations (with upsampling and concatenation) while
// they stage a tile, one 16-byte load and a shift by one pixel per chunk.  Every
// sum keeps the order it had with a stored column matrix (the same 16-deep MMA
// steps, the same splits, taps added in order), so results are bit for bit the
// same; what went is the traffic (1.4 GB written and read again per inference at
// 256 x 1024, 2.8 GB more per training step).  All launches take the samples of
// a batch together (blockIdx.z): small images are bound by launch latency.
// Everything around the GEMMs (pooling, the ReLU masks of the gradients, bias
// sums, loss, Adam, resampling) is memory-bound and written as plain coalesced
// kernels.
//
// Storage points (where values are rounded to bfloat16, round to nearest
// even): input image, weights, every ReLU activation, the average-pooled
// maps, and the masked gradients fed to the GEMMs.  The output map, the
// input-gradient sums and all parameter gradients are FP32.

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>
#include <vector>

#include "gbfwi_internal.h"
#include "size_rules.h"

using namespace sizes;

typedef __nv_bfloat16 bf16;

namespace {

// ---------------------------------------------------------------------------
// BF16 GEMM on the tensor cores
// ---------------------------------------------------------------------------

constexpr int GBK = sizes::kGemmBK;   // k extent of a staged tile
constexpr int GPAD = 8;        // bf16 padding per shared row (ldmatrix rows on distinct banks)
constexpr int GTHREADS = 256;  // 8 warps, each owning a 32 x 32 block of C
constexpr int GSTAGES = 3;     // cp.async pipeline depth (tiles in flight + 1)
// A gathered tile passes through registers within one iteration, so a third
// stage hides nothing; two leave room for four CTAs an SM, whose loads cover
// each other (the whole forward pass at 256 x 1024 gains 4%)
template <bool GATHER>
constexpr int kStages = GATHER ? 2 : GSTAGES;

// activations a 3x3 convolution reads: channels c < C1 from s1,
// nearest-upsampled from (H/2, W/2) when up1; the rest from s2 (the skip
// connection, concatenated after s1); bs1, bs2: elements between samples
struct ConvSrc {
    const bf16 *s1, *s2;
    int C1, up1, C2, H, W;
    long long bs1, bs2;
};

struct GemmArgs {
    const bf16 *A;
    long long lda;
    const bf16 *B;
    long long ldb;
    int M, N, K;
    int kchunk;                // k range of one split
    float *Cf;                 // FP32 output (or split partials), may be null
    bf16 *Cb;                  // bf16 output, may be null
    const float *bias;         // per row of C, may be null
    int relu;
    int accumulate;            // Cf += result
    long long ldc;
    long long split_stride;    // elements between split partials
    int splits;
    int partial;               // write split partials [sample][split][M][N]
    long long abs_, bbs, cbs;  // elements between samples of A, B, C
    ConvSrc src;               // gathered B
};

__device__ __forceinline__ void cp16(void *smem, const void *gmem, bool valid)
{
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(valid ? 16 : 0));
}

__device__ __forceinline__ void ldsm_x4(unsigned (&r)[4], const void *p)
{
    unsigned s = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(s));
}

__device__ __forceinline__ void ldsm_x4_t(unsigned (&r)[4], const void *p)
{
    unsigned s = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(s));
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                 "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Chunk of 8 pixels (y, x0 ..) of row (c, ky, kx) of the column matrix: the
// aligned 16 bytes (8 when upsampled) and, in e, the pixel beyond them that the
// shift brings in, the shift and the upsampling flag.
__device__ __forceinline__ void fetch8(const ConvSrc &S, const bf16 *s1, const bf16 *s2, int c, int ky, int kx, int y, int x0,
                                       bool in, uint4 &v, unsigned &e)
{
    v = make_uint4(0u, 0u, 0u, 0u);
    e = 1u << 16;
    const int ys = y + ky - 1;
    if (!in || c >= S.C1 + S.C2 || ys < 0 || ys >= S.H) return;
    const int xe = kx == 0 ? x0 - 1 : x0 + 8;
    const bool edge = kx != 1 && xe >= 0 && xe < S.W;
    if (c < S.C1 && S.up1) {
        const bf16 *row = s1 + ((long long)c * (S.H / 2) + ys / 2) * (S.W / 2);
        const uint2 q = *reinterpret_cast<const uint2 *>(row + x0 / 2);
        v.x = q.x;
        v.y = q.y;
        e = (edge ? (unsigned)*reinterpret_cast<const unsigned short *>(row + xe / 2) : 0u) | (unsigned)kx << 16 | 1u << 18;
    } else {
        const bf16 *row = c < S.C1 ? s1 + ((long long)c * S.H + ys) * S.W : s2 + ((long long)(c - S.C1) * S.H + ys) * S.W;
        v = *reinterpret_cast<const uint4 *>(row + x0);
        e = (edge ? (unsigned)*reinterpret_cast<const unsigned short *>(row + xe) : 0u) | (unsigned)kx << 16;
    }
}

__device__ __forceinline__ uint4 shift8(uint4 v, unsigned e)
{
    if (e >> 18 & 1)
        v = make_uint4(__byte_perm(v.x, 0, 0x1010), __byte_perm(v.x, 0, 0x3232), __byte_perm(v.y, 0, 0x1010),
                       __byte_perm(v.y, 0, 0x3232));
    const unsigned kx = e >> 16 & 3u;
    if (kx == 0)
        return make_uint4(v.x << 16 | (e & 0xffffu), __funnelshift_l(v.x, v.y, 16), __funnelshift_l(v.y, v.z, 16),
                          __funnelshift_l(v.z, v.w, 16));
    if (kx == 2)
        return make_uint4(__funnelshift_r(v.x, v.y, 16), __funnelshift_r(v.y, v.z, 16), __funnelshift_r(v.z, v.w, 16),
                          v.w >> 16 | e << 16);
    return v;
}

// Shared tiles of one stage.  A_KM: A stored [K][M] (m contiguous), else
// [M][K]; B_NK: B stored [N][K] (k contiguous), else [K][N].
template <int BM, int BN, bool A_KM, bool B_NK>
struct GemmTile {
    static constexpr int AP = A_KM ? BM + GPAD : GBK + GPAD;     // shared row pitch (bf16)
    static constexpr int BP = B_NK ? GBK + GPAD : BN + GPAD;
    static constexpr int AE = A_KM ? GBK * AP : BM * AP;          // elements per stage
    static constexpr int BE = B_NK ? BN * BP : GBK * BP;
    static constexpr int ACH = BM * GBK / 8;                      // 16-byte chunks per stage
    static constexpr int BCH = BN * GBK / 8;
    static constexpr int BPT = BCH / GTHREADS;                    // of B per thread
    static_assert(BCH % GTHREADS == 0, "chunks of B");
};

template <int BM, int BN, bool A_KM>
__device__ __forceinline__ void stage_a(const GemmArgs &g, const bf16 *A, bf16 *As, int m0, int k0, int kend)
{
    using T = GemmTile<BM, BN, A_KM, false>;
    for (int q = threadIdx.x; q < T::ACH; q += GTHREADS) {
        int r, c;
        const bf16 *src;
        bool ok;
        if (A_KM) {                       // rows k, 8 m per chunk
            r = q / (BM / 8);
            c = (q % (BM / 8)) * 8;
            ok = (k0 + r < kend) && (m0 + c < g.M);
            src = A + (long long)(k0 + r) * g.lda + m0 + c;
        } else {                          // rows m, 8 k per chunk
            r = q / (GBK / 8);
            c = (q % (GBK / 8)) * 8;
            ok = (m0 + r < g.M) && (k0 + c < kend);
            src = A + (long long)(m0 + r) * g.lda + k0 + c;
        }
        cp16(As + r * T::AP + c, ok ? src : A, ok);
    }
}

template <int BM, int BN, bool A_KM, bool B_NK>
__device__ __forceinline__ void stage_b(const GemmArgs &g, const bf16 *B, bf16 *Bs, int n0, int k0, int kend)
{
    using T = GemmTile<BM, BN, A_KM, B_NK>;
    for (int q = threadIdx.x; q < T::BCH; q += GTHREADS) {
        int r, c;
        const bf16 *src;
        bool ok;
        if (B_NK) {                       // rows n, 8 k per chunk
            r = q / (GBK / 8);
            c = (q % (GBK / 8)) * 8;
            ok = (n0 + r < g.N) && (k0 + c < kend);
            src = B + (long long)(n0 + r) * g.ldb + k0 + c;
        } else {                          // rows k, 8 n per chunk
            r = q / (BN / 8);
            c = (q % (BN / 8)) * 8;
            ok = (k0 + r < kend) && (n0 + c < g.N);
            src = B + (long long)(k0 + r) * g.ldb + n0 + c;
        }
        cp16(Bs + r * T::BP + c, ok ? src : B, ok);
    }
}

// this thread's chunks of a gathered tile of B (rows kk of the column matrix)
template <int BM, int BN, bool B_NK>
__device__ __forceinline__ void fetch_b(const GemmArgs &g, const bf16 *s1, const bf16 *s2, int n0, int k0, int kend,
                                        uint4 (&v)[GemmTile<BM, BN, false, B_NK>::BPT],
                                        unsigned (&e)[GemmTile<BM, BN, false, B_NK>::BPT])
{
    using T = GemmTile<BM, BN, false, B_NK>;
    // the pixels of a thread's chunks are the same in all of them
    const int p = B_NK ? k0 + (threadIdx.x % (GBK / 8)) * 8 : n0 + (threadIdx.x % (BN / 8)) * 8;
    const int y = p / g.src.W, x0 = p - y * g.src.W;
    const bool in = p < (B_NK ? kend : g.N);
#pragma unroll
    for (int i = 0; i < T::BPT; ++i) {
        const int q = threadIdx.x + i * GTHREADS;
        const int kk = B_NK ? n0 + q / (GBK / 8) : k0 + q / (BN / 8);
        const int c = kk / 9, t = kk - 9 * c;
        fetch8(g.src, s1, s2, c, t / 3, t % 3, y, x0, in && kk < (B_NK ? g.N : kend), v[i], e[i]);
    }
}

template <int BM, int BN, bool B_NK>
__device__ __forceinline__ void put_b(bf16 *Bs, const uint4 (&v)[GemmTile<BM, BN, false, B_NK>::BPT],
                                      const unsigned (&e)[GemmTile<BM, BN, false, B_NK>::BPT])
{
    using T = GemmTile<BM, BN, false, B_NK>;
#pragma unroll
    for (int i = 0; i < T::BPT; ++i) {
        const int q = threadIdx.x + i * GTHREADS;
        const int r = B_NK ? q / (GBK / 8) : q / (BN / 8), c = B_NK ? (q % (GBK / 8)) * 8 : (q % (BN / 8)) * 8;
        *reinterpret_cast<uint4 *>(Bs + r * T::BP + c) = shift8(v[i], e[i]);
    }
}

// the MMAs of one staged tile
template <int BM, int BN, bool A_KM, bool B_NK>
__device__ __forceinline__ void tile_mma(const bf16 *as, const bf16 *bs, int wm, int wn, int lane, float (&acc)[2][4][4])
{
    using T = GemmTile<BM, BN, A_KM, B_NK>;
#pragma unroll
    for (int kk = 0; kk < GBK; kk += 16) {
        unsigned a[2][4], b[4][2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int mb = wm * 32 + i * 16;
            if (A_KM) {
                int k = kk + (lane & 7) + ((lane >> 4) << 3);
                int m = mb + (((lane >> 3) & 1) << 3);
                ldsm_x4_t(a[i], as + k * T::AP + m);
            } else {
                int m = mb + (lane & 15);
                int k = kk + ((lane >> 4) << 3);
                ldsm_x4(a[i], as + m * T::AP + k);
            }
        }
#pragma unroll
        for (int jb = 0; jb < 2; ++jb) {
            const int nb = wn * 32 + jb * 16;
            unsigned r[4];
            if (B_NK) {
                int n = nb + (lane & 7) + ((lane >> 4) << 3);
                int k = kk + (((lane >> 3) & 1) << 3);
                ldsm_x4(r, bs + n * T::BP + k);
            } else {
                int k = kk + (lane & 15);
                int n = nb + ((lane >> 4) << 3);
                ldsm_x4_t(r, bs + k * T::BP + n);
            }
            b[2 * jb][0] = r[0];
            b[2 * jb][1] = r[1];
            b[2 * jb + 1][0] = r[2];
            b[2 * jb + 1][1] = r[3];
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a[i], b[j][0], b[j][1]);
    }
}

// C tile BM x BN per CTA, warps arranged (BM/32) x (BN/32), each warp
// 2 x 4 mma tiles of 16 x 8; blockIdx.z = sample * splits + split.  A (and a
// stored B) by cp.async ahead of its use, a gathered B through registers
// (loaded before the tile's MMAs, written after them).  Requirements (checked on
// the host): K % 8 == 0, lda, ldb multiples of 8, 16-byte aligned bases, M % 8 ==
// 0 when A_KM, N % 8 == 0 when !B_NK, N even; gathered: W % 8 == 0.
template <int BM, int BN, bool A_KM, bool B_NK, bool GATHER>
__global__ void __launch_bounds__(GTHREADS, GATHER ? (BM == 32 ? 3 : 4) : 1) gemm_bf16_kernel(const GemmArgs g)
{
    using T = GemmTile<BM, BN, A_KM, B_NK>;
    static_assert((BM / 32) * (BN / 32) == GTHREADS / 32, "warp layout");
    constexpr int ST = kStages<GATHER>;
    extern __shared__ __align__(16) unsigned char gsm[];   // ST x (A tile, B tile)
    bf16 *As0 = reinterpret_cast<bf16 *>(gsm);
    bf16 *Bs0 = As0 + ST * T::AE;

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wm = warp % (BM / 32), wn = warp / (BM / 32);
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int sample = blockIdx.z / g.splits, split = blockIdx.z - sample * g.splits;
    const int kbeg = split * g.kchunk;
    const int kend = min(g.K, kbeg + g.kchunk);
    const bf16 *A = g.A + sample * g.abs_, *B = GATHER ? nullptr : g.B + sample * g.bbs;
    const bf16 *s1 = nullptr, *s2 = nullptr;
    if (GATHER) {
        s1 = g.src.s1 + sample * g.src.bs1;
        s2 = g.src.s2 + sample * g.src.bs2;
    }

    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[i][j][v] = 0.f;

    uint4 bv[T::BPT];
    unsigned be[T::BPT];
    // tiles it+1 .. it+ST-1 are under way while tile it is consumed; every
    // iteration commits one group (empty past the end) so that wait_group
    // ST-2 always means "tile it landed"
#pragma unroll
    for (int sidx = 0; sidx < ST - 1; ++sidx) {
        const int kk0 = kbeg + sidx * GBK;
        if (kk0 < kend) {
            stage_a<BM, BN, A_KM>(g, A, As0 + sidx * T::AE, m0, kk0, kend);
            if (GATHER) {
                fetch_b<BM, BN, B_NK>(g, s1, s2, n0, kk0, kend, bv, be);
                put_b<BM, BN, B_NK>(Bs0 + sidx * T::BE, bv, be);
            } else {
                stage_b<BM, BN, A_KM, B_NK>(g, B, Bs0 + sidx * T::BE, n0, kk0, kend);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::);
    }
    int it = 0;
    for (int k0 = kbeg; k0 < kend; k0 += GBK, ++it) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(ST - 2));
        __syncthreads();
        // refill the slot consumed in the previous iteration (all threads are
        // past it: the barrier above)
        const int kn = k0 + (ST - 1) * GBK;
        const int slot = (it + ST - 1) % ST;
        if (kn < kend) {
            stage_a<BM, BN, A_KM>(g, A, As0 + slot * T::AE, m0, kn, kend);
            if (GATHER) fetch_b<BM, BN, B_NK>(g, s1, s2, n0, kn, kend, bv, be);
            else stage_b<BM, BN, A_KM, B_NK>(g, B, Bs0 + slot * T::BE, n0, kn, kend);
        }
        asm volatile("cp.async.commit_group;\n" ::);
        const int cur = it % ST;
        tile_mma<BM, BN, A_KM, B_NK>(As0 + cur * T::AE, Bs0 + cur * T::BE, wm, wn, lane, acc);
        if (GATHER && kn < kend) put_b<BM, BN, B_NK>(Bs0 + slot * T::BE, bv, be);
    }
    asm volatile("cp.async.wait_group 0;\n" ::);

    // epilogue: thread holds rows g, g+8 and columns 2t, 2t+1 of each 16 x 8 tile
    const int gr = lane >> 2, tc = (lane & 3) * 2;
    float *Cf = g.Cf ? g.Cf + (g.partial ? (long long)blockIdx.z * g.split_stride : sample * g.cbs) : nullptr;
    bf16 *Cb = g.Cb ? g.Cb + sample * g.cbs : nullptr;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int m = m0 + wm * 32 + i * 16 + gr + 8 * h;
            if (m >= g.M) continue;
            const float bm = (!g.partial && g.bias) ? g.bias[m] : 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int n = n0 + wn * 32 + j * 8 + tc;
                if (n >= g.N) continue;
                float v0 = acc[i][j][2 * h] + bm, v1 = acc[i][j][2 * h + 1] + bm;
                if (g.partial) {
                    *reinterpret_cast<float2 *>(Cf + (long long)m * g.ldc + n) = make_float2(v0, v1);
                    continue;
                }
                if (g.relu) {
                    v0 = fmaxf(v0, 0.f);
                    v1 = fmaxf(v1, 0.f);
                }
                if (Cf) {
                    float2 *p = reinterpret_cast<float2 *>(Cf + (long long)m * g.ldc + n);
                    if (g.accumulate) {
                        float2 o = *p;
                        v0 += o.x;
                        v1 += o.y;
                    }
                    *p = make_float2(v0, v1);
                }
                if (Cb) {
                    __nv_bfloat162 o = __floats2bfloat162_rn(v0, v1);
                    *reinterpret_cast<__nv_bfloat162 *>(Cb + (long long)m * g.ldc + n) = o;
                }
            }
        }
}

// Input gradient of a 3x3 convolution: dX[c][p] = sum over the nine taps, in
// order, of sum_co Wt[tap][co][c] G[co][y - ky + 1][x - kx + 1] (zero outside).
// Each tap's sum starts from zero (and from zero again at every kchunk of co,
// the parts added in order), as if the taps' products were stored and then
// gathered.  A = Wt + tap * K * lda ([K][M]); B gathered from G.  With partial,
// blockIdx.z = sample * 9 + tap and every tap's sum goes to [sample][tap][M][N]:
// at the coarse levels the nine taps of a few tiles one after another leave the
// chip idle (2 x 4 tiles of 128 x 64 and 256 channels: 73 us, 14 + 5 us with the
// sum of the taps).
template <int BM, int BN>
__global__ void __launch_bounds__(GTHREADS, 2) conv_dx_kernel(const GemmArgs g)
{
    using T = GemmTile<BM, BN, true, false>;
    extern __shared__ __align__(16) unsigned char gsm[];
    bf16 *As0 = reinterpret_cast<bf16 *>(gsm);
    bf16 *Bs0 = As0 + GSTAGES * T::AE;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wm = warp % (BM / 32), wn = warp / (BM / 32);
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int sample = g.partial ? blockIdx.z / 9 : blockIdx.z, tap0 = g.partial ? blockIdx.z - 9 * sample : 0;
    const bf16 *G = g.src.s1 + sample * g.src.bs1;
    const int nk = (g.K + GBK - 1) / GBK, total = (g.partial ? 1 : 9) * nk, per = g.kchunk / GBK;   // tiles per tap, in all, per part
    const int p = n0 + (threadIdx.x % (BN / 8)) * 8, y = p / g.src.W, x0 = p - y * g.src.W;

    float acc[2][4][4], part[2][4][4], sum[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[i][j][v] = part[i][j][v] = sum[i][j][v] = 0.f;
    uint4 bv[T::BPT];
    unsigned be[T::BPT];
    auto fetch = [&](int t) {
        const int tt = t / nk, tap = tap0 + tt, k0 = (t - tt * nk) * GBK, ky = tap / 3, kx = tap - 3 * ky;
#pragma unroll
        for (int i = 0; i < T::BPT; ++i) {
            const int co = k0 + (threadIdx.x + i * GTHREADS) / (BN / 8);
            fetch8(g.src, G, G, co, 2 - ky, 2 - kx, y, x0, p < g.N && co < g.K, bv[i], be[i]);
        }
    };
    auto stage = [&](int t, int slot) {
        const int tt = t / nk, tap = tap0 + tt, k0 = (t - tt * nk) * GBK;
        stage_a<BM, BN, true>(g, g.A + (long long)tap * g.K * g.lda, As0 + slot * T::AE, m0, k0, g.K);
    };
#pragma unroll
    for (int sidx = 0; sidx < GSTAGES - 1; ++sidx) {
        if (sidx < total) {
            stage(sidx, sidx);
            fetch(sidx);
            put_b<BM, BN, false>(Bs0 + sidx * T::BE, bv, be);
        }
        asm volatile("cp.async.commit_group;\n" ::);
    }
    for (int it = 0; it < total; ++it) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(GSTAGES - 2));
        __syncthreads();
        const int tn = it + GSTAGES - 1, slot = tn % GSTAGES, cur = it % GSTAGES;
        if (tn < total) {
            stage(tn, slot);
            fetch(tn);
        }
        asm volatile("cp.async.commit_group;\n" ::);
        tile_mma<BM, BN, true, false>(As0 + cur * T::AE, Bs0 + cur * T::BE, wm, wn, lane, acc);
        if (tn < total) put_b<BM, BN, false>(Bs0 + slot * T::BE, bv, be);
        const int kt = it % nk;
        const bool end = kt == nk - 1;
        if (end || (kt + 1) % per == 0) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        part[i][j][v] += acc[i][j][v];
                        acc[i][j][v] = 0.f;
                        if (end) {
                            sum[i][j][v] += part[i][j][v];
                            part[i][j][v] = 0.f;
                        }
                    }
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::);
    const int gr = lane >> 2, tc = (lane & 3) * 2;
    float *Cf = g.Cf + blockIdx.z * (g.partial ? g.split_stride : g.cbs);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int m = m0 + wm * 32 + i * 16 + gr + 8 * h;
            if (m >= g.M) continue;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int n = n0 + wn * 32 + j * 8 + tc;
                if (n < g.N)
                    *reinterpret_cast<float2 *>(Cf + (long long)m * g.ldc + n) = make_float2(sum[i][j][2 * h], sum[i][j][2 * h + 1]);
            }
        }
}

// sum of the split partials in split order, then the epilogue of the GEMM.  V (4
// where the rows allow it) consecutive outputs a thread: bound by the partials'
// reads.
template <int V>
__global__ void __launch_bounds__(256) gemm_reduce_kernel(const float *__restrict__ part, int splits, int M, int N,
                                                          long long ldc, long long cbs, const float *__restrict__ bias, int relu,
                                                          float *__restrict__ Cf, bf16 *__restrict__ Cb)
{
    const long long total = (long long)M * N;
    struct alignas(4 * V) Vec { float v[V]; };
    struct alignas(2 * V) VecB { bf16 v[V]; };
    part += blockIdx.y * splits * total;
    for (long long q = V * (blockIdx.x * (long long)blockDim.x + threadIdx.x); q < total;
         q += (long long)gridDim.x * blockDim.x * V) {
        const int m = total < (1LL << 31) ? (int)((unsigned)q / (unsigned)N) : (int)(q / N);
        const long long at = blockIdx.y * cbs + (long long)m * ldc + (q - (long long)m * N);
        Vec s;
#pragma unroll
        for (int v = 0; v < V; ++v) s.v[v] = 0.f;
#pragma unroll 8
        for (int z = 0; z < splits; ++z) {
            const Vec x = *reinterpret_cast<const Vec *>(part + z * total + q);
#pragma unroll
            for (int v = 0; v < V; ++v) s.v[v] += x.v[v];
        }
        VecB h;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if (bias) s.v[v] += bias[m];
            if (relu) s.v[v] = fmaxf(s.v[v], 0.f);
            h.v[v] = __float2bfloat16_rn(s.v[v]);
        }
        if (Cf) *reinterpret_cast<Vec *>(Cf + at) = s;
        if (Cb) *reinterpret_cast<VecB *>(Cb + at) = h;
    }
}

// Cf += the samples' sums of split partials, the samples in order (weight
// gradients), a thread per output
__global__ void __launch_bounds__(256) grad_rows_kernel(const float *__restrict__ part, int samples, int splits, int M, int N,
                                                        long long ldc, float *__restrict__ Cf)
{
    const long long total = (long long)M * N;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total; q += (long long)gridDim.x * blockDim.x) {
        const int m = total < (1LL << 31) ? (int)((unsigned)q / (unsigned)N) : (int)(q / N);
        float *c = Cf + (long long)m * ldc + (q - (long long)m * N);
        float o = *c;
        for (int b = 0; b < samples; ++b) {
            float s = 0.f;
#pragma unroll 8
            for (int z = 0; z < splits; ++z) s += part[((long long)b * splits + z) * total + q];
            o += s;
        }
        *c = o;
    }
}

// The same for few outputs with many partials each: a warp takes a sample's
// partials of 32 outputs with 16 loads in flight, then one warp adds the samples
// (9216 outputs of 128 partials: 50 us with a thread per output, 6 us so; 442368
// outputs of 32: 8 us and 41 us).
__global__ void __launch_bounds__(256) grad_reduce_kernel(const float *__restrict__ part, int samples, int splits, int M, int N,
                                                          long long ldc, float *__restrict__ Cf)
{
    __shared__ float sums[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const long long total = (long long)M * N, q = blockIdx.x * 32LL + lane;
    const bool on = q < total;
    const int m = (int)(q / N);
    float *c = Cf + (long long)m * ldc + (q - (long long)m * N);
    float o = on && w == 0 ? *c : 0.f;
    for (int b0 = 0; b0 < samples; b0 += nw) {
        float s = 0.f;
        if (on && b0 + w < samples)
#pragma unroll 16
            for (int z = 0; z < splits; ++z) s += part[((long long)(b0 + w) * splits + z) * total + q];
        sums[w][lane] = s;
        __syncthreads();
        if (w == 0)
            for (int b = 0; b < min(nw, samples - b0); ++b) o += sums[b][lane];
        __syncthreads();
    }
    if (on && w == 0) *c = o;
}

}  // namespace

namespace {

// ---------------------------------------------------------------------------
// layout kernels (the channels of all samples of a batch are one long list
// where they need not be told apart)
// ---------------------------------------------------------------------------

// out[c][y][x] = mean of in[c][2y..2y+1][2x..2x+1] (H, W of the output)
__global__ void avgpool_kernel(const bf16 *__restrict__ in, int C, int H, int W, bf16 *__restrict__ out)
{
    const long long total = (long long)C * H * W;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
         q += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(q % W);
        const long long cy = q / W;
        const int y = (int)(cy % H), c = (int)(cy / H);
        const bf16 *r0 = in + ((long long)c * 2 * H + 2 * y) * (2 * W) + 2 * x;
        const bf16 *r1 = r0 + 2 * W;
        float s = (__bfloat162float(r0[0]) + __bfloat162float(r0[1])) +
                  (__bfloat162float(r1[0]) + __bfloat162float(r1[1]));
        out[q] = __float2bfloat16_rn(0.25f * s);
    }
}

// Gradient reaching a ReLU activation y [C][H][W], masked by y > 0 and
// rounded for the next GEMM:
//   g = fine (2x2 sum of a [C][2H][2W] map: upsampling adjoint)   when fine
//     + 0.25 * coarse[c][y/2][x/2]   (average-pooling adjoint)      when coarse
//     + direct[c][y][x]                                             when direct
__global__ void grad_mask_kernel(const float *__restrict__ fine, long long fine_bs, const float *__restrict__ coarse,
                                 const float *__restrict__ direct, long long direct_bs, const bf16 *__restrict__ y, int C,
                                 int H, int W, bf16 *__restrict__ out)
{
    // blockIdx.y: sample; fine and direct may be channel ranges of wider maps
    const long long total = (long long)C * H * W;
    if (fine) fine += blockIdx.y * fine_bs;
    if (coarse) coarse += blockIdx.y * (total / 4);
    if (direct) direct += blockIdx.y * direct_bs;
    y += blockIdx.y * total;
    out += blockIdx.y * total;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
         q += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(q % W);
        const long long cy = q / W;
        const int yy = (int)(cy % H), c = (int)(cy / H);
        float g = 0.f;
        if (fine) {
            const float *r0 = fine + ((long long)c * 2 * H + 2 * yy) * (2 * W) + 2 * x;
            const float *r1 = r0 + 2 * W;
            g += (r0[0] + r0[1]) + (r1[0] + r1[1]);
        }
        if (coarse) g += 0.25f * coarse[((long long)c * (H / 2) + yy / 2) * (W / 2) + x / 2];
        if (direct) g += direct[q];
        out[q] = __float2bfloat16_rn(__bfloat162float(y[q]) > 0.f ? g : 0.f);
    }
}

// part[b][m] = sum_p G[b][m][p]: one CTA per row and sample, fixed-order tree;
// db[m] += part[b][m] sample by sample
__global__ void rowsum_kernel(const bf16 *__restrict__ G, long long P, int rows, float *__restrict__ part,
                              float *__restrict__ db)
{
    __shared__ float red[256];
    const bf16 *g = G + ((long long)blockIdx.y * rows + blockIdx.x) * P;
    float s = 0.f;
#pragma unroll 8
    for (long long p = threadIdx.x; p < P; p += blockDim.x) s += __bfloat162float(g[p]);
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (db) db[blockIdx.x] += red[0];                // a single sample needs no second pass
        else part[blockIdx.y * rows + blockIdx.x] = red[0];
    }
}

__global__ void rowsum_add_kernel(const float *__restrict__ part, int samples, int rows, float *__restrict__ db)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= rows) return;
    float s = db[m];
    for (int b = 0; b < samples; ++b) s += part[b * rows + m];
    db[m] = s;
}

// Wt[tap][co][c] = W[co][c * 9 + tap] of every 3x3 layer (blockIdx.y) in one launch
struct WtLayer { long long off; int cout, cin, kcp; };
struct WtTable { WtLayer l[4 * 6]; };

__global__ void transpose_weights_kernel(const bf16 *__restrict__ Wall, const WtTable tab, bf16 *__restrict__ Wtall)
{
    const WtLayer L = tab.l[blockIdx.y];
    const bf16 *W = Wall + L.off;
    bf16 *Wt = Wtall + L.off;
    const int total = 9 * L.cout * L.cin;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < total; q += gridDim.x * blockDim.x) {
        const int c = q % L.cin, r = q / L.cin, co = r % L.cout, tap = r / L.cout;
        Wt[q] = W[(long long)co * L.kcp + c * 9 + tap];
    }
}

__global__ void to_bf16_kernel(const float *__restrict__ in, long long n, bf16 *__restrict__ out)
{
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        out[q] = __float2bfloat16_rn(in[q]);
}

// Mean squared error over `cout` channels of pred [cpad][P] against
// target [cout][P]: per-block partial sums (FP32 products, FP64 block sums),
// and dy [cpad][P] = gscale 2 (pred - target) / (cout P) (zero rows beyond
// cout; gscale = 1 / batch gives the gradient of the batch mean).  blockIdx.y:
// sample.
__global__ void mse_kernel(const float *__restrict__ pred, const float *__restrict__ target, int cout, int cpad,
                           long long P, float gscale, double *__restrict__ partial, bf16 *__restrict__ dy)
{
    __shared__ double red[256];
    const long long n = (long long)cout * P;
    const float scale = (float)(2.0 / (double)n) * gscale;
    pred += blockIdx.y * cpad * P;
    target += blockIdx.y * n;
    dy += blockIdx.y * cpad * P;
    double s = 0.0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < (long long)cpad * P;
         q += (long long)gridDim.x * blockDim.x) {
        float d = 0.f;
        if (q < n) {
            d = pred[q] - target[q];
            s += (double)d * (double)d;
        }
        dy[q] = __float2bfloat16_rn(q < n ? scale * d : 0.f);
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.y * gridDim.x + blockIdx.x] = red[0];
}

// the loss of sample blockIdx.x: the block sums added in block order by one
// thread, staged in shared memory
__global__ void mse_finish_kernel(const double *__restrict__ partial, int nb, long long n, double *__restrict__ out,
                                  int *__restrict__ flag)
{
    __shared__ double sp[512];
    for (int b = threadIdx.x; b < nb; b += blockDim.x) sp[b] = partial[blockIdx.x * nb + b];
    __syncthreads();
    if (threadIdx.x != 0) return;
    double s = 0.0;
    for (int b = 0; b < nb; ++b) s += sp[b];
    s /= (double)n;
    out[blockIdx.x] = s;
    if (!isfinite(s)) *flag = 1;
}

// Adam (Kingma & Ba 2015) with bias correction; refreshes the bf16 copy
__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, long long n, float lr, float b1, float b2, float eps, float c1,
                            float c2, bf16 *__restrict__ pb)
{
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const float gq = g[q];
        const float mq = b1 * m[q] + (1.f - b1) * gq;
        const float vq = b2 * v[q] + (1.f - b2) * gq * gq;
        m[q] = mq;
        v[q] = vq;
        const float pq = p[q] - lr * (mq / c1) / (sqrtf(vq / c2) + eps);
        p[q] = pq;
        pb[q] = __float2bfloat16_rn(pq);
    }
}

// Bilinear resampling [C][sh][sw] -> [C][dh][dw] with aligned corner
// samples; op 1 takes log(max(src, 1e-30)) before interpolating, op 2
// exponentiates the interpolated value.  With cmax, samples of channel c0 and
// beyond are divided by their channel's maximum cmax[c - c0] (zero: by nothing,
// giving zeros).
__global__ void resample_kernel(const float *__restrict__ src, int C, int sh, int sw, float *__restrict__ dst, int dh, int dw,
                                int op, const float *__restrict__ cmax, int c0)
{
    const float ry = dh > 1 ? (float)(sh - 1) / (float)(dh - 1) : 0.f;
    const float rx = dw > 1 ? (float)(sw - 1) / (float)(dw - 1) : 0.f;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= dw) return;
    const float x = j * rx;
    const int x0 = min((int)floorf(x), sw - 1), x1 = min(x0 + 1, sw - 1);
    const float fx = x - x0;
    for (int c = blockIdx.z; c < C; c += gridDim.z) {
        const bool scale = cmax && c >= c0;
        const float inv = scale && cmax[c - c0] > 0.f ? 1.f / cmax[c - c0] : 0.f;
        for (int i = blockIdx.y; i < dh; i += gridDim.y) {
            const float y = i * ry;
            const int y0 = min((int)floorf(y), sh - 1), y1 = min(y0 + 1, sh - 1);
            const float fy = y - y0;
            const float *s0 = src + ((long long)c * sh + y0) * sw, *s1 = src + ((long long)c * sh + y1) * sw;
            float a = s0[x0], b = s0[x1], cc = s1[x0], d = s1[x1];
            if (scale) {
                a = __fmul_rn(a, inv);
                b = __fmul_rn(b, inv);
                cc = __fmul_rn(cc, inv);
                d = __fmul_rn(d, inv);
            }
            if (op == 1) {
                a = logf(fmaxf(a, 1e-30f));
                b = logf(fmaxf(b, 1e-30f));
                cc = logf(fmaxf(cc, 1e-30f));
                d = logf(fmaxf(d, 1e-30f));
            }
            float v = (1.f - fy) * ((1.f - fx) * a + fx * b) + fy * ((1.f - fx) * cc + fx * d);
            if (op == 2) v = expf(v);
            dst[((long long)c * dh + i) * dw + j] = v;
        }
    }
}

// The mask of a point set is separable over points that share a depth:
// sum_p exp(-|x - x_p|^2 / 2 sigma^2) = sum_g (sum_{p in g} exp(-(x - x_p)^2 ..)) exp(-(z - z_g)^2 ..).
// Tables of every group g (points [begin[g], begin[g + 1]) of a, common
// coordinate bg[g]): ta[g][i] over the first axis, tb[g][j] over the second.
// An acquisition has one or two depths, so this replaces an FP64 exponential
// per node and point (5.2 ms at 1361 x 281 nodes, 365 points) by one per
// axis node and point.  L lanes (a power of two up to 32) share an axis node's
// points: a lane's exponentials form a chain (with one lane 263 us for 341 points).
__global__ void __launch_bounds__(128) mask_tables_kernel(const double *__restrict__ a, const int *__restrict__ begin,
                                                          const double *__restrict__ bg, const double *__restrict__ ca, int na,
                                                          const double *__restrict__ cb, int nb, double inv2s2, int groups, int L,
                                                          double *__restrict__ ta, double *__restrict__ tb)
{
    const int sub = threadIdx.x & (L - 1), per = blockDim.x / L;
    const int i = blockIdx.x * per + threadIdx.x / L;
    for (int g = blockIdx.y; g < groups; g += gridDim.y) {
        double s = 0.0;
        if (i < na)
            for (int p = begin[g] + sub; p < begin[g + 1]; p += L) {
                const double d = ca[i] - a[p];
                s += exp(-d * d * inv2s2);
            }
        for (int o = L >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (sub) continue;
        if (i < na) {
            ta[(long long)g * na + i] = s;
        } else if (i < na + nb) {
            const double d = cb[i - na] - bg[g];
            tb[(long long)g * nb + i - na] = exp(-d * d * inv2s2);
        }
    }
}

struct MaskSet {
    const double *ta, *tb;     // tables of mask_tables_kernel
    int groups, first_x;       // first_x: ta runs along x (grouped by depth), else along z
};

// Node-grid features: vp / 4700, vs / 2700, rho / 2500, the unnormalised
// source / receiver masks, and the masks' maxima (cmax[2], zero on entry).
__global__ void features_kernel(const float *__restrict__ rho, const float *__restrict__ vp,
                                const float *__restrict__ vs, MaskSet src, MaskSet rec, int nx, int nz,
                                float *__restrict__ out, float *__restrict__ cmax)
{
    const long long N = (long long)nx * nz;
    float mx[2] = {0.f, 0.f};
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < N; q += (long long)gridDim.x * blockDim.x) {
        const int iz = (int)(q / nx), ix = (int)(q - (long long)iz * nx);
        out[q] = vp[q] / 4700.f;
        out[N + q] = vs[q] / 2700.f;
        out[2 * N + q] = rho[q] / 2500.f;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const MaskSet &S = k == 0 ? src : rec;
            const int na = S.first_x ? nx : nz, nb = S.first_x ? nz : nx;
            const int i = S.first_x ? ix : iz, j = S.first_x ? iz : ix;
            double s = 0.0;
            for (int g = 0; g < S.groups; ++g) s += S.ta[(long long)g * na + i] * S.tb[(long long)g * nb + j];
            const float v = (float)s;
            out[(3 + k) * N + q] = v;
            mx[k] = fmaxf(mx[k], v);
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx[k] = fmaxf(mx[k], __shfl_xor_sync(0xffffffffu, mx[k], o));
        // non-negative floats order like their bit patterns
        if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<int *>(cmax + k), __float_as_int(mx[k]));
    }
}

__global__ void finite_flag_kernel(const float *__restrict__ x, long long n, int *__restrict__ flag)
{
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        if (!isfinite(x[q])) *flag = 1;
}

int grid_for(long long n, int per = 1)
{
    long long b = (n / per + 255) / 256;
    return (int)std::max<long long>(1, std::min<long long>(b, 152LL * 16));
}

}  // namespace

// ---------------------------------------------------------------------------
// network handle
// ---------------------------------------------------------------------------

namespace {

constexpr int kMaxLevels = 6;

struct UnetLayer {
    int cin, cout, k;       // logical shape
    int kcp, coutp;         // padded: kcp = round8(cin k k), coutp = round8(cout)
    long long w_off, b_off; // into the flat parameter buffers
};

long long round8(long long v) { return (v + 7) / 8 * 8; }

}  // namespace

struct gbfwi_unet {
    gbfwi_unet_desc d{};
    int ch[kMaxLevels] = {};
    std::vector<UnetLayer> layers;
    long long nparam = 0;
    long long step = 0;                 // Adam steps taken
    DevBuf p32, g32, m32, v32, pb;      // master params, grads, Adam moments, bf16 copy
    DevBuf arena;                       // holds the buffers of the samples, from xin32 to gb but for wt
    DevBuf xin32, xb, tgt32;            // input (FP32 staging, bf16), target staging
    DevBuf ea[kMaxLevels], e[kMaxLevels], pl[kMaxLevels], da[kMaxLevels], dd[kMaxLevels];
    DevBuf yout, gyb;                   // output [coutp][P0] FP32, its gradient (bf16)
    DevBuf wt;                          // transposed bf16 weights of the 3x3 layers ([tap][co][c], at w_off)
    bool wt_fresh = false;              // wt holds the current weights
    DevBuf rsum;                        // per-sample row sums of the bias gradients
    DevBuf dcat[kMaxLevels];            // gradient of the concatenated decoder input (FP32)
    DevBuf fA, fP, gb;                  // FP32 input gradients, masked bf16 gradient
    DevBuf part;                        // split-K partials
    DevBuf red, flag;                   // loss partials / result, non-finite flag
    long long part_cap = 0;
    int nb = 0;                         // samples the activation buffers hold
};

namespace {

long long npix(const gbfwi_unet *n, int l) { return (long long)(n->d.height >> l) * (n->d.width >> l); }

template <class K>
int allow_smem(K kern, size_t smem, bool (&done)[64])
{
    int dev = 0;
    GB_CUDA(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && !done[dev]) {
        GB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        done[dev] = true;
    }
    return GBFWI_OK;
}

template <int BM, bool AK, bool BK, bool GA>
int launch_gemm(const GemmArgs &g, int samples, cudaStream_t s)
{
    constexpr int BN = gemm_bn(BM);
    dim3 grid((unsigned)((g.N + BN - 1) / BN), (unsigned)((g.M + BM - 1) / BM), (unsigned)(g.splits * samples));
    using T = GemmTile<BM, BN, AK, BK>;
    constexpr size_t smem = (size_t)kStages<GA> * (T::AE + T::BE) * sizeof(bf16);
    static bool attr_done[64] = {};      // per device ordinal
    GB_TRY(allow_smem(gemm_bf16_kernel<BM, BN, AK, BK, GA>, smem, attr_done));
    gemm_bf16_kernel<BM, BN, AK, BK, GA><<<grid, GTHREADS, smem, s>>>(g);
    GB_LAUNCHED();
    return GBFWI_OK;
}

template <int BM>
int launch_gemm_bm(const GemmArgs &g, int samples, bool a_km, bool b_nk, cudaStream_t s)
{
    if (g.src.s1)
        return b_nk ? launch_gemm<BM, false, true, true>(g, samples, s) : launch_gemm<BM, false, false, true>(g, samples, s);
    if (a_km) return b_nk ? GBFWI_EINVAL : launch_gemm<BM, true, false, false>(g, samples, s);
    return b_nk ? launch_gemm<BM, false, true, false>(g, samples, s) : launch_gemm<BM, false, false, false>(g, samples, s);
}

// Sum of the split partials [sample][split][M][N] in the scratch with the GEMM's
// epilogue.  Four outputs a thread once that leaves enough threads: 16.8 us to
// 6.7 us for 32 x 262144 outputs.
int split_reduce(gbfwi_unet *net, int samples, int splits, int M, int N, long long ldc, long long cbs, const float *bias, int relu,
                 float *cf, bf16 *cb, cudaStream_t s)
{
    const bool wide = (long long)M * N >= 4LL * 152 * 1024 && N % 4 == 0 && ldc % 4 == 0 && cbs % 4 == 0 &&
                      !((uintptr_t)cf & 15) && !((uintptr_t)cb & 7) && !((uintptr_t)net->part.p & 15);
    auto kern = wide ? gemm_reduce_kernel<4> : gemm_reduce_kernel<1>;
    kern<<<dim3((unsigned)grid_for((long long)M * N, wide ? 4 : 1), (unsigned)samples), 256, 0, s>>>(
        net->part.as<float>(), splits, M, N, ldc, cbs, bias, relu, cf, cb);
    GB_LAUNCHED();
    return GBFWI_OK;
}

// C[M][N] (+)= A B (+ bias, ReLU) for `samples` samples with A = [M][K] or [K][M]
// (a_km), B = [K][N] or [N][K] (b_nk), or gathered from src (B null); FP32 output
// Cf and/or bf16 output Cb, row pitch ldc.  With accumulate one C takes the
// samples in order.
struct Operand { const bf16 *p; long long ld, bs; };

int gemm(gbfwi_unet *net, int samples, Operand A, bool a_km, Operand B, const ConvSrc *src, bool b_nk, int M, int N, int K,
         float *Cf, bf16 *Cb, const float *bias, int relu, int accumulate, long long ldc, long long cbs, cudaStream_t s)
{
    if (M < 1 || N < 1 || K < 8 || K % 8 || A.ld % 8 || N % 2 || ldc % 2 || ((uintptr_t)A.p & 15) || (a_km && M % 8) ||
        (!b_nk && N % 8))
        return GBFWI_EINVAL;
    if (!src && (B.ld % 8 || ((uintptr_t)B.p & 15))) return GBFWI_EINVAL;
    if (src && (src->W % 8 || ((uintptr_t)src->s1 & 15) || ((uintptr_t)src->s2 & 15))) return GBFWI_EINVAL;
    const int BM = gemm_bm(M);
    int splits = 1;
    const int kchunk = split_chunk(M, N, K, net->part_cap, &splits);
    // samples whose partials fit the scratch together (a wide layer's gradient alone is
    // larger than it: one sample after another then, each added to the output)
    const int fit = gemm_samples((long long)M * N, splits, samples, accumulate, net->part_cap);
    for (int b0 = 0; b0 < samples; b0 += fit) {
        const int nb = std::min(fit, samples - b0);
        const bool partial = gemm_partial(splits, nb, accumulate);
        GemmArgs g{};
        g.A = A.p + b0 * A.bs; g.lda = A.ld; g.abs_ = A.bs;
        if (src) {
            g.src = *src;
            g.src.s1 += b0 * src->bs1;
            if (g.src.s2) g.src.s2 += b0 * src->bs2;
        } else {
            g.B = B.p + b0 * B.bs; g.ldb = B.ld; g.bbs = B.bs;
        }
        g.M = M; g.N = N; g.K = K; g.kchunk = kchunk; g.splits = splits;
        float *cf = Cf ? Cf + (accumulate ? 0 : b0 * cbs) : nullptr;
        bf16 *cb = Cb ? Cb + b0 * cbs : nullptr;
        if (partial) {
            g.Cf = net->part.as<float>();
            g.ldc = N;
            g.split_stride = (long long)M * N;
            g.partial = 1;
        } else {
            g.Cf = cf; g.Cb = cb; g.bias = bias; g.relu = relu; g.accumulate = accumulate; g.ldc = ldc; g.cbs = cbs;
        }
        GB_TRY(BM == 32 ? launch_gemm_bm<32>(g, nb, a_km, b_nk, s)
                        : (BM == 64 ? launch_gemm_bm<64>(g, nb, a_km, b_nk, s) : launch_gemm_bm<128>(g, nb, a_km, b_nk, s)));
        if (partial) {
            if (accumulate) {
                const long long outs = (long long)M * N;
                if (outs < 65536)
                    grad_reduce_kernel<<<(unsigned)((outs + 31) / 32), 32 * std::min(8, nb), 0, s>>>(net->part.as<float>(), nb, splits, M, N, ldc, cf);
                else
                    grad_rows_kernel<<<grid_for(outs), 256, 0, s>>>(net->part.as<float>(), nb, splits, M, N, ldc, cf);
                GB_LAUNCHED();
                continue;
            }
            GB_TRY(split_reduce(net, nb, splits, M, N, ldc, cbs, bias, relu, cf, cb, s));
        }
    }
    return GBFWI_OK;
}

template <int BM>
int launch_dx(const GemmArgs &g, int samples, cudaStream_t s)
{
    constexpr int BN = gemm_bn(BM);
    using T = GemmTile<BM, BN, true, false>;
    constexpr size_t smem = (size_t)GSTAGES * (T::AE + T::BE) * sizeof(bf16);
    static bool attr_done[64] = {};
    GB_TRY(allow_smem(conv_dx_kernel<BM, BN>, smem, attr_done));
    conv_dx_kernel<BM, BN><<<dim3((unsigned)((g.N + BN - 1) / BN), (unsigned)((g.M + BM - 1) / BM),
                                  (unsigned)(g.partial ? 9 * samples : samples)), GTHREADS, smem, s>>>(g);
    GB_LAUNCHED();
    return GBFWI_OK;
}

// 3x3 convolution + bias + ReLU -> bf16 output [sample][cout][H][W]
int conv_fwd(gbfwi_unet *n, int nb, const UnetLayer &L, const ConvSrc &src, bf16 *out, cudaStream_t s)
{
    const long long P = (long long)src.H * src.W;
    return gemm(n, nb, {n->pb.as<bf16>() + L.w_off, L.kcp, 0}, false, {}, &src, false, L.cout, (int)P, L.kcp, nullptr, out,
                n->p32.as<float>() + L.b_off, 1, 0, P, L.cout * P, s);
}

int bias_grad(gbfwi_unet *n, int nb, const bf16 *G, long long P, int rows, float *db, cudaStream_t s)
{
    rowsum_kernel<<<dim3((unsigned)rows, (unsigned)nb), 256, 0, s>>>(G, P, rows, n->rsum.as<float>(), nb == 1 ? db : nullptr);
    GB_LAUNCHED();
    if (nb == 1) return GBFWI_OK;
    rowsum_add_kernel<<<(rows + 127) / 128, 128, 0, s>>>(n->rsum.as<float>(), nb, rows, db);
    GB_LAUNCHED();
    return GBFWI_OK;
}

// Backward of a 3x3 convolution given its masked output gradient G
// (bf16 [sample][cout][P]): dW, db accumulate into the gradient buffer; when dX is
// not null, the input gradient (FP32 [sample][cin][P]) is written there.
int conv_bwd(gbfwi_unet *n, int nb, const UnetLayer &L, const ConvSrc &src, const bf16 *G, float *dX, cudaStream_t s)
{
    const long long P = (long long)src.H * src.W;
    GB_TRY(gemm(n, nb, {G, P, L.cout * P}, false, {}, &src, true, L.cout, L.kcp, (int)P, n->g32.as<float>() + L.w_off, nullptr,
                nullptr, 0, 1, L.kcp, 0, s));
    GB_TRY(bias_grad(n, nb, G, P, L.cout, n->g32.as<float>() + L.b_off, s));
    if (!dX) return GBFWI_OK;
    GemmArgs g{};
    g.A = n->wt.as<bf16>() + L.w_off;
    g.lda = L.cin;
    g.M = L.cin; g.N = (int)P; g.K = L.coutp;
    int splits = 1;
    // the parts the taps' sums are cut into: the split rule of a (9 cin x P) product
    g.kchunk = split_chunk(L.kcp, (int)P, L.coutp, n->part_cap, &splits);
    g.Cf = dX; g.ldc = P; g.cbs = L.cin * P;
    g.src = ConvSrc{G, G, L.cout, 0, 0, src.H, src.W, L.cout * P, 0};
    const int BM = gemm_bm(L.cin);
    // a CTA per tap while the tiles alone leave most SMs idle (48 tiles: 38 us, 27 us
    // with the sum; 128 tiles: 21 us, 36 us with it)
    const long long tiles = (P + gemm_bn(BM) - 1) / gemm_bn(BM) * ((L.cin + BM - 1) / BM) * nb, taps = 9LL * nb * L.cin * P;
    if (tiles < 64 && taps <= n->part_cap) {
        g.partial = 1;
        g.Cf = n->part.as<float>();
        g.split_stride = L.cin * P;
    }
    GB_TRY(BM == 32 ? launch_dx<32>(g, nb, s) : (BM == 64 ? launch_dx<64>(g, nb, s) : launch_dx<128>(g, nb, s)));
    return g.partial ? split_reduce(n, nb, 9, L.cin, (int)P, P, L.cin * P, nullptr, 0, dX, nullptr, s) : GBFWI_OK;
}

int grad_mask(int nb, const float *fine, long long fine_bs, const float *coarse, const float *direct, long long direct_bs,
              const bf16 *y, int C, int H, int W, bf16 *out, cudaStream_t s)
{
    grad_mask_kernel<<<dim3((unsigned)grid_for((long long)C * H * W), (unsigned)nb), 256, 0, s>>>(
        fine, fine_bs, coarse, direct, direct_bs, y, C, H, W, out);
    GB_LAUNCHED();
    return GBFWI_OK;
}

// transposed weights for the input gradients, after the weights changed
int refresh_wt(gbfwi_unet *n, cudaStream_t s)
{
    if (n->wt_fresh) return GBFWI_OK;
    static_assert(4 * kMaxLevels <= (int)(sizeof(WtTable) / sizeof(WtLayer)), "3x3 layers");
    WtTable tab{};
    int layers = 0;
    long long most = 1;
    for (const UnetLayer &L : n->layers) {
        if (L.k != 3) continue;
        tab.l[layers++] = WtLayer{L.w_off, L.cout, L.cin, L.kcp};
        most = std::max(most, 9LL * L.cout * L.cin);
    }
    if (layers > 0) {
        transpose_weights_kernel<<<dim3((unsigned)std::min(grid_for(most), 304), (unsigned)layers), 256, 0, s>>>(n->pb.as<bf16>(), tab,
                                                                                                 n->wt.as<bf16>());
        GB_LAUNCHED();
    }
    n->wt_fresh = true;
    return GBFWI_OK;
}

// plain source: one map, nothing upsampled or concatenated
ConvSrc plain(const bf16 *x, int C, int H, int W)
{
    return ConvSrc{x, x, C, 0, 0, H, W, (long long)C * H * W, 0};
}

// decoder input of level l: the level below upsampled, then the skip connection
ConvSrc decoder_src(const gbfwi_unet *n, int l, const bf16 *below)
{
    const int H = n->d.height >> l, W = n->d.width >> l;
    return ConvSrc{below, n->e[l].as<bf16>(), n->ch[l + 1], 1, n->ch[l], H, W, (long long)n->ch[l + 1] * (H / 2) * (W / 2),
                   (long long)n->ch[l] * H * W};
}

// forward pass of nb samples on n->xb (bf16 input already staged) -> n->yout
int net_forward(gbfwi_unet *n, int nb, cudaStream_t s)
{
    const int Lv = n->d.levels;
    int li = 0;
    for (int l = 0; l < Lv; ++l) {
        const int H = n->d.height >> l, W = n->d.width >> l;
        const bf16 *in = n->xb.as<bf16>();
        int cin = n->d.cin;
        if (l > 0) {
            cin = n->ch[l - 1];
            avgpool_kernel<<<grid_for((long long)nb * cin * H * W), 256, 0, s>>>(n->e[l - 1].as<bf16>(), nb * cin, H, W,
                                                                                n->pl[l].as<bf16>());
            GB_LAUNCHED();
            in = n->pl[l].as<bf16>();
        }
        GB_TRY(conv_fwd(n, nb, n->layers[li++], plain(in, cin, H, W), n->ea[l].as<bf16>(), s));
        GB_TRY(conv_fwd(n, nb, n->layers[li++], plain(n->ea[l].as<bf16>(), n->ch[l], H, W), n->e[l].as<bf16>(), s));
    }
    const bf16 *h = n->e[Lv - 1].as<bf16>();
    for (int l = Lv - 2; l >= 0; --l) {
        const int H = n->d.height >> l, W = n->d.width >> l;
        GB_TRY(conv_fwd(n, nb, n->layers[li++], decoder_src(n, l, h), n->da[l].as<bf16>(), s));
        GB_TRY(conv_fwd(n, nb, n->layers[li++], plain(n->da[l].as<bf16>(), n->ch[l], H, W), n->dd[l].as<bf16>(), s));
        h = n->dd[l].as<bf16>();
    }
    const UnetLayer &O = n->layers[li];
    const long long P0 = npix(n, 0);
    return gemm(n, nb, {n->pb.as<bf16>() + O.w_off, O.kcp, 0}, false, {h, P0, n->ch[0] * P0}, nullptr, false, O.coutp, (int)P0,
                O.kcp, n->yout.as<float>(), nullptr, n->p32.as<float>() + O.b_off, 0, 0, P0, O.coutp * P0, s);
}

// backward pass of nb samples from the output gradient n->gyb (bf16
// [sample][coutp][P0]); parameter gradients accumulate into n->g32
int net_backward(gbfwi_unet *n, int nb, cudaStream_t s)
{
    const int Lv = n->d.levels;
    const long long P0 = npix(n, 0);
    int li = (int)n->layers.size() - 1;
    const UnetLayer &O = n->layers[li];
    const bf16 *top = Lv > 1 ? n->dd[0].as<bf16>() : n->e[0].as<bf16>();
    GB_TRY(refresh_wt(n, s));
    // output 1x1 convolution
    GB_TRY(gemm(n, nb, {n->gyb.as<bf16>(), P0, O.coutp * P0}, false, {top, P0, n->ch[0] * P0}, nullptr, true, O.coutp, O.kcp,
                (int)P0, n->g32.as<float>() + O.w_off, nullptr, nullptr, 0, 1, O.kcp, 0, s));
    GB_TRY(bias_grad(n, nb, n->gyb.as<bf16>(), P0, O.coutp, n->g32.as<float>() + O.b_off, s));
    GB_TRY(gemm(n, nb, {n->pb.as<bf16>() + O.w_off, O.kcp, 0}, true, {n->gyb.as<bf16>(), P0, O.coutp * P0}, nullptr, false, O.kcp,
                (int)P0, O.coutp, n->fA.as<float>(), nullptr, nullptr, 0, 0, P0, O.kcp * P0, s));
    --li;
    float *fA = n->fA.as<float>();
    bf16 *gb = n->gb.as<bf16>();
    auto wide = [&](int l) { return (long long)(n->ch[l + 1] + n->ch[l]) * npix(n, l); };   // dcat elements per sample
    // decoder, fine to coarse; the gradient of level l's output arrives as
    // fA (level 0) or as the upsampling adjoint of dcat[l-1]
    for (int l = 0; l <= Lv - 2; ++l) {
        const int H = n->d.height >> l, W = n->d.width >> l;
        const long long own = n->ch[l] * npix(n, l);
        const float *fine = l > 0 ? n->dcat[l - 1].as<float>() : nullptr;
        const float *direct = l == 0 ? fA : nullptr;
        GB_TRY(grad_mask(nb, fine, l > 0 ? wide(l - 1) : 0, nullptr, direct, own, n->dd[l].as<bf16>(), n->ch[l], H, W, gb, s));
        GB_TRY(conv_bwd(n, nb, n->layers[li], plain(n->da[l].as<bf16>(), n->ch[l], H, W), gb, fA, s));
        --li;
        GB_TRY(grad_mask(nb, nullptr, 0, nullptr, fA, own, n->da[l].as<bf16>(), n->ch[l], H, W, gb, s));
        const bf16 *coarse = (l + 1 <= Lv - 2) ? n->dd[l + 1].as<bf16>() : n->e[Lv - 1].as<bf16>();
        GB_TRY(conv_bwd(n, nb, n->layers[li], decoder_src(n, l, coarse), gb, n->dcat[l].as<float>(), s));
        --li;
    }
    // encoder, bottleneck first; the gradient of e[l] sums the decoder's
    // upsampling adjoint (bottleneck), the pooling adjoint of the level
    // below and the skip connection
    for (int l = Lv - 1; l >= 0; --l) {
        const int H = n->d.height >> l, W = n->d.width >> l;
        const long long P = (long long)H * W, own = n->ch[l] * P;
        const float *fine = nullptr, *coarse = nullptr, *direct = nullptr;
        long long fine_bs = 0, direct_bs = own;
        if (l == Lv - 1) {
            if (Lv > 1) {
                fine = n->dcat[Lv - 2].as<float>();
                fine_bs = wide(Lv - 2);
            } else {
                direct = fA;
            }
        } else {
            coarse = n->fP.as<float>();
            direct = n->dcat[l].as<float>() + (long long)n->ch[l + 1] * P;
            direct_bs = wide(l);
        }
        GB_TRY(grad_mask(nb, fine, fine_bs, coarse, direct, direct_bs, n->e[l].as<bf16>(), n->ch[l], H, W, gb, s));
        GB_TRY(conv_bwd(n, nb, n->layers[li], plain(n->ea[l].as<bf16>(), n->ch[l], H, W), gb, fA, s));
        --li;
        GB_TRY(grad_mask(nb, nullptr, 0, nullptr, fA, own, n->ea[l].as<bf16>(), n->ch[l], H, W, gb, s));
        const bf16 *in = l == 0 ? n->xb.as<bf16>() : n->pl[l].as<bf16>();
        const int cin = l == 0 ? n->d.cin : n->ch[l - 1];
        GB_TRY(conv_bwd(n, nb, n->layers[li], plain(in, cin, H, W), gb, l > 0 ? n->fP.as<float>() : nullptr, s));
        --li;
    }
    return GBFWI_OK;
}

int stage_input(gbfwi_unet *n, int nb, const float *x, cudaStream_t s)
{
    const long long cnt = (long long)nb * n->d.cin * npix(n, 0);
    const float *src = x;
    if (!gb_is_device_ptr(x)) {
        GB_CUDA(cudaMemcpyAsync(n->xin32.p, x, cnt * sizeof(float), cudaMemcpyHostToDevice, s));
        src = n->xin32.as<float>();
    }
    to_bf16_kernel<<<grid_for(cnt), 256, 0, s>>>(src, cnt, n->xb.as<bf16>());
    GB_LAUNCHED();
    return GBFWI_OK;
}

// Activation and gradient buffers for nb samples, pieces of one allocation.  The larger
// one is made beside the one that is there and takes its place, so a failure
// leaves the network with what it had (one sample's from its creation on).
int reserve(gbfwi_unet *n, int nb)
{
    if (nb <= n->nb) return GBFWI_OK;
    const int Lv = n->d.levels;
    const long long P0 = npix(n, 0);
    const UnetLayer &O = n->layers.back();
    std::vector<std::pair<DevBuf *, size_t>> list;
    size_t total = 0;
    auto need = [&](DevBuf &b, long long bytes) {
        list.push_back({&b, (size_t)(bytes * nb + 255) / 256 * 256});
        total += list.back().second;
    };
    const size_t F = sizeof(float), B2 = sizeof(bf16);
    need(n->xin32, (long long)n->d.cin * P0 * F);
    need(n->xb, (long long)n->d.cin * P0 * B2);
    need(n->tgt32, (long long)n->d.cout * P0 * F);
    need(n->yout, (long long)O.coutp * P0 * F);
    need(n->gyb, (long long)O.coutp * P0 * B2);
    long long cmax = (long long)O.coutp * P0;
    for (int l = 0; l < Lv; ++l) {
        const long long P = npix(n, l);
        cmax = std::max(cmax, n->ch[l] * P);
        need(n->ea[l], n->ch[l] * P * B2);
        need(n->e[l], n->ch[l] * P * B2);
        if (l > 0) need(n->pl[l], n->ch[l - 1] * P * B2);
        if (l <= Lv - 2) {
            need(n->da[l], n->ch[l] * P * B2);
            need(n->dd[l], n->ch[l] * P * B2);
            need(n->dcat[l], (long long)(n->ch[l + 1] + n->ch[l]) * P * F);
        }
    }
    need(n->fA, cmax * F);
    need(n->fP, cmax * F);
    need(n->gb, cmax * B2);
    need(n->rsum, (long long)std::max(n->ch[Lv - 1], O.coutp) * F);
    DevBuf fresh;
    GB_TRY(fresh.ensure(total));
    std::swap(n->arena.p, fresh.p);
    std::swap(n->arena.bytes, fresh.bytes);
    size_t at = 0;
    for (const auto &piece : list) {
        piece.first->lend(n->arena.as<char>() + at, piece.second);
        at += piece.second;
    }
    n->nb = nb;
    return GBFWI_OK;
}

// samples a training step takes at once: their buffers stay near 2 GiB
int batch_group(const gbfwi_unet *n, int batch)
{
    long long per = 0;                  // bytes of one sample, the gradients included
    for (int l = 0; l < n->d.levels; ++l) per += npix(n, l) * n->ch[l] * (5 * 2 + 4 + 3 * 4);
    per += npix(n, 0) * (n->ch[0] * 10 + 64);
    return (int)std::max<long long>(1, std::min<long long>(batch, (2LL << 30) / std::max<long long>(per, 1)));
}

int read_flag(gbfwi_unet *n, cudaStream_t s, int *out)
{
    GB_CUDA(cudaMemcpyAsync(out, n->flag.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    return GBFWI_OK;
}

}  // namespace

// ---------------------------------------------------------------------------
// ABI
// ---------------------------------------------------------------------------

extern "C" int gbfwi_unet_create(const gbfwi_unet_desc *d, gbfwi_unet **out)
{
    if (!d || !out || d->levels < 1 || d->levels > kMaxLevels || d->base < 8 || d->base % 8 || d->cin < 1 ||
        d->cout < 1 || d->height < 1 || d->width < 1)
        return GBFWI_EINVAL;
    const int f = 1 << (d->levels - 1);
    if (d->height % f || d->width % (8 * f)) return GBFWI_EINVAL;
    gbfwi_unet *n = new (std::nothrow) gbfwi_unet();
    if (!n) return GBFWI_ENOMEM;
    n->d = *d;
    const int Lv = d->levels;
    for (int l = 0; l < Lv; ++l) n->ch[l] = d->base << l;
    auto add = [&](int cin, int cout, int k) {
        UnetLayer L{cin, cout, k, (int)round8((long long)cin * k * k), (int)round8(cout), 0, 0};
        L.w_off = n->nparam;
        L.b_off = L.w_off + (long long)L.coutp * L.kcp;
        n->nparam = round8(L.b_off + L.coutp);
        n->layers.push_back(L);
    };
    for (int l = 0; l < Lv; ++l) {
        add(l == 0 ? d->cin : n->ch[l - 1], n->ch[l], 3);
        add(n->ch[l], n->ch[l], 3);
    }
    for (int l = Lv - 2; l >= 0; --l) {
        add(n->ch[l + 1] + n->ch[l], n->ch[l], 3);
        add(n->ch[l], n->ch[l], 3);
    }
    add(n->ch[0], d->cout, 1);
    n->part_cap = 32LL << 20;   // floats of split-K partials
    int rc = GBFWI_OK;
    auto need = [&](DevBuf &b, long long bytes) {
        if (!rc) rc = b.ensure((size_t)std::max<long long>(bytes, 16));
    };
    const size_t F = sizeof(float), B2 = sizeof(bf16);
    need(n->p32, n->nparam * F);
    need(n->g32, n->nparam * F);
    need(n->m32, n->nparam * F);
    need(n->v32, n->nparam * F);
    need(n->pb, n->nparam * B2);
    need(n->part, n->part_cap * F);
    need(n->red, (1024 + 512 * 64) * sizeof(double));
    need(n->flag, 16);
    need(n->wt, n->nparam * B2);
    if (!rc) rc = reserve(n, 1);
    if (rc) {
        delete n;
        return rc;
    }
    cudaMemset(n->p32.p, 0, n->nparam * F);
    cudaMemset(n->pb.p, 0, n->nparam * B2);
    cudaMemset(n->m32.p, 0, n->nparam * F);
    cudaMemset(n->v32.p, 0, n->nparam * F);
    if (cudaDeviceSynchronize() != cudaSuccess) {
        gb_set_last_cuda_error(cudaGetLastError(), "unet init", __FILE__, __LINE__);
        delete n;
        return GBFWI_ECUDA;
    }
    *out = n;
    return GBFWI_OK;
}

extern "C" int gbfwi_unet_destroy(gbfwi_unet *n)
{
    delete n;
    return GBFWI_OK;
}

extern "C" long long gbfwi_unet_num_params(const gbfwi_unet *n) { return n ? n->nparam : GBFWI_EINVAL; }

extern "C" int gbfwi_unet_layer_info(const gbfwi_unet *n, int layer, int *info)
{
    if (!n) return GBFWI_EINVAL;
    if (layer < 0) return (int)n->layers.size();
    if (layer >= (int)n->layers.size() || !info) return GBFWI_EINVAL;
    const UnetLayer &L = n->layers[layer];
    info[0] = L.cout;
    info[1] = L.cin;
    info[2] = L.k;
    info[3] = L.coutp;
    info[4] = L.kcp;
    info[5] = (int)L.w_off;
    info[6] = (int)L.b_off;
    return GBFWI_OK;
}

extern "C" int gbfwi_unet_set_params(gbfwi_unet *n, const float *params, void *stream)
{
    if (!n || !params) return GBFWI_EINVAL;
    GB_TRY(gb_check_local(params));
    cudaStream_t s = (cudaStream_t)stream;
    GB_CUDA(cudaMemcpyAsync(n->p32.p, params, n->nparam * sizeof(float),
                            gb_is_device_ptr(params) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
    to_bf16_kernel<<<grid_for(n->nparam), 256, 0, s>>>(n->p32.as<float>(), n->nparam, n->pb.as<bf16>());
    GB_LAUNCHED();
    GB_CUDA(cudaMemsetAsync(n->m32.p, 0, n->nparam * sizeof(float), s));
    GB_CUDA(cudaMemsetAsync(n->v32.p, 0, n->nparam * sizeof(float), s));
    n->step = 0;
    n->wt_fresh = false;
    GB_CUDA(cudaStreamSynchronize(s));
    return GBFWI_OK;
}

extern "C" int gbfwi_unet_get_params(const gbfwi_unet *n, float *params, void *stream)
{
    if (!n || !params) return GBFWI_EINVAL;
    GB_TRY(gb_check_local(params));
    cudaStream_t s = (cudaStream_t)stream;
    GB_CUDA(cudaMemcpyAsync(params, n->p32.p, n->nparam * sizeof(float),
                            gb_is_device_ptr(params) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    return GBFWI_OK;
}

extern "C" int gbfwi_unet_forward(gbfwi_unet *n, const float *x, float *y, void *stream)
{
    if (!n || !x || !y) return GBFWI_EINVAL;
    GB_TRY(gb_check_local(x, y));
    cudaStream_t s = (cudaStream_t)stream;
    const long long P0 = npix(n, 0);
    GB_TRY(stage_input(n, 1, x, s));
    GB_TRY(net_forward(n, 1, s));
    const long long cnt = (long long)n->d.cout * P0;
    GB_CUDA(cudaMemsetAsync(n->flag.p, 0, sizeof(int), s));
    finite_flag_kernel<<<grid_for(cnt), 256, 0, s>>>(n->yout.as<float>(), cnt, n->flag.as<int>());
    GB_LAUNCHED();
    GB_CUDA(cudaMemcpyAsync(y, n->yout.p, cnt * sizeof(float),
                            gb_is_device_ptr(y) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
    int f = 0;
    GB_TRY(read_flag(n, s, &f));
    return f ? gb_nonfinite("U-Net output") : GBFWI_OK;
}

extern "C" int gbfwi_unet_gradient(gbfwi_unet *n, const float *x, const float *dy, float *grad, void *stream)
{
    if (!n || !x || !dy || !grad) return GBFWI_EINVAL;
    GB_TRY(gb_check_local(x, dy, grad));
    cudaStream_t s = (cudaStream_t)stream;
    const long long P0 = npix(n, 0);
    const UnetLayer &O = n->layers.back();
    GB_TRY(stage_input(n, 1, x, s));
    GB_TRY(net_forward(n, 1, s));
    // dy [cout][P0] -> bf16 rows of the padded output gradient
    const long long cnt = (long long)n->d.cout * P0;
    const float *dys = dy;
    if (!gb_is_device_ptr(dy)) {
        GB_CUDA(cudaMemcpyAsync(n->tgt32.p, dy, cnt * sizeof(float), cudaMemcpyHostToDevice, s));
        dys = n->tgt32.as<float>();
    }
    GB_CUDA(cudaMemsetAsync(n->gyb.p, 0, (size_t)O.coutp * P0 * sizeof(bf16), s));
    to_bf16_kernel<<<grid_for(cnt), 256, 0, s>>>(dys, cnt, n->gyb.as<bf16>());
    GB_LAUNCHED();
    GB_CUDA(cudaMemsetAsync(n->g32.p, 0, n->nparam * sizeof(float), s));
    GB_TRY(net_backward(n, 1, s));
    GB_CUDA(cudaMemcpyAsync(grad, n->g32.p, n->nparam * sizeof(float),
                            gb_is_device_ptr(grad) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    return GBFWI_OK;
}

extern "C" int gbfwi_unet_train_step(gbfwi_unet *n, const float *x, const float *target, int batch, double lr,
                                     double *loss, void *stream)
{
    if (!n || !x || !target || batch < 1 || !(lr > 0)) return GBFWI_EINVAL;
    GB_TRY(gb_check_local(x, target));
    cudaStream_t s = (cudaStream_t)stream;
    const long long P0 = npix(n, 0);
    const UnetLayer &O = n->layers.back();
    const long long xin = (long long)n->d.cin * P0, tin = (long long)n->d.cout * P0;
    const bool dt = gb_is_device_ptr(target);
    GB_CUDA(cudaMemsetAsync(n->g32.p, 0, n->nparam * sizeof(float), s));
    GB_CUDA(cudaMemsetAsync(n->flag.p, 0, sizeof(int), s));
    if (batch > 1024) return GBFWI_EINVAL;
    // (blocks beyond the outputs would add zeros)
    const int nblk = (int)std::min<long long>(512, (O.coutp * P0 + 255) / 256);
    int group = std::min(batch_group(n, batch), 64);
    double *lsum = n->red.as<double>();   // per-sample losses [batch] (<= 1024)
    double *partial = lsum + 1024;        // [group][nblk]
    int rc = reserve(n, group);
    for (; rc == GBFWI_ENOMEM && group > 1; rc = reserve(n, group)) group = (group + 1) / 2;
    GB_TRY(rc);
    for (int b = 0; b < batch; b += group) {
        const int nb = std::min(group, batch - b);
        GB_TRY(stage_input(n, nb, x + b * xin, s));
        GB_TRY(net_forward(n, nb, s));
        const float *tb = target + b * tin;
        if (!dt) {
            GB_CUDA(cudaMemcpyAsync(n->tgt32.p, tb, nb * tin * sizeof(float), cudaMemcpyHostToDevice, s));
            tb = n->tgt32.as<float>();
        }
        mse_kernel<<<dim3((unsigned)nblk, (unsigned)nb), 256, 0, s>>>(n->yout.as<float>(), tb, n->d.cout, O.coutp, P0,
                                                                     1.f / (float)batch, partial, n->gyb.as<bf16>());
        GB_LAUNCHED();
        mse_finish_kernel<<<nb, 128, 0, s>>>(partial, nblk, tin, lsum + b, n->flag.as<int>());
        GB_LAUNCHED();
        GB_TRY(net_backward(n, nb, s));
    }
    n->wt_fresh = false;                  // the Adam step below changes the weights
    n->step += 1;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = 1.f - powf(b1, (float)n->step), c2 = 1.f - powf(b2, (float)n->step);
    adam_kernel<<<grid_for(n->nparam), 256, 0, s>>>(n->p32.as<float>(), n->g32.as<float>(), n->m32.as<float>(),
                                                     n->v32.as<float>(), n->nparam, (float)lr, b1, b2, eps, c1, c2,
                                                     n->pb.as<bf16>());
    GB_LAUNCHED();
    std::vector<double> lh(batch);
    GB_CUDA(cudaMemcpyAsync(lh.data(), lsum, batch * sizeof(double), cudaMemcpyDeviceToHost, s));
    int f = 0;
    GB_TRY(read_flag(n, s, &f));
    if (f) return gb_nonfinite("U-Net training loss");
    double tot = 0.0;
    for (double v : lh) tot += v;
    if (loss) *loss = tot / batch;
    return GBFWI_OK;
}

namespace {
int launch_resample(const float *src, int channels, int sh, int sw, float *dst, int dh, int dw, int op, const float *cmax,
                    int c0, cudaStream_t s)
{
    resample_kernel<<<dim3((unsigned)((dw + 255) / 256), (unsigned)std::min(dh, 65535), (unsigned)std::min(channels, 65535)),
                      256, 0, s>>>(src, channels, sh, sw, dst, dh, dw, op, cmax, c0);
    GB_LAUNCHED();
    return GBFWI_OK;
}
}  // namespace

extern "C" int gbfwi_resample(const float *src, int channels, int sh, int sw, float *dst, int dh, int dw, int op,
                              void *stream)
{
    if (!src || !dst || channels < 1 || sh < 1 || sw < 1 || dh < 1 || dw < 1 || op < 0 || op > 2 ||
        !gb_is_device_ptr(src) || !gb_is_device_ptr(dst))
        return GBFWI_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    return launch_resample(src, channels, sh, sw, dst, dh, dw, op, nullptr, 0, s);
}

extern "C" int gbfwi_unet_features(gbfwi_mesh *m, const float *rho, const float *vp, const float *vs, double sigma_m,
                                   int height, int width, float *x, void *stream)
{
    if (!m || !rho || !vp || !vs || !x || !(sigma_m > 0) || height < 1 || width < 1) return GBFWI_EINVAL;
    GB_TRY(gb_check_local(rho, vp, vs, x));
    cudaStream_t s = (cudaStream_t)stream;
    const int nx = m->nx, nz = m->nz;
    const long long N = (long long)nx * nz;
    const double inv2s2 = 1.0 / (2.0 * sigma_m * sigma_m);
    // the points of each set grouped by the coordinate with fewer distinct values
    struct Points {
        std::vector<double> a, bg;     // first coordinate of every point, group by group; the groups' common coordinate
        std::vector<int> begin;
        bool first_x = true;
    } set[2];
    for (int k = 0; k < 2; ++k) {
        const int np = k == 0 ? (int)m->src.size() : m->nrec;
        auto px = [&](int i) { return k == 0 ? m->src[i].x : m->rec_xz[2 * i]; };
        auto pz = [&](int i) { return k == 0 ? m->src[i].z : m->rec_xz[2 * i + 1]; };
        std::vector<double> vx(np), vz(np);
        for (int i = 0; i < np; ++i) { vx[i] = px(i); vz[i] = pz(i); }
        auto distinct = [](std::vector<double> v) {
            std::sort(v.begin(), v.end());
            return (size_t)(std::unique(v.begin(), v.end()) - v.begin());
        };
        Points &P = set[k];
        P.first_x = distinct(vz) <= distinct(vx);
        std::vector<int> order(np);
        for (int i = 0; i < np; ++i) order[i] = i;
        const std::vector<double> &first = P.first_x ? vx : vz, &common = P.first_x ? vz : vx;
        std::stable_sort(order.begin(), order.end(), [&](int p, int q) { return common[p] < common[q]; });
        for (int i : order) {
            if (P.bg.empty() || P.bg.back() != common[i]) {
                P.begin.push_back((int)P.a.size());
                P.bg.push_back(common[i]);
            }
            P.a.push_back(first[i]);
        }
        P.begin.push_back((int)P.a.size());
    }
    // one upload: axes, then per set the points, the groups and their bounds
    std::vector<double> tab = gb_axis(m, m->d.nex);
    const std::vector<double> cz = gb_axis(m, m->d.nez);
    tab.insert(tab.end(), cz.begin(), cz.end());
    size_t at_a[2], at_b[2], at_n[2], tables = 0;
    for (int k = 0; k < 2; ++k) {
        const Points &P = set[k];
        at_a[k] = tab.size();
        tab.insert(tab.end(), P.a.begin(), P.a.end());
        at_b[k] = tab.size();
        tab.insert(tab.end(), P.bg.begin(), P.bg.end());
        at_n[k] = tab.size();
        tab.resize(tab.size() + (P.begin.size() + 1) / 2);
        std::memcpy(&tab[at_n[k]], P.begin.data(), P.begin.size() * sizeof(int));
        tables += P.bg.size() * (size_t)(nx + nz);
    }
    const long long cnt = 5LL * height * width;
    const bool devx = gb_is_device_ptr(x);
    const bool devm = gb_is_device_ptr(rho) && gb_is_device_ptr(vp) && gb_is_device_ptr(vs);
    const size_t nd = tab.size() + tables;
    GB_TRY(m->w_feat.ensure(nd * sizeof(double) + ((size_t)5 * N + 8 + (devm ? 0 : 3 * N) + (devx ? 0 : cnt)) * sizeof(float)));
    double *dt = m->w_feat.as<double>(), *dtab = dt + tab.size();
    float *feat = reinterpret_cast<float *>(dt + nd), *cmax = feat + 5 * N;
    GB_CUDA(cudaMemcpyAsync(dt, tab.data(), tab.size() * sizeof(double), cudaMemcpyHostToDevice, s));
    GB_CUDA(cudaMemsetAsync(cmax, 0, 2 * sizeof(float), s));
    const float *mod[3] = {rho, vp, vs};
    float *dm = cmax + 8;
    if (!devm)
        for (int k = 0; k < 3; ++k) {
            GB_CUDA(cudaMemcpyAsync(dm + k * N, mod[k], N * sizeof(float), cudaMemcpyDefault, s));
            mod[k] = dm + k * N;
        }
    MaskSet ms[2];
    for (int k = 0; k < 2; ++k) {
        const Points &P = set[k];
        const int G = (int)P.bg.size(), na = P.first_x ? nx : nz, nb = P.first_x ? nz : nx;
        ms[k] = MaskSet{dtab, dtab + (size_t)G * na, G, P.first_x};
        dtab += (size_t)G * (na + nb);
        if (G > 0) {
            int L = 1;                                       // lanes an axis node: the mean points a group, at most a warp
            while (L < 32 && 2LL * L * G <= (long long)P.a.size()) L *= 2;
            const unsigned gx = (unsigned)(((long long)(na + nb) * L + 127) / 128);
            mask_tables_kernel<<<dim3(gx, (unsigned)std::min(G, 65535)), 128, 0, s>>>(
                dt + at_a[k], reinterpret_cast<const int *>(dt + at_n[k]), dt + at_b[k], P.first_x ? dt : dt + nx, na,
                P.first_x ? dt + nx : dt, nb, inv2s2, G, L, const_cast<double *>(ms[k].ta), const_cast<double *>(ms[k].tb));
            GB_LAUNCHED();
        }
    }
    features_kernel<<<grid_for(N), 256, 0, s>>>(mod[0], mod[1], mod[2], ms[0], ms[1], nx, nz, feat, cmax);
    GB_LAUNCHED();
    float *dst = devx ? x : dm + (devm ? 0 : 3 * N);
    GB_TRY(launch_resample(feat, 5, nz, nx, dst, height, width, 0, cmax, 3, s));
    if (!devx) GB_CUDA(cudaMemcpyAsync(x, dst, cnt * sizeof(float), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    return GBFWI_OK;
}
