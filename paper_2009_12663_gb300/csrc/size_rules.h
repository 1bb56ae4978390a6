// Sizes of scratch that one piece of host code reserves and another fills, as
// plain C++ without CUDA types: both sides call the same function, and the rules
// can be checked on a machine without a GPU.
#pragma once

#include <algorithm>
#include <cstddef>

namespace sizes {

// shots of the last of the batches that take `nshot` shots `most` at a time
inline int last_batch(int nshot, int most) { return nshot - (nshot - 1) / most * most; }

// Tries reserve(choice) for the choices in order, the preferred one first, until one
// does not fail with `no_memory`; what a failed one holds is given back before the next.
template <class Choices, class Reserve, class Release>
int first_that_fits(const Choices &choices, int no_memory, Reserve reserve, Release release)
{
    int rc = no_memory;
    bool first = true;
    for (const auto &c : choices) {
        if (!first) release();
        first = false;
        rc = reserve(c);
        if (rc != no_memory) break;
    }
    return rc;
}

// Time chunks of the strain sums of the preconditioner maps (sem_integrals.cu):
// about five warps an SM from one shot, at least 16 steps each.  By the mesh and
// the time axis only: a rule on the warps of a whole batch let a smaller batch
// need more room than the one the buffer was sized for, and made the order of the
// sums depend on the batch.
inline int strain_chunks(long long elements, int nt)
{
    const long long warps = (elements + 31) / 32;
    return (int)std::min<long long>({std::max<long long>(1, 152 * 5 / warps), std::max(1, nt / 16), 64});
}

// bytes of those sums for `shots` shots: 25 points x 3 products of every element and chunk
inline size_t integral_bytes(long long elements, int nt, int shots)
{
    return (size_t)strain_chunks(elements, nt) * shots * 75 * elements * sizeof(float);
}

// Tiles of the U-Net's products (unet.cu): BM x BN outputs a CTA, kGemmBK deep stages
constexpr int kGemmBK = 32;
constexpr int gemm_bm(int M) { return M <= 32 ? 32 : (M <= 64 ? 64 : 128); }
constexpr int gemm_bn(int BM) { return 256 * 32 / BM; }

// k range of a split of an (M x N) output over K: enough splits to fill the
// SMs, each at least four tiles long, their partials within `cap` floats (one
// split needs none).  The rule fixes where the sums are cut, so it depends on one
// sample's shape only.
inline int split_chunk(int M, int N, int K, long long cap, int *splits_out)
{
    const int BM = gemm_bm(M), BN = gemm_bn(BM);
    const long long tiles = (long long)((M + BM - 1) / BM) * ((N + BN - 1) / BN);
    int splits = 1;
    if (tiles < 2 * 152 && K >= 8 * kGemmBK) {
        long long want = (2 * 152 + tiles - 1) / tiles;
        want = std::min<long long>(want, K / (4 * kGemmBK));
        want = std::min<long long>(want, std::max<long long>(1, cap / ((long long)M * N)));
        splits = (int)std::max<long long>(1, want);
    }
    const int kchunk = (int)(((K + splits - 1) / splits + kGemmBK - 1) / kGemmBK * kGemmBK);
    *splits_out = (K + kchunk - 1) / kchunk;
    return kchunk;
}

// Samples a product takes at once.  Its partials ([sample][split][M][N], `cap` floats
// in all) are needed for several splits, and for several samples that add to
// one output; a single sample with one split goes straight to its output.
inline int gemm_samples(long long outputs, int splits, int samples, bool accumulate, long long cap)
{
    if (splits == 1 && !accumulate) return samples;
    return (int)std::max<long long>(1, std::min<long long>(samples, cap / (outputs * splits)));
}
inline bool gemm_partial(int splits, int samples, bool accumulate) { return splits > 1 || (accumulate && samples > 1); }

}  // namespace sizes
