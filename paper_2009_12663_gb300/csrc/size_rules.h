// Sizes of scratch that one piece of host code reserves and another fills, as
// plain C++ without CUDA types: both sides call the same function, and the rules
// can be checked on a machine without a GPU.
#pragma once

#include <algorithm>
#include <cstddef>

namespace sizes {

// shots of the last of the batches that take `nshot` shots `most` at a time
inline int last_batch(int nshot, int most) { return nshot - (nshot - 1) / most * most; }

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

}  // namespace sizes
