// What a tile of the resident time loop (sem_resident.cu) can hold, the shared
// memory it takes and the choice of the tile for a number of shots, as plain C++
// without CUDA types (the kernel, its host side and a host check share it).
#pragma once

#include <algorithm>
#include <cstddef>

#ifdef __CUDACC__
#define GB_HOSTDEV __host__ __device__
#else
#define GB_HOSTDEV
#endif

namespace resident {

// Window cells ((TX+2) (TZ+2)), owned elements and exchanged nodes a thread of a
// tile of NT element threads (limits checked by fits()).
struct Limits { int cells, owned, halo; };
GB_HOSTDEV constexpr Limits limits_of(int NT)
{
    return NT == 64 ? Limits{90, 49, 5} : NT == 128 ? Limits{153, 105, 4} : Limits{220, 162, 4};
}
constexpr int kTileThreads[] = {64, 128, 192};

// correlation threads (adjoint), and resident CTAs an SM: as many as shared memory holds
GB_HOSTDEV constexpr int corr_threads(int NT, bool adj) { return adj ? (limits_of(NT).owned + 31) / 32 * 32 : 0; }
GB_HOSTDEV constexpr int blocks_per_sm(int NT, bool adj) { return adj ? (NT == 64 ? 3 : 1) : (NT == 64 ? 6 : NT == 128 ? 3 : 2); }
// float4 before the exchange inside the tile: field window (two in the adjoint), moduli
// window, 1/M; adjoint: accelerations [8], strain sums [13] and mass sums [4] of every owned element
GB_HOSTDEV constexpr int window_f4(int NT) { return 8 * limits_of(NT).cells; }
GB_HOSTDEV constexpr int head_f4(int NT, bool adj) { return (adj ? 3 : 2) * window_f4(NT) + 4 * NT + (adj ? 25 * limits_of(NT).owned : 0); }
GB_HOSTDEV constexpr size_t head_bytes(int NT, bool adj) { return (size_t)head_f4(NT, adj) * 16 + (size_t)(9 * NT) * 8; }   // before the Tail

// Shared memory behind the windows and per-element arrays, in floats (every
// piece a multiple of 4 floats)
struct Tail {
    int edge, ev, vx, xi, ent, sig, inj, grp, rec, recw, recv, send, total;
};
GB_HOSTDEV inline int up4(int v) { return (v + 3) & ~3; }
GB_HOSTDEV inline Tail tail_of(bool adj, bool one_tile, int TX, int TZ, int edge_cap, int grp_cap, int ent_cap, int rec_cap)
{
    Tail q;
    int o = 0;
    auto take = [&](int n) { const int at = o; o += up4(n); return at; };
    q.edge = take(4 * edge_cap);                  // Stacey factors of the tile's absorbing edges (float4)
    q.ev = take(adj ? 4 * edge_cap : 0);          // mean velocity and acceleration there (two float2)
    q.vx = take(2 * (4 * (TX + TZ) + 1));         // velocity of the extra node lines (float2)
    q.xi = take(4 * (4 * (TX + TZ) + 1));         // their places (int4, see the element threads)
    q.ent = take(4 * ent_cap);                    // injection entries: (offset x, offset z, weight x, weight z)
    q.sig = take(4 * ent_cap);                    // their signals, two steps
    q.inj = take(2 * grp_cap);                    // injected forces (float2)
    q.grp = take(grp_cap + 1);                    // first entry of every group
    q.rec = take(4 * rec_cap);                    // recorded receivers: id and the cells of their patch (int, 4 shorts)
    q.recw = take(25 * rec_cap);                  // their weights
    q.recv = take(one_tile ? 0 : 2 * (20 * (TX + TZ) + 25));   // nodes to receive and to send (int2: node, window slot)
    q.send = take(one_tile ? 0 : 2 * (20 * (TX + TZ) + 25));
    q.total = o;
    return q;
}

inline bool fits(int NT, int TX, int TZ)
{
    const Limits L = limits_of(NT);
    return (TX + 1) * (TZ + 1) <= NT && (TX + 2) * (TZ + 2) <= L.cells && TX * TZ <= L.owned &&
           20 * (TX + TZ) + 25 <= L.halo * NT;
}

// edge slots of a tile: the sides it can touch
inline int edge_cap(int TX, int TZ, int ntx, int ntz, bool free_top)
{
    return (4 * TZ + 1) * (ntx == 1 ? 2 : 1) + (4 * TX + 1) * (ntz == 1 && !free_top ? 2 : 1);
}

inline size_t smem_bytes(int NT, bool adj, int TX, int TZ, int ntx, int ntz, bool free_top, int grp_cap, int ent_cap, int rec_cap)
{
    return head_bytes(NT, adj) + sizeof(float) * (size_t)tail_of(adj, ntx * ntz == 1, TX, TZ, edge_cap(TX, TZ, ntx, ntz, free_top),
                                                                 grp_cap, ent_cap, rec_cap).total;
}

struct Tile { int NT, TX, TZ, ntx, ntz; };   // NT 0: none

// The tile whose model time per step of all `shots` is smallest among those of
// which at least one whole shot is resident at once, also with the lists of the
// acquisition.  slots(NT, smem, nsm) gives the resident CTAs of a variant on the device and its
// SMs; usable(tile) whether a shot is resident with its lists.  Whether any tile is found
// depends on the mesh and the acquisition only, not on `shots`: gradients of the
// resident loop and of the step kernels round alike but for the order of the strain
// sums, so a mesh keeps to one of them whatever its batches.
template <class Slots, class Usable>
Tile best_tile(int nex, int nez, bool free_top, bool adj, int shots, Slots slots, Usable usable)
{
    Tile best{};
    double best_cost = 1e300;
    for (int NT : kTileThreads) {
        int nsm = 0, have = 0;
        size_t known = 0;                        // shared bytes `have` was looked up for
        for (int tx = 1; tx < NT; ++tx) {
            // shapes with equal tile counts differ only in their padding: balance them
            const int tz = std::min(NT / (tx + 1) - 1, nez);
            if (tz < 1 || tx > nex) continue;
            const int ntx = (nex + tx - 1) / tx, ntz = (nez + tz - 1) / tz;
            const int TX = (nex + ntx - 1) / ntx, TZ = (nez + ntz - 1) / ntz;
            if (!fits(NT, TX, TZ)) continue;
            const long long T = (long long)ntx * ntz;
            const size_t smem = smem_bytes(NT, adj, TX, TZ, ntx, ntz, free_top, 8, 8, 0);
            if (smem != known) have = slots(NT, smem, nsm);
            known = smem;
            const int cap = (int)std::min<long long>(shots, have / T);
            int asked = -1;                      // usable(): not asked yet
            for (int c = 1; c <= cap; ++c) {
                // a step takes the larger of a warp's latency (with the exchange
                // between tiles) and the busiest SM's issue time
                const double warps = ((TX + 1) * (TZ + 1) + 31) / 32 * (double)((c * T + nsm - 1) / nsm);
                // (us; measured: 4.2 us forward and 5.7 us adjoint a step with one CTA an SM,
                // 5.3 us forward with two)
                const double issue = (adj ? 0.90 : 0.43) * warps;
                const double lat = (adj ? 3.6 : 2.6) + (T > 1 ? 1.2 : 0.0) + 0.05 * warps;
                const double cost = ((shots + c - 1) / c) * std::max(issue, lat);
                if (cost < best_cost * (1 - 1e-9)) {
                    const Tile t{NT, TX, TZ, ntx, ntz};
                    if (asked < 0) asked = usable(t);
                    if (!asked) break;
                    best_cost = cost;
                    best = t;
                }
            }
        }
    }
    return best;
}

// bytes of the exchange of node lines between the tiles of one launch: two slots
// of two 64-bit words a node (pitched) and shot; `shots` of a batch go per_launch at a time
inline size_t exchange_bytes(int ntiles, int shots, int per_launch, long long nodes)
{
    return ntiles > 1 ? (size_t)32 * std::min(shots, per_launch) * nodes : 16;
}

}  // namespace resident
