// Block order of the batched stencil kernels: z-slabs along t.
//
// A stencil kernel over N right-hand sides runs one block per (site block, right-hand
// side), right-hand side fastest, so each block's neighbour gathers hit data that other
// blocks brought into L2.  In the plain site order (x fastest, t slowest) a t-neighbour
// lies one whole 3-D slice away.  With 16 right-hand sides on 24^3 x 48 the vectors that the
// kernels of an iteration go through in a slice do not stay in L2, so those gathers go to DRAM
// a second time.
//
// The walk here takes slabs of bz z-planes at one t, each a contiguous range of
// bz * plane sites: the slabs of z-slab 0 for t = 0 .. Lt-1, then those of z-slab 1, and so
// on.  A t-neighbour is then one slab behind or ahead of the block that gathers it.  The
// price is the z-neighbours across a slab edge (2 of bz planes), which come from DRAM
// again.  bz = Lz is the plain order.
//
// `plane` counts the sites of one (x, y) plane of the field: Lx Ly for a full lattice,
// Lx Ly / 2 for one parity of an even-odd field (its checkerboard index s >> 1 keeps the
// planes contiguous).
#pragma once

#include <algorithm>
#include <cstdlib>

#include "fast_div.cuh"

namespace dlz {

constexpr int kSlabBlock = 128;     // sites per block

struct SlabWalk {
    int bz;          // z-planes per slab
    int bps;         // blocks per slab
    int plane;       // sites per plane
    int Lz, Lt;
    FastDiv dbps, dLt, dN;   // divisors: bps, Lt and the right-hand sides of the launch
};

// the right-hand side q and site block sb of a launch with right-hand sides fastest
__device__ inline void slab_rhs(const SlabWalk &w, int block, int &q, int &sb) {
    sb = w.dN.div(block);
    q = block - sb * (int)w.dN.d;
}

// first site s0 and site count nb of site block sb (nb = 0 for the spare blocks of a
// short last z-slab)
__host__ __device__ inline void slab_block(const SlabWalk &w, int sb, int &s0, int &nb) {
    const int j = w.dbps.div(sb), off = (sb - j * w.bps) * kSlabBlock;
    const int zs = w.dLt.div(j), t = j - zs * w.Lt, z0 = zs * w.bz;
    const int planes = w.bz < w.Lz - z0 ? w.bz : w.Lz - z0;
    const int len = planes * w.plane;
    s0 = (t * w.Lz + z0) * w.plane + off;
    const int rest = len - off;
    nb = rest <= 0 ? 0 : (rest < kSlabBlock ? rest : kSlabBlock);
}

// The walk with slabs of bz planes, for N right-hand sides
inline SlabWalk slab_walk_of(int plane, int Lz, int Lt, int bz, int N = 1) {
    SlabWalk w;
    w.plane = plane;
    w.Lz = Lz;
    w.Lt = Lt;
    w.bz = std::max(1, std::min(bz, Lz));
    w.bps = (w.bz * plane + kSlabBlock - 1) / kSlabBlock;
    w.dbps = FastDiv((unsigned)w.bps);
    w.dLt = FastDiv((unsigned)Lt);
    w.dN = FastDiv((unsigned)(N > 0 ? N : 1));
    return w;
}

// The walk for N right-hand sides of weight `bytes` per site and right-hand side: the plain
// order when a slab weighs 36 MB at most, else the largest divisor of Lz whose slab does (at
// least one plane).  The weights are set by measurement, not equal to a kernel's streams.  With
// 900 the fused kernels take 4 planes on 24^3 x 48 with 16 right-hand sides, where K1 / K23 took,
// relative to that, 1.29 / 1.27 with 1 plane, 1.06 / 1.06 with 2, 1.03 / 1.03 with 3, 0.99 / 1.00
// with 6, 1.02 / 1.02 with 8, 1.03 / 1.05 with 12 and 1.12 / 1.16 in the plain order; MinRes K1
// with 11 right-hand sides (6 planes) 1.05, 1.01, 1.00, 1.00 and 1.04 with 3, 4, 8, 12 and 24.  The
// even-odd pairs with 16 (8 planes, the hop in the plain order) are fastest so.  Lighter launches
// (24^3 x 48 with 4 right-hand sides, 16^3 x 32 with 11 and 16) would gain 1 to 3 % in the plain
// order.  DLZ_SLAB=n fixes n planes.
inline SlabWalk make_slab_walk(int plane, int Lz, int Lt, int N, double bytes) {
    const double per_plane = (double)plane * N * bytes;
    int bmax = per_plane > 0.0 ? (int)std::min((double)Lz, 36.0e6 / per_plane) : Lz;
    int bz = 1;
    for (int d = 1; d <= std::max(1, bmax); ++d)
        if (Lz % d == 0) bz = d;
    if (const char *env = std::getenv("DLZ_SLAB")) {
        const int v = std::atoi(env);
        if (v > 0) bz = v;
    }
    return slab_walk_of(plane, Lz, Lt, bz, N);
}

// blocks per right-hand side
inline long slab_blocks(const SlabWalk &w) { return (long)w.bps * w.Lt * ((w.Lz + w.bz - 1) / w.bz); }

}  // namespace dlz
