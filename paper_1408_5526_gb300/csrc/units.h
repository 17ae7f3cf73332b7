// units.h -- how a plan's M replications of N points are cut into work units (host arithmetic).
//
// A unit is a tile of threads x ppt consecutive points of one replication.  Kernels and reductions
// index units in 32 bits, and N M reaches 2^47, so plans too large for their kernel's usual tile
// take one with more points per thread.
#pragma once
#include <cstdint>

namespace rqmc {

struct UnitShape {
    int ppt;                 // points per thread
    uint32_t tile;           // points of a unit
    uint32_t tiles_per_m;    // units of a replication
    uint32_t units;
};

// threads x ppt points per unit, ppt doubled until M replications of N points have fewer than 2^32
// units (N <= 2^31, M < 2^16, 32 to 256 threads: ppt ends below 2^14).
inline UnitShape unit_shape(uint64_t N, uint32_t M, int threads, int ppt) {
    for (;; ppt *= 2) {
        const uint64_t tile = (uint64_t)threads * (uint64_t)ppt, tiles = (N + tile - 1) / tile, units = tiles * M;
        if (units < 0xFFFFFFFFull) return UnitShape{ppt, (uint32_t)tile, (uint32_t)tiles, (uint32_t)units};
    }
}

}  // namespace rqmc
