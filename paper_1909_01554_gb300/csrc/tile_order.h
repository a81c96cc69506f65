// The order in which the tensor kernels walk the tiles of C.
#pragma once

#include <stdint.h>

namespace bmm {

// Tile raster: groups of GROUP_M row-tiles, column by column within a
// group. Each Bt tile is read from DRAM once per group while the group's
// rows of A (32 x 256 rows x k bits: 32 MiB at k = 32768 for pairs) stay in
// L2 (measured: 64 row-tiles no longer fit and A is re-read).
constexpr int GROUP_M = 32;

struct TileCoord {
    int leaf, tm, tn;
};

// t / d for 0 <= t < 2^31 by a multiplication (the compiler's division takes some
// 25 instructions; three of them in a row were 650 of the 2700 cycles that the
// epilogue of a short tile took).
struct FastDiv {
    uint32_t d = 1, mul = 1, shift = 0;
    void set(uint32_t div) {
        d = div;
        for (shift = 0; (1ull << shift) < div;) shift++;
        mul = (uint32_t)((((1ull << shift) - div) << 32) / div + 1);
    }
#ifdef __CUDACC__
    __device__ __forceinline__ uint32_t operator()(uint32_t t) const {
        return (__umulhi(t, mul) + t) >> shift;
    }
#endif
};

// The raster over `count` leaves of one shape, tiles_m * tiles_n * count < 2^31.
struct TileOrder {
    FastDiv per_leaf, group, last_rows;  // last_rows: row-tiles of the last group
    int last_group = 0;
    void set(int tiles_m, int tiles_n) {
        per_leaf.set((uint32_t)tiles_m * (uint32_t)tiles_n);
        group.set((uint32_t)(GROUP_M * tiles_n));
        last_group = (tiles_m - 1) / GROUP_M;
        last_rows.set((uint32_t)(tiles_m - last_group * GROUP_M));
    }
#ifdef __CUDACC__
    __device__ __forceinline__ TileCoord tile(int t) const {
        TileCoord c;
        c.leaf = (int)per_leaf((uint32_t)t);
        const int r = t - c.leaf * (int)per_leaf.d;
        const int g = (int)group((uint32_t)r);
        const uint32_t in = (uint32_t)(r - g * (int)group.d);
        const bool last = g == last_group;
        c.tn = (int)(last ? last_rows(in) : in / GROUP_M);
        c.tm = g * GROUP_M + (int)in - c.tn * (last ? (int)last_rows.d : GROUP_M);
        return c;
    }
#endif
};

}  // namespace bmm
