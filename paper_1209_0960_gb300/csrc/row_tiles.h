// The entries of 32 consecutive CSR rows, [s, e), in tiles: what the
// allocation-free residual norm copies to shared memory at a time.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define AMG_HD __host__ __device__ __forceinline__
#else
#define AMG_HD inline
#endif

namespace amg {

// entries per tile: 32 rows of a 7-point stencil fit in one, longer runs take more
constexpr int32_t kNaTile = 224;

// Entry counts go up to the largest int32, so positions are compared by their
// distance from the tile's start: base + kNaTile may lie past the last one.
struct RowTiles {
    int32_t base, e;
    AMG_HD RowTiles(int32_t s, int32_t e_) : base(s), e(e_) {}
    // where the entries of a row that ends at k1 end within the tile
    AMG_HD int32_t end_in_tile(int32_t k1) const { return k1 - base < kNaTile ? k1 : base + kNaTile; }
    // on to the next tile; false after the last
    AMG_HD bool next() {
        if (e - base <= kNaTile) return false;
        base += kNaTile;
        return true;
    }
};

}  // namespace amg
