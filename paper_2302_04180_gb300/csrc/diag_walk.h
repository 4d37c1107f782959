// Which chunks of 32 rows a warp of the diagonal product takes (spmv_rows_diag,
// kernels.cuh), and their rows. Index arithmetic only, so that the CPU can run it.
#pragma once

#ifdef __CUDACC__
#define RBS_HD __host__ __device__ __forceinline__
#else
#define RBS_HD inline
#endif

namespace rbs {

// The chunks [begin, end) over nblk blocks of nw warps, this warp being wid of block
// blk: whole rounds of tiles (TILE groups of a block's consecutive chunks, one per
// warp, before it moves on), then chunk by chunk, so that the last round is even
// over the blocks. A walk at or past `end` is over.
template <int TILE>
struct DiagChunks {
    int begin, end, blk, nblk, wid, nw;
    struct Walk {
        int c, left;  // the chunk; steps to go in its tile
    };
    RBS_HD int round() const { return nblk * nw; }
    RBS_HD int tiled() const {
        return TILE == 1 ? begin : begin + (end - begin) / (round() * TILE) * (round() * TILE);
    }
    RBS_HD Walk first() const {
        return tiled() > begin ? Walk{begin + blk * (TILE * nw) + wid, TILE - 1} : Walk{begin + blk * nw + wid, 0};
    }
    RBS_HD Walk next(Walk w) const {
        if (TILE == 1 || (w.left == 0 && w.c >= tiled())) return Walk{w.c + round(), 0};
        if (w.left > 0) return Walk{w.c + nw, w.left - 1};
        w = Walk{w.c + (round() - nw) * TILE + nw, TILE - 1};  // the next round's tile
        return w.c < tiled() ? w : Walk{tiled() + blk * nw + wid, 0};
    }
    // The row of `lane` in chunk c; n or more, up to n = 2^31 - 1, past the last
    // chunk, where a walk goes on for up to two rounds and 32 c leaves an int.
    // (Asking for c < end instead costs K1 and K3 2 %.)
    RBS_HD static unsigned row(int c, int lane) { return (unsigned)c * 32u + (unsigned)lane; }
};

}  // namespace rbs
