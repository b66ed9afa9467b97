// Reconstruction by merging regions along their best passes (recon_forest.cu):
// internal interface between the host API and its kernels.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>
#include "recon_internal.h"

namespace rf {

constexpr int BS = 64;                // block edge in pixels
constexpr int BPX = BS * BS;
constexpr int MAX_TERM = 256;         // node slots per block (at most 252 used: one per boundary pixel)
constexpr unsigned MAX_GROUP_BLOCKS = 1u << 16;   // blocks per launch group (268 Mpx) unless one tile needs more
constexpr unsigned MAX_BLOCKS = 1u << 23;         // node numbers (block * MAX_TERM + slot) stay below 2^31

// One tile of a launch group.
struct Tile {
    const uint8_t *I;
    uint8_t *J;
    int H, W, pitch;
    int nbx, nby;         // blocks across / down
    int dual, fill;       // as in rk::TileDesc
    int index;            // the tile's index in the caller's batch
};

// What the later kernels need to know of a block, in one 16-byte load.
struct alignas(16) Block {
    int tile;             // of the group
    unsigned local;       // block of the tile
    int nbx;              // the tile's blocks across
    unsigned nterm;       // nodes, and which neighbours exist
};
constexpr unsigned B_RIGHT = 1u << 8, B_DOWN = 1u << 9, B_UP = 1u << 10;

// Scratch of one launch group, per block: 2 bytes per pixel (value, node), the
// same for the four boundary lines, the node links, the block's record.
struct Params {
    Tile one;                     // the only tile, when tiles is NULL
    const Tile *tiles;            // tiles of the group
    const unsigned *base;         // ntiles + 1 cumulative block counts
    int ntiles;
    unsigned nblocks;
    uint16_t *px;                 // nblocks * BPX
    uint16_t *rim;                // nblocks * 4 * BS: top, bottom, left, right lines
    unsigned long long *link;     // nblocks * MAX_TERM: weight << 32 | parent node
    Block *block;                 // nblocks
    rk::Ctl *ctl;
    int *tile_err;                // by caller's tile index
    rk::Work *work;               // by caller's tile index
    int check;                    // check J <= I
    int flat;                     // 1: every tile is one block (no links between blocks)
    struct Status *next;          // cleared for the next call (may be NULL)
};

// Status and counters of a call on one tile. Two take turns: a call clears the
// other one, so that it needs no upload (its tile travels with the launches):
// 20.5 us a call in a row of asynchronous calls on 64^2, 30 with a copy before
// each; 64^2 with a synchronisation 59 -> 52 us, 512^2 83 -> 72.
struct Status {
    rk::Ctl ctl;
    int tile_err;
    rk::Work work;
};

inline size_t scratch_bytes(size_t nblocks)
{
    return nblocks * (sizeof(uint16_t) * (BPX + 4 * BS) + sizeof(unsigned long long) * MAX_TERM + sizeof(Block));
}

}  // namespace rf

extern "C" cudaError_t rf_configure();
extern "C" cudaError_t rf_launch(int conn, const rf::Params *P, cudaStream_t st);
