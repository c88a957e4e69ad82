// slice.h -- the bit-sliced step (slice.cu): plan and entry
// points (internal; not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "internal.cuh"

struct fractal;

namespace fr {

// Tiles of k^L cells (level-L subtrees) in groups of 32: bit t of word
// (g, slot) of a packed state is cell `slot` of tile 32 g + t.  Every tile
// has the same neighbour structure, so one word operation advances the same
// cell of 32 tiles.
struct SliceGeo {
    int L = 0;
    int KL = 0, KLp = 0;      // cells per tile; the same rounded up to 32 (words per group)
    int NC = 0;               // 32-cell chunks per tile
    int64_t NT = 0, NG = 0;   // tiles, groups of 32
    int H = 0;                // halo cells per tile
    int D = 0;                // neighbours per cell the kernel adds (the largest degree, as 4, 6, 7, 8, 20 or 26)
    int ND = 8;               // directions
    int NJ = 0, XW = 0;       // halo words a tile takes, export words it gives (at most 32 cells each)
    int BP = 0, RP = 0, AW = 0;   // shared-memory geometry (SliceArgs)
    uint4 *tab = nullptr;        // per cell: byte offsets (8 x uint16) of its neighbours' words in a group's word array
    uint32_t *jobs = nullptr;    // [NJ]: export word | direction << 8
    uint16_t *xlist = nullptr;   // [XW][32]: cells of the export words
    uint2 *cells = nullptr;      // [H]: cell of the neighbouring tile, its word in a group's array | direction << 16
    int32_t *nbr = nullptr;      // [NG][ND][32]: neighbouring tile of each tile of a group by direction, -1 = none
};

// When to try an allocation again that was refused (which takes 5 ms): after
// 16 calls, after twice as many at each further refusal, at most 1024.
struct Retry {
    int left = 0, next = 16;
    bool skip()   // whether this call goes without
    {
        if (left == 0) return false;
        --left;
        return true;
    }
    void refused()
    {
        left = next;
        next = next < 1024 ? 2 * next : next;
    }
    void granted() { next = 16; }
};

struct SlicePlan {
    bool several = false;     // a call of several generations has run
    bool single = false;      // a single generation has run on the tile kernels before the tables were built
    int state = 0;            // 0: not planned yet, 1: planned, 2: its tables exist, -1: not possible for this fractal
    Retry memory;             // its allocations
    SliceGeo geo;
    bool resident = false;    // the packed state stays in shared memory: one launch for all generations
    int per_block = 0, rounds = 0, block_resident = 0, grid_resident = 0, smem_resident = 0;
    int block = 256;          // streaming kernels: threads per block
    int smem_pack = 0, smem_step = 0, smem_bytes = 0, smem_single = 0;
    int grid_pack = 0, grid_step[2] = {0, 0}, grid_bytes[2] = {0, 0}, grid_single[2] = {0, 0};   // [1]: with the constant rule
    // packed states (NG x KLp words, then the exports, NG x XW x 32): two of calls of several generations, one of single ones
    uint32_t *bits[3] = {nullptr, nullptr, nullptr};
    uint8_t *packed[2] = {nullptr, nullptr};  // those that are not in the arena: of several generations, of single ones
    uint8_t *arena = nullptr;                 // the tables, packed states of the first kind of call that needs some, and:
    uint8_t *groups = nullptr;                // batches: the groups (SliceGroup)
    uint32_t *ex[3] = {nullptr, nullptr, nullptr};   // resident kernel: the exports alone, likewise
    uint32_t *bar = nullptr;                  // grid barriers: arrivals, exits; single generations' own behind them
};

void free_slice_plan(SlicePlan &p);

// `steps` >= 1 generations from bytes to bytes; *done = false (and nothing
// launched) when the fractal, the handle's settings or the memory at hand
// rule the sliced step out.
int try_slice_step(fractal *f, const uint8_t *in, uint8_t *out, int64_t steps, uint32_t birth, uint32_t survive,
                   cudaStream_t st, bool *done);

// Batches: the instances that may go through sliced launches, their launches
// (all items of one fractal table and one rule), and running them.
struct SliceBatchItem {
    fractal *f;
    const uint8_t *in;
    uint8_t *out;
    int64_t steps;
};
struct SliceBatch;
bool slice_batch_takes(const fractal *f, int64_t steps);
int build_slice_batch(const std::vector<SliceBatchItem> &items, uint32_t birth, uint32_t survive, cudaStream_t st, SliceBatch **out);
int run_slice_batch(const SliceBatch *b, cudaStream_t st);
int slice_batch_launches(const SliceBatch *b);
void free_slice_batch(SliceBatch *b);

}  // namespace fr
