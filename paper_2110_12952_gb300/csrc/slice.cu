// slice.cu -- the bit-sliced compact step (Sec. 3 stencil procedure on 32
// tiles at a time).
//
// A tile is a level-L subtree (k^L cells, contiguous in omega).  All tiles
// have the same local neighbour structure: cell l of a tile has, for each
// Moore direction, either no neighbour at all, a fixed local cell of the same
// tile, or a fixed local cell of the neighbouring tile in a fixed direction.
// So 32 tiles are packed into words, bit t of word l being cell l of tile
// 32 g + t, and one generation of a word is: load the words of its member
// neighbours (at most 8, addresses from a table that is the same for every
// group), add them bit-sliced, apply the rule as logic.  Cells off the
// fractal take no storage, no loads and no operations.
//
// The cells of neighbouring tiles that touch a tile (its halo: 8 for the
// triangle, 4 x 81 + 4 for the carpet's 81 x 81 tiles) travel as bit strings:
// with every state goes, per tile, a word for each run of at most 32 border
// cells (its exports).  Lane t of a warp loads the export of tile 32 g + t's
// neighbour, and a 32 x 32 bit transposition across the warp turns the lanes'
// words into the halo cells' words; the exports of the new state are made by
// the same transposition from its words.
//
// Bytes become bits first, in omega order (16 consecutive bytes per thread and
// load, a nibble per word by a carry-free multiply), so that everything that
// is not aligned happens in bits: lane t takes 32 cells of tile t out of the
// bit string with one funnel shift, and a 32 x 32 bit transposition across
// the warp (five shuffle stages) leaves lane p with cell p of 32 tiles.  The
// way back is the same in reverse.
#include <cuda_runtime.h>
#include <stdint.h>

#include <string.h>

#include <algorithm>
#include <cmath>
#include <list>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "handle.h"
#include "step.h"
#include "tma.cuh"

namespace fr {

constexpr int kSliceBlock = 256;   // threads per block of the streaming kernels
constexpr int kSliceBlock3 = 512;  // the same in 3D, where a group is larger (Menger: 8000 words and 3700 halo words)
constexpr int kSliceAhead = 2;     // halo words per warp loaded ahead of their group
constexpr int kSliceBatch = 4;     // 16-byte units per thread and batch copied to shared memory ahead
constexpr int kSliceMost = 112 * 1024;   // the other kernels': most shared memory per block
constexpr int kSliceSmem = 220 * 1024;   // resident kernel: shared memory per block
constexpr int64_t kSliceBatchCells = 60000000;   // batches: most cells of an instance
constexpr int kSliceSingleHalo = 32;   // most halo cells of a tile for the single-pass kernel
constexpr int kSliceRounds = 32;   // resident kernel: most 32-cell chunks per warp

// One group of a batch: its bytes, its tiles and where its instance lies
// among the launch's groups.
struct SliceGroup {
    const uint8_t *in;
    uint8_t *out;
    int32_t nt;                 // tiles (at most 32)
    int32_t tile0, levels;      // first tile in its instance, the instance's levels above the tiles
    int32_t group0;             // the instance's first group
    int32_t steps;              // generations; groups come in order of decreasing steps
};

struct SliceArgs {
    int64_t NT, NG;
    int KL, KLp, NC, NJ, XW, H;
    int ND;                 // directions: 8, or 26 in 3D
    uint32_t birth, survive;
    int64_t ex;             // word offset of a state's exports behind its cells
    int BP;                 // packing: words between tiles' bit strings when a tile is 2^bsh words, else 0
    int bsh;                // (30: another number)
    uint32_t lane_bits;     // packing: bits between tiles' bit strings
    int RP;                 // unpacking: words between tiles' bit strings (odd)
    int AW, A_zero;         // words of one group's array, index of its 32 zero words
    DivU32 kdiv, cdiv, jdiv, xdiv;   // division by KL, NC, NJ and XW
    uint32_t mb[9], ms[9];  // rule: all ones where a dead / live cell with c live neighbours becomes live
    const uint4 *tab;
    const uint32_t *jobs;   // halo words: export word | direction << 8
    const uint16_t *xlist;  // [XW][32]: cells of the export words
    const uint2 *cells;     // [H] halo cells: cell of the neighbouring tile, word index | direction << 16
    const int32_t *nbr;
    const SliceGroup *groups;   // batches: [NG], else null
    uint32_t *bar;
    int *status;
};

// Transpose of a 32 x 32 bit matrix held as a row per lane: afterwards bit t
// of lane p is what bit p of lane t was.  Five exchanges of halves: of 16 and
// 8 bits by byte permutes, of 4, 2 and 1 by a rotation and a bit select.
struct Transpose32 {
    uint32_t sel16, sel8, keep[3], rot[3];
    __device__ __forceinline__ Transpose32(int lane)
    {
        sel16 = (lane & 16) ? 0x3276u : 0x5410u;
        sel8 = (lane & 8) ? 0x3715u : 0x6240u;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int s = 4 >> i;
            const uint32_t lowm = s == 4 ? 0x0f0f0f0fu : s == 2 ? 0x33333333u : 0x55555555u;
            const bool low = (lane & s) == 0;
            keep[i] = low ? lowm : ~lowm;
            rot[i] = low ? s : 32 - s;
        }
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t x) const
    {
        x = __byte_perm(x, __shfl_xor_sync(0xffffffffu, x, 16), sel16);
        x = __byte_perm(x, __shfl_xor_sync(0xffffffffu, x, 8), sel8);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const uint32_t y = __shfl_xor_sync(0xffffffffu, x, 4 >> i);
            x = (x & keep[i]) | (__funnelshift_l(y, y, rot[i]) & ~keep[i]);
        }
        return x;
    }
};

__device__ __forceinline__ uint32_t sl_xor3(uint32_t a, uint32_t b, uint32_t c) { return a ^ b ^ c; }
__device__ __forceinline__ uint32_t sl_maj3(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a | b)); }
__device__ __forceinline__ uint32_t sl_mux(uint32_t s, uint32_t a, uint32_t b) { return (s & a) | (~s & b); }

// N bits of one weight added: their sum's low bit, and the carries.
template <int N>
__device__ __forceinline__ uint32_t sl_reduce(const uint32_t *x, uint32_t *carry)
{
    uint32_t s = x[0];
    int c = 0;
#pragma unroll
    for (int i = 1; i + 1 < N; i += 2) {
        carry[c++] = sl_maj3(s, x[i], x[i + 1]);
        s = sl_xor3(s, x[i], x[i + 1]);
    }
    if (N % 2 == 0) {
        carry[c] = s & x[N - 1];
        s ^= x[N - 1];
    }
    return s;
}

// 3D: next state from up to D neighbours' words; LIFE: B5/S45, else a sum
// over the counts the rule maps to "alive".
template <int D, bool LIFE>
__device__ __forceinline__ uint32_t slice_rule3(const SliceArgs &a, const uint32_t *n, uint32_t alive)
{
    constexpr int N1 = D / 2, N2 = N1 / 2, N3 = N2 / 2;   // carries of each weight (sl_reduce of n leaves n / 2)
    uint32_t c1[N1], c2[N2], c3[N3], c4[1];
    const uint32_t t0 = sl_reduce<D>(n, c1), t1 = sl_reduce<N1>(c1, c2), t2 = sl_reduce<N2>(c2, c3), t3 = sl_reduce<N3>(c3, c4);
    static_assert(N3 / 2 == 1, "five planes");
    const uint32_t t4 = c4[0];
    if (LIFE) return t2 & ~t1 & ~t3 & ~t4 & (t0 | alive);
    uint32_t r = 0u;
    for (uint32_t m = a.birth | a.survive; m; m &= m - 1u) {
        const int v = __ffs((int)m) - 1;
        const uint32_t eq = ((v & 1) ? t0 : ~t0) & ((v & 2) ? t1 : ~t1) & ((v & 4) ? t2 : ~t2) & ((v & 8) ? t3 : ~t3) &
                            ((v & 16) ? t4 : ~t4);
        r |= eq & (((a.survive >> v) & 1u ? alive : 0u) | ((a.birth >> v) & 1u ? ~alive : 0u));
    }
    return r;
}

// Next state of 32 cells from their neighbours' words n[0..D-1] (absent ones
// zero): bit-sliced count, then the rule.
template <int D, bool LIFE>
__device__ __forceinline__ uint32_t slice_rule(const SliceArgs &a, const uint32_t *n, uint32_t alive)
{
    uint32_t t0, t1, t2, t3 = 0u;
    if constexpr (D == 4) {
        const uint32_t s = sl_xor3(n[0], n[1], n[2]), c = sl_maj3(n[0], n[1], n[2]);
        const uint32_t k = s & n[3];
        t0 = s ^ n[3];
        t1 = c ^ k;
        t2 = c & k;
    } else {
        const uint32_t s0 = sl_xor3(n[0], n[1], n[2]), c0 = sl_maj3(n[0], n[1], n[2]);
        const uint32_t s1 = sl_xor3(n[3], n[4], n[5]), c1 = sl_maj3(n[3], n[4], n[5]);
        if constexpr (D == 6) {
            const uint32_t k = s0 & s1;
            t0 = s0 ^ s1;
            t1 = sl_xor3(c0, c1, k);
            t2 = sl_maj3(c0, c1, k);
        } else if constexpr (D == 7) {
            const uint32_t k = sl_maj3(s0, s1, n[6]);
            t0 = sl_xor3(s0, s1, n[6]);
            t1 = sl_xor3(c0, c1, k);
            t2 = sl_maj3(c0, c1, k);
        } else {
            const uint32_t s2 = n[6] ^ n[7], c2 = n[6] & n[7];
            const uint32_t k = sl_maj3(s0, s1, s2);
            t0 = sl_xor3(s0, s1, s2);
            const uint32_t u = sl_xor3(c0, c1, c2), v = sl_maj3(c0, c1, c2);
            t1 = u ^ k;
            const uint32_t w = u & k;
            t2 = v ^ w;
            t3 = v & w;
        }
    }
    if constexpr (LIFE) return t1 & ~t2 & (t0 | alive);   // B3/S23 (a count of 8 has t1 = 0)
    uint32_t b = sl_mux(t2, sl_mux(t1, sl_mux(t0, a.mb[7], a.mb[6]), sl_mux(t0, a.mb[5], a.mb[4])),
                        sl_mux(t1, sl_mux(t0, a.mb[3], a.mb[2]), sl_mux(t0, a.mb[1], a.mb[0])));
    uint32_t s = sl_mux(t2, sl_mux(t1, sl_mux(t0, a.ms[7], a.ms[6]), sl_mux(t0, a.ms[5], a.ms[4])),
                        sl_mux(t1, sl_mux(t0, a.ms[3], a.ms[2]), sl_mux(t0, a.ms[1], a.ms[0])));
    if constexpr (D == 8) {
        b = sl_mux(t3, a.mb[8], b);
        s = sl_mux(t3, a.ms[8], s);
    }
    return sl_mux(alive, s, b);
}

// ---------------------------------------------------------------- pack

// 16 cells (bytes of any nonzero value) -> 16 bits.
__device__ __forceinline__ uint32_t slice_bits16(uint4 v)
{
    if ((v.x | v.y | v.z | v.w) & 0xfefefefeu) {   // bytes other than 0 and 1
        v.x = (((v.x & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v.x) >> 7 & 0x01010101u;
        v.y = (((v.y & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v.y) >> 7 & 0x01010101u;
        v.z = (((v.z & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v.z) >> 7 & 0x01010101u;
        v.w = (((v.w & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v.w) >> 7 & 0x01010101u;
    }
    // the four 0/1 bytes of a word land in the product's top nibble
    uint32_t x = (v.w * 0x10204080u) >> 28;
    x = __funnelshift_l(v.z * 0x10204080u, x, 4);
    x = __funnelshift_l(v.y * 0x10204080u, x, 4);
    return __funnelshift_l(v.x * 0x10204080u, x, 4);
}

// The exports of a group from its words in memory (written by this block and
// behind a barrier; a copy in shared memory would cost a block or two per SM):
// lane i takes cell i of an export word, lane t gets tile t's bits.
__device__ __forceinline__ void slice_export(const SliceArgs &a, const Transpose32 &tr, const uint32_t *words, uint32_t *ex,
                                             int warp, int nw, int lane)
{
#pragma unroll 2
    for (int x = warp; x < a.XW; x += nw) ex[32 * x + lane] = tr(words[__ldg(a.xlist + 32 * x + lane)]);
}

// Words of a group's bit string in shared memory (one to spare for the funnel shifts).
__device__ __forceinline__ int slice_string_words(const SliceArgs &a) { return a.BP ? 32 * a.BP : a.KLp + 1; }

// Half word i of a group's bit string.  A tile of 2^bsh words (bsh = 30:
// other tiles) takes one word more, so that the 32 tiles' rows fall into
// different banks.
__device__ __forceinline__ void slice_put16(const SliceArgs &a, uint32_t *B, int i, uint32_t x)
{
    reinterpret_cast<uint16_t *>(B)[i + 2 * (i >> (a.bsh + 1))] = (uint16_t)x;
}

// Units of 16 bytes from `from` on (of a buffer that is not 16-byte aligned:
// all of them), byte by byte.
__device__ __forceinline__ void slice_odd_units(const SliceArgs &a, const uint8_t *__restrict__ src, int bytes, int from,
                                                uint32_t *B, int tid, int nth)
{
    for (int i = from + tid; 16 * i < bytes; i += nth) {
        uint32_t x = 0;
        for (int j = 0; j < 16 && 16 * i + j < bytes; ++j) x |= (uint32_t)(src[16 * i + j] != 0) << j;
        slice_put16(a, B, i, x);
    }
}

// The bytes of a group of nt tiles as a bit string in omega order, by nth threads.
__device__ __forceinline__ void slice_bytes_to_string(const SliceArgs &a, const uint8_t *__restrict__ src, int nt, uint32_t *B,
                                                      int tid, int nth)
{
    const int bytes = nt * a.KL;
    const int whole = ((uintptr_t)src & 15) == 0 ? bytes / 16 : 0;
#pragma unroll 4
    for (int i = tid; i < whole; i += nth)
        slice_put16(a, B, i, slice_bits16(__ldcs(reinterpret_cast<const uint4 *>(src) + i)));
    slice_odd_units(a, src, bytes, whole, B, tid, nth);
}

// The same for blocks that walk the groups: every thread copies the 16-byte
// units it will convert into its own slots of shared memory, a batch ahead
// and across group boundaries, and waits for its own copies only.  A slot is
// refilled as soon as it has been read; the addresses are worked out once per
// batch (kSliceBatch units).
template <int BLK>
struct SliceRing {
    uint8_t *slot;       // this thread's first slot
    int64_t g;           // the batch to be copied next: its group, first unit, the group's units
    int first, whole;
    static constexpr int kUnits = kSliceBatch * BLK;   // per batch
    __device__ __forceinline__ int units(const SliceArgs &a, const uint8_t *in, int64_t gq) const
    {
        if (gq >= a.NG || ((uintptr_t)in & 15)) return 0;
        return (int)min((int64_t)32, a.NT - 32 * gq) * a.KL / 16;
    }
    // the source of this thread's units of the next batch and how many units
    // are left from its first on; then on to the batch after it
    __device__ __forceinline__ const uint8_t *next(const SliceArgs &a, const uint8_t *__restrict__ in, int *left)
    {
        *left = whole - first - (int)threadIdx.x;
        const uint8_t *src = in + 32 * g * a.KL + 16 * (int64_t)(first + (int)threadIdx.x);
        first += kUnits;
        if (first >= whole) {
            g += gridDim.x;
            first = 0;
            whole = units(a, in, g);
        }
        return src;
    }
    __device__ __forceinline__ void copy(const uint8_t *src, int left, int k)
    {
        if (BLK * k < left)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(slot) + 16 * BLK * k), "l"(src + 16 * BLK * k)
                         : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    __device__ __forceinline__ void start(const SliceArgs &a, const uint8_t *__restrict__ in, void *ring)
    {
        slot = (uint8_t *)ring + 16 * threadIdx.x;
        g = blockIdx.x;
        first = 0;
        whole = units(a, in, g);
        int left;
        const uint8_t *src = next(a, in, &left);
#pragma unroll
        for (int k = 0; k < kSliceBatch; ++k) copy(src, left, k);
    }
    // the bit string of group gc (the groups in the order of the walk)
    __device__ __forceinline__ void string(const SliceArgs &a, const uint8_t *__restrict__ in, int64_t gc, uint32_t *B)
    {
        const int n = units(a, in, gc);
        for (int f = 0; f < n; f += kUnits) {
            int ahead;
            const uint8_t *src = next(a, in, &ahead);
            const uint4 *p = reinterpret_cast<const uint4 *>(slot);
            const int left = n - f - (int)threadIdx.x;
#pragma unroll
            for (int k = 0; k < kSliceBatch; ++k) {
                asm volatile("cp.async.wait_group %0;" ::"n"(kSliceBatch - 1) : "memory");
                if (BLK * k < left) slice_put16(a, B, f + (int)threadIdx.x + BLK * k, slice_bits16(p[BLK * k]));
                copy(src, ahead, k);
            }
        }
        const int bytes = (int)min((int64_t)32, a.NT - 32 * gc) * a.KL;
        slice_odd_units(a, in + 32 * gc * a.KL, bytes, n, B, threadIdx.x, BLK);
    }
};

// Chunk c of the string, transposed: lane p gets cell 32 c + p of the tiles.
__device__ __forceinline__ uint32_t slice_string_chunk(const SliceArgs &a, const Transpose32 &tr, const uint32_t *B, int c,
                                                       int nt, int lane)
{
    const uint32_t b = (uint32_t)lane * a.lane_bits + 32u * (uint32_t)c;
    const uint32_t *wp = B + (b >> 5);
    const uint32_t x = __funnelshift_r(wp[0], wp[1], b & 31u);
    return tr(lane < nt ? x : 0u);
}

// Bytes -> packed state: blocks walk the groups.  The cells of a group are
// contiguous in omega (32 k^L bytes, a multiple of 32 from the buffer's
// start); their bits go to shared memory in that order, and each warp then
// takes 32 cells of 32 tiles at a time through the transposition.  Bound by
// issue slots and the latency of its loads (carpet r = 10, 1.07e9 cells:
// 0.20 ms, 5.9 TB/s read and written).
template <int BLK>
__global__ void __launch_bounds__(BLK, BLK == kSliceBlock ? 6 : 3)
slice_pack_kernel(SliceArgs a, const uint8_t *__restrict__ in, uint32_t *__restrict__ bits)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const Transpose32 tr(lane);
    SliceRing<BLK> ring;
    ring.start(a, in, smem);
    uint32_t *B = smem + 4 * kSliceBatch * BLK;
    for (int64_t g = blockIdx.x; g < a.NG; g += gridDim.x) {
        const int nt = (int)min((int64_t)32, a.NT - 32 * g);
        ring.string(a, in, g, B);
        __syncthreads();
        uint32_t *dst = bits + g * a.KLp;
#pragma unroll 2
        for (int c = warp; c < a.NC; c += nw) {
            dst[32 * c + lane] = slice_string_chunk(a, tr, B, c, nt, lane);
        }
        __syncthreads();
        slice_export(a, tr, dst, bits + a.ex + g * a.XW * 32, warp, nw, lane);
    }
}

// ---------------------------------------------------------------- step

// Tile 32 g + lane's neighbour for halo word j, and the export word it sends.
__device__ __forceinline__ int32_t slice_nbr(const SliceArgs &a, int64_t g, uint32_t job, int lane)
{
    return __ldg(a.nbr + (g * a.ND + (job >> 8)) * 32 + lane);
}
__device__ __forceinline__ uint32_t slice_import(const SliceArgs &a, const uint32_t *ex, int32_t Q, uint32_t job)
{
    // (the exports may have been written by other blocks of this launch: loads go to L2)
    return Q < 0 ? 0u : __ldcg(ex + ((int64_t)(Q >> 5) * a.XW + (job & 0xffu)) * 32 + (Q & 31));
}

// The group's words into shared memory, asynchronously.
__device__ __forceinline__ void slice_load(const SliceArgs &a, uint32_t *A, const uint32_t *sg)
{
    for (int i = threadIdx.x; i < a.KLp / 4; i += blockDim.x)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(A + 4 * i)), "l"(sg + 4 * i) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// All blocks of the launch have arrived `n` times (n = 1, 2, ...): bounded.
__device__ __forceinline__ bool slice_grid_barrier(const SliceArgs &a, uint32_t n)
{
    __syncthreads();
    bool ok = true;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(a.bar, 1u);
        const uint32_t want = n * gridDim.x;
        ok = false;
        for (uint32_t i = 0; i < kWaitLimit; ++i) {
            uint32_t v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.bar) : "memory");
            if ((int32_t)(v - want) >= 0) {
                ok = true;
                break;
            }
        }
        if (!ok) atomicExch(a.status, FR_ETIMEOUT);
        __threadfence();
    }
    return __syncthreads_or(!ok) == 0;
}

// 32 cells of a group from cell o of its omega order on, from the tiles' bit
// strings (rows of RP words; bits past a tile's k^L cells are not defined).
__device__ __forceinline__ uint32_t slice_take32(const SliceArgs &a, const uint32_t *R, uint32_t o, uint32_t nt)
{
    uint32_t t = divu(a.kdiv, o), l = o - t * (uint32_t)a.KL;
    const uint32_t *p = R + t * (uint32_t)a.RP + (l >> 5);
    uint32_t x = __funnelshift_r(p[0], p[1], l & 31u);
    uint32_t have = (uint32_t)a.KL - l;   // cells of this tile from here on
    while (have < 32u && ++t < nt) {
        x = (x & ((1u << have) - 1u)) | R[t * (uint32_t)a.RP] << have;
        have += (uint32_t)a.KL;
    }
    return x;
}

// Byte J of x, a nibble -> 4 bytes of 0/1: the byte alone, a carry-free
// multiply, a mask.
template <int J>
__device__ __forceinline__ uint32_t slice_nib(uint32_t x)
{
    return (__byte_perm(x, 0u, 0x4440 | J) * 0x00204081u) & 0x01010101u;
}

// The new bytes of a group of nt tiles from the tiles' bit strings: 32 cells per thread.
__device__ __forceinline__ void slice_string_to_bytes(const SliceArgs &a, const uint32_t *R, uint8_t *__restrict__ ob, int nt,
                                                      int tid, int nth)
{
    const int bytes = nt * a.KL;
    const int whole = ((uintptr_t)ob & 15) == 0 ? bytes / 16 : 0;   // 16-byte units
    const int lane = tid & 31;
    // a warp's 32 x 32 cells; the lanes pass halves on so that consecutive
    // lanes store consecutive 16 bytes
#pragma unroll 2
    for (int i = tid - lane; 2 * i < whole; i += nth) {
        uint32_t x = 0u;
        if (2 * (i + lane) < whole) x = slice_take32(a, R, 32u * (uint32_t)(i + lane), (uint32_t)nt);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t y = __shfl_sync(0xffffffffu, x, 16 * h + (lane >> 1)) >> (16 * (lane & 1));
            const int u = 2 * i + 32 * h + lane;
            const uint32_t e = y & 0x0f0fu, o = (y >> 4) & 0x0f0fu;
            if (u < whole)
                __stcs(reinterpret_cast<uint4 *>(ob) + u,
                       make_uint4(slice_nib<0>(e), slice_nib<0>(o), slice_nib<1>(e), slice_nib<1>(o)));
        }
    }
    for (int i = 16 * whole + tid; i < bytes; i += nth) {
        const uint32_t t = divu(a.kdiv, (uint32_t)i), l = (uint32_t)i - t * (uint32_t)a.KL;
        ob[i] = (uint8_t)((R[t * (uint32_t)a.RP + (l >> 5)] >> (l & 31u)) & 1u);
    }
}

// A cell's row of the neighbour table: byte offsets of its neighbours' words,
// two per word; columns of 8, 8 and 4 (D = 20) or 8, 8, 8 and 2 (D = 26)
// neighbours, each contiguous over the cells.
template <int D>
struct SliceRow {
    uint32_t r[(D + 1) / 2];
    __device__ __forceinline__ void load(const SliceArgs &a, int i)
    {
        const uint4 v = __ldg(a.tab + i);
        r[0] = v.x;
        r[1] = v.y;
        if constexpr (D > 4) r[2] = v.z;
        if constexpr (D > 6) r[3] = v.w;
        if constexpr (D > 8) {
            const uint4 u = __ldg(a.tab + a.KLp + i);
            r[4] = u.x; r[5] = u.y; r[6] = u.z; r[7] = u.w;
            if constexpr (D == 20) {
                const uint2 x = __ldg(reinterpret_cast<const uint2 *>(a.tab + 2 * a.KLp) + i);
                r[8] = x.x; r[9] = x.y;
            } else {
                const uint4 x = __ldg(a.tab + 2 * a.KLp + i);
                r[8] = x.x; r[9] = x.y; r[10] = x.z; r[11] = x.w;
                r[12] = __ldg(reinterpret_cast<const uint32_t *>(a.tab + 3 * a.KLp) + i);
            }
        }
    }
};

// Next state of cells 32 c .. 32 c + 31 of a group's tiles from its words A.
template <int D, bool LIFE>
__device__ __forceinline__ uint32_t slice_next(const SliceArgs &a, const SliceRow<D> &row, const uint32_t *A, int c, int lane)
{
    uint32_t n[D < 8 ? 8 : D];
#pragma unroll
    for (int k = 0; k < D; ++k)
        n[k] = *reinterpret_cast<const uint32_t *>(reinterpret_cast<const uint8_t *>(A) +
                                                   ((k & 1) ? row.r[k / 2] >> 16 : row.r[k / 2] & 0xffffu));
    if constexpr (D > 8) return slice_rule3<D, LIFE>(a, n, A[32 * c + lane]);
    else return slice_rule<D, LIFE>(a, n, A[32 * c + lane]);
}

// In 3D a group's neighbour table (Menger: 8000 cells x 40 bytes) comes from
// L2 chunk by chunk; latency and issue slots bound it.  Menger r = 7 (1.28e9
// cells): one generation with packing 1.61 -> 0.70 ms, further ones 0.69 ->
// 0.31 ms each; r = 6 (250 groups, one or two per SM), 50 generations 1.96 ->
// 1.07 ms.

// `gens` generations of a packed state, blocks walking the groups; between
// generations the launch's blocks meet at a grid barrier (a cooperative
// launch when there is more than one block).  BYTES: one generation whose
// results leave as bytes.
template <int D, bool LIFE, bool BYTES>
__global__ void __launch_bounds__(D > 8 ? kSliceBlock3 : kSliceBlock, D > 8 ? 2 : (LIFE ? 5 : 4))
slice_step_kernel(SliceArgs a, const uint32_t *src, uint32_t *dst, uint8_t *__restrict__ out, int gens)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const Transpose32 tr(lane);
    constexpr bool kAhead = D <= 8;   // two arrays, the next group's words loaded ahead (3D: no room, two blocks per SM instead)
    uint32_t *R = smem + (kAhead ? 2 : 1) * a.AW;   // BYTES: the results' bit strings
    if (tid < (kAhead ? 64 : 32)) smem[(tid >> 5) * a.AW + a.A_zero + lane] = 0u;   // the words of absent neighbours
    uint32_t job[kSliceAhead];
#pragma unroll
    for (int i = 0; i < kSliceAhead; ++i) job[i] = warp + i * nw < a.NJ ? __ldg(a.jobs + warp + i * nw) : 0u;
    uint32_t buf = 0;
    for (int gen = 0; gen < gens; ++gen) {
        uint32_t e[kSliceAhead];   // halo words of the next group, loaded ahead
        if (blockIdx.x < a.NG) {
            slice_load(a, smem + buf * a.AW, src + (int64_t)blockIdx.x * a.KLp);
#pragma unroll
            for (int i = 0; i < kSliceAhead; ++i)
                e[i] = warp + i * nw < a.NJ ? slice_import(a, src + a.ex, slice_nbr(a, blockIdx.x, job[i], lane), job[i]) : 0u;
        }
        for (int64_t g = blockIdx.x; g < a.NG; g += gridDim.x, buf ^= kAhead ? 1u : 0u) {
            uint32_t *A = smem + buf * a.AW;
            const int64_t gn = g + gridDim.x;
#pragma unroll
            for (int i = 0; i < kSliceAhead; ++i)
                if (warp + i * nw < a.NJ) A[a.KLp + 32 * (warp + i * nw) + lane] = tr(e[i]);
#pragma unroll 4
            for (int j = warp + kSliceAhead * nw; j < a.NJ; j += nw) {
                const uint32_t jb = __ldg(a.jobs + j);
                A[a.KLp + 32 * j + lane] = tr(slice_import(a, src + a.ex, slice_nbr(a, g, jb, lane), jb));
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            int32_t Q[kSliceAhead];
            if (gn < a.NG) {
                if (kAhead) slice_load(a, smem + (buf ^ 1) * a.AW, src + gn * a.KLp);
#pragma unroll
                for (int i = 0; i < kSliceAhead; ++i) Q[i] = warp + i * nw < a.NJ ? slice_nbr(a, gn, job[i], lane) : -1;
            }
            uint32_t *dg = BYTES ? nullptr : dst + g * a.KLp;
#pragma unroll 2
            for (int c = warp; c < a.NC; c += nw) {
                SliceRow<D> row;
                row.load(a, 32 * c + lane);
                const uint32_t w = slice_next<D, LIFE>(a, row, A, c, lane);
                if (BYTES) {
                    R[lane * a.RP + c] = tr(w);
                } else {
                    dg[32 * c + lane] = w;
                }
            }
            if (gn < a.NG) {
#pragma unroll
                for (int i = 0; i < kSliceAhead; ++i) e[i] = slice_import(a, src + a.ex, Q[i], job[i]);
            }
            __syncthreads();
            if (!kAhead && gn < a.NG) slice_load(a, smem, src + gn * a.KLp);   // (this group's words have been read)
            if (BYTES) {
                slice_string_to_bytes(a, R, out + 32 * g * a.KL, (int)min((int64_t)32, a.NT - 32 * g), tid, blockDim.x);
            } else {
                slice_export(a, tr, dg, dst + a.ex + g * a.XW * 32, warp, nw, lane);
            }
        }
        if (!BYTES && gen + 1 < gens) {
            if (gridDim.x > 1) {
                if (!slice_grid_barrier(a, (uint32_t)gen + 1u)) break;
            } else {
                __syncthreads();
            }
            const uint32_t *t = src;
            src = dst;
            dst = const_cast<uint32_t *>(t);
        }
    }
    if (!BYTES && gens > 1 && gridDim.x > 1 && tid == 0) {
        // the last block to leave resets the barrier for the next launch
        if (atomicAdd(a.bar + 1, 1u) == gridDim.x - 1) {
            a.bar[0] = 0u;
            a.bar[1] = 0u;
            __threadfence();
        }
    }
}

// One generation from bytes to bytes in one pass, for fractals whose tiles
// have a halo of at most 32 cells (the triangle 8, the Vicsek fractal 4):
// those cells are read as bytes from the neighbouring tiles (lane t follows
// tile 32 g + t, a ballot makes the word), the rest as in the two-pass
// kernels.  The bit strings of the old and of the new state share a place.
// Issue-bound (67 % of the slots, HBM at 80 %): triangle r = 20 in 1.29 ms
// against 1.49 ms of the tap kernel and 1.45 ms of the two-pass kernels.
// Tiles of 2187 cells: with 729 it took 1.57 ms (a group's fixed work, about
// 1600 instructions, per fewer cells), with 6561 1.72 ms (the neighbour table
// no longer stays near the SM).
template <int D, bool LIFE>
__global__ void __launch_bounds__(kSliceBlock, LIFE ? 5 : 4)
slice_single_kernel(SliceArgs a, const uint8_t *__restrict__ in, uint8_t *__restrict__ out)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const Transpose32 tr(lane);
    SliceRing<kSliceBlock> ring;
    ring.start(a, in, smem);
    uint32_t *A = smem + 4 * kSliceBatch * kSliceBlock, *B = A + a.AW;
    if (tid < 32) A[a.A_zero + tid] = 0u;   // the words of absent neighbours
    // this warp's first halo cell of the next group, loaded ahead
    const uint2 h0 = warp < a.H ? __ldg(a.cells + warp) : make_uint2(0u, 0u);
    uint32_t hv = 0u;
    auto halo = [&](int64_t g, uint2 h) -> uint32_t {
        const int32_t Q = __ldg(a.nbr + (g * 8 + (h.y >> 16)) * 32 + lane);
        return Q < 0 ? 0u : (uint32_t)__ldg(in + (int64_t)Q * a.KL + h.x);
    };
    if (warp < a.H && blockIdx.x < a.NG) hv = halo(blockIdx.x, h0);
    for (int64_t g = blockIdx.x; g < a.NG; g += gridDim.x) {
        const int nt = (int)min((int64_t)32, a.NT - 32 * g);
        const int64_t gn = g + gridDim.x;
        ring.string(a, in, g, B);
        if (warp < a.H) {
            const uint32_t b = __ballot_sync(0xffffffffu, hv != 0u);
            if (lane == 0) A[h0.y & 0xffffu] = b;
            if (gn < a.NG) hv = halo(gn, h0);
        }
        for (int h = warp + nw; h < a.H; h += nw) {
            const uint2 e = __ldg(a.cells + h);
            const uint32_t b = __ballot_sync(0xffffffffu, halo(g, e) != 0u);
            if (lane == 0) A[e.y & 0xffffu] = b;
        }
        __syncthreads();
#pragma unroll 2
        for (int c = warp; c < a.NC; c += nw) A[32 * c + lane] = slice_string_chunk(a, tr, B, c, nt, lane);
        __syncthreads();
#pragma unroll 2
        for (int c = warp; c < a.NC; c += nw) {
            SliceRow<D> row;
            row.load(a, 32 * c + lane);
            B[lane * a.RP + c] = tr(slice_next<D, LIFE>(a, row, A, c, lane));
        }
        __syncthreads();
        slice_string_to_bytes(a, B, out + 32 * g * a.KL, nt, tid, blockDim.x);
        __syncthreads();
    }
}

// States whose packed words fit in the SMs' shared memory together: one
// launch packs the bytes, runs all generations and writes the bytes.  A block
// owns fixed groups, whose words stay in shared memory and are replaced in
// place (the new words wait in registers until the block has read the old
// ones; the groups' bit strings of the first and the last step take the same
// place); only the exports go through memory (ex0 / ex1 in turn), with a grid
// barrier per generation.  The neighbour table, the export lists and the
// places of the tiles' halo words in the exports are kept in shared memory as
// well: with so much of it in use little is left of L1.  ONE: a single block;
// its exports stay in shared memory too.  Bound by issue slots and, for small
// states, by the barrier and the chain of latencies around it.  Microseconds
// per call, byte-wise tile kernels -> here: triangle r = 8, 100 generations
// 614 -> 52, r = 16, 50 generations 1151 -> 331, carpet r = 9, 20 generations
// 1950 -> 328, H-fractal r = 9, 4 generations 426 -> 52.

// A block's items (item j of its group q, n per group) dealt to its warps, a
// run of `rounds` items each; past the last item a warp repeats it.
struct SliceWalk {
    int q, j, n, groups;
    __device__ __forceinline__ SliceWalk(int n_, const DivU32 &ndiv, int groups_, int first)
        : q(n_ > 1 ? (int)divu(ndiv, (uint32_t)first) : first), n(n_), groups(groups_)
    {
        j = first - q * n;
        clamp();
    }
    __device__ __forceinline__ void clamp()
    {
        if (q >= groups) {
            q = groups - 1;
            j = n - 1;
        }
    }
    __device__ __forceinline__ void next()
    {
        if (++j == n) {
            j = 0;
            ++q;
            clamp();
        }
    }
};

template <int D, bool LIFE, bool ONE, int ROUNDS, bool BATCH>
__global__ void __launch_bounds__(1024, 1)
slice_resident_kernel(SliceArgs a, const uint8_t *__restrict__ in, uint8_t *__restrict__ out, uint32_t *ex0, uint32_t *ex1,
                      int per_block, int64_t steps)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
    const Transpose32 tr(lane);
    uint4 *tab = reinterpret_cast<uint4 *>(smem);
    uint32_t *exs = smem + 4 * a.KLp;   // ONE: both export buffers
    const int exw = ONE ? (int)a.NG * a.XW * 32 : 0;
    uint16_t *xlist = reinterpret_cast<uint16_t *>(exs + 2 * exw);
    int32_t *from = reinterpret_cast<int32_t *>(exs + 2 * exw + a.XW * 16);
    int32_t *left = from + per_block * a.NJ * 32;   // generations of the block's groups, decreasing
    uint32_t *A0 = reinterpret_cast<uint32_t *>(left + per_block);
    if (ONE) {
        ex0 = exs;
        ex1 = exs + exw;
    }
    const int64_t g0 = blockIdx.x, gs = gridDim.x;
    const int mine = (int)min((int64_t)per_block, (a.NG - g0 + gs - 1) / gs);   // this block's groups
    const int rounds = (mine * a.NC + nw - 1) / nw;
    for (int i = tid; i < a.KLp; i += nth) tab[i] = __ldg(a.tab + i);
    for (int i = tid; i < a.XW * 32; i += nth) xlist[i] = __ldg(a.xlist + i);
    for (int x = warp; x < mine * a.NJ; x += nw) {
        const int q = x / a.NJ;
        const uint32_t jb = __ldg(a.jobs + (x - q * a.NJ));
        const int32_t Q = slice_nbr(a, g0 + q * gs, jb, lane);
        from[x * 32 + lane] = Q < 0 ? -1 : ((Q >> 5) * a.XW + (int)(jb & 0xffu)) * 32 + (Q & 31);
    }
    auto tiles = [&](int64_t g) { return BATCH ? a.groups[g].nt : (int)min((int64_t)32, a.NT - 32 * g); };
    if (BATCH)
        for (int q = tid; q < mine; q += nth) left[q] = a.groups[g0 + q * gs].steps;
    for (int q = 0; q < mine; ++q) {
        const int64_t g = g0 + q * gs;
        slice_bytes_to_string(a, BATCH ? a.groups[g].in : in + 32 * g * a.KL, tiles(g), A0 + q * a.AW, tid, nth);
    }
    __syncthreads();
    uint32_t w[ROUNDS];
    {
        // (bits of tiles past a group's last are never read by others)
        SliceWalk k(a.NC, a.cdiv, mine, warp * rounds);
#pragma unroll
        for (int i = 0; i < ROUNDS; ++i)
            if (i < rounds) {
                w[i] = slice_string_chunk(a, tr, A0 + k.q * a.AW, k.j, 32, lane);
                k.next();
            }
    }
    __syncthreads();
    for (int q = warp; q < mine; q += nw) A0[q * a.AW + a.A_zero + lane] = 0u;   // the words of absent neighbours
    // groups with generations left (the first ones; all of them unless BATCH) and the rounds their items take
    int active = mine, now = rounds, im_n = (mine * a.NJ + nw - 1) / nw, ex_n = (mine * a.XW + nw - 1) / nw;
    const SliceWalk chunks0(a.NC, a.cdiv, mine, warp * rounds), im0(max(a.NJ, 1), a.jdiv, mine, warp * im_n),
        ex0w(max(a.XW, 1), a.xdiv, mine, warp * ex_n);
    auto chunk_walk = [&]() { return BATCH ? SliceWalk(a.NC, a.cdiv, active, warp * now) : chunks0; };
    // the new words of the first `groups` groups
    auto put_words = [&](int groups) {
        SliceWalk k = chunk_walk();
#pragma unroll
        for (int i = 0; i < ROUNDS; ++i)
            if (i < now) {
                if (!BATCH || k.q < groups) A0[k.q * a.AW + 32 * k.j + lane] = w[i];
                k.next();
            }
    };
    // the bit strings of the groups from `from` on
    auto put_strings = [&](int first) {
        SliceWalk k = chunk_walk();
#pragma unroll
        for (int i = 0; i < ROUNDS; ++i)
            if (i < now) {
                if (!BATCH || k.q >= first) A0[k.q * a.AW + lane * a.RP + k.j] = tr(w[i]);
                k.next();
            }
    };
    auto put_exports = [&](int groups, uint32_t *ex) {
        if (BATCH && groups == 0) return;
        if (BATCH && groups != active) ex_n = (groups * a.XW + nw - 1) / nw;
        SliceWalk k = BATCH ? SliceWalk(max(a.XW, 1), a.xdiv, groups, warp * ex_n) : ex0w;
        for (int i = 0; i < ex_n; ++i, k.next()) {
            const uint32_t v = tr(A0[k.q * a.AW + xlist[32 * k.j + lane]]);
            if (ONE) ex[(k.q * a.XW + k.j) * 32 + lane] = v;
            else __stcg(ex + ((g0 + k.q * gs) * a.XW + k.j) * 32 + lane, v);
        }
    };
    auto put_bytes = [&](int first, int end) {
        for (int q = first; q < end; ++q) {
            const int64_t g = g0 + q * gs;
            slice_string_to_bytes(a, A0 + q * a.AW, BATCH ? a.groups[g].out : out + 32 * g * a.KL, tiles(g), tid, nth);
        }
    };
    put_words(mine);
    __syncthreads();
    put_exports(mine, ex0);
    for (int64_t gen = 1; gen <= steps; ++gen) {
        // everybody's exports of the state before this generation are there
        if (ONE) __syncthreads();
        else if (!slice_grid_barrier(a, (uint32_t)gen)) break;
        if (BATCH && active == 0) continue;
        int going = active;   // groups with more generations after this one
        if (BATCH)
            while (going > 0 && left[going - 1] == gen) --going;
        const uint32_t *ei = (gen & 1) ? ex0 : ex1;
        {
            SliceWalk k = BATCH ? SliceWalk(max(a.NJ, 1), a.jdiv, active, warp * im_n) : im0;
#pragma unroll 2
            for (int i = 0; i < im_n; ++i, k.next()) {
                const int at = from[(k.q * a.NJ + k.j) * 32 + lane];
                uint32_t e = 0u;
                if (at >= 0) e = ONE ? ei[at] : __ldcg(ei + at);
                A0[k.q * a.AW + a.KLp + 32 * k.j + lane] = tr(e);
            }
        }
        __syncthreads();
        {
            SliceWalk k = chunk_walk();
#pragma unroll
            for (int i = 0; i < ROUNDS; ++i)
                if (i < now) {
                    const uint4 v = tab[32 * k.j + lane];
                    SliceRow<D> row;
                    row.r[0] = v.x;
                    row.r[1] = v.y;
                    if constexpr (D > 4) row.r[2] = v.z;
                    if constexpr (D > 6) row.r[3] = v.w;
                    w[i] = slice_next<D, LIFE>(a, row, A0 + k.q * a.AW, k.j, lane);
                    k.next();
                }
        }
        __syncthreads();
        if (BATCH ? going > 0 : gen < steps) {
            put_words(going);
            if (!BATCH) {
                __syncthreads();
                put_exports(mine, (gen & 1) ? ex1 : ex0);
            }
        }
        if (BATCH) {
            if (going < active) put_strings(going);   // the last generation of some groups
            __syncthreads();
            put_exports(going, (gen & 1) ? ex1 : ex0);
            if (going < active) {
                put_bytes(going, active);
                active = going;
                now = (active * a.NC + nw - 1) / nw;
                im_n = (active * a.NJ + nw - 1) / nw;
                ex_n = (active * a.XW + nw - 1) / nw;
            }
        }
    }
    if (!BATCH) {
        put_strings(0);
        __syncthreads();
        put_bytes(0, mine);
    }
    if (!ONE && tid == 0) {
        // the last block to leave resets the barrier for the next launch
        if (atomicAdd(a.bar + 1, 1u) == gridDim.x - 1) {
            a.bar[0] = 0u;
            a.bar[1] = 0u;
            __threadfence();
        }
    }
}

// Neighbours of every tile, a row of 32 lanes per group and direction (tiles
// past the last have none).  A move changes the lowest digit, and goes on one
// level up in the direction it leaves the block in; most end after a digit or
// two, where lambda and nu would decode every level of every neighbour: first
// call of the triangle at r = 20 (1.6 million tiles) 2.10 -> 1.88 ms.
template <int DIM>
__global__ void __launch_bounds__(256) slice_nbr_kernel(FracDev F, int64_t NT, int64_t NG, int levels,
                                                        const SliceGroup *__restrict__ groups, int32_t *__restrict__ out)
{
    constexpr int Q = DIM == 3 ? 27 : 9, ND = Q - 1;
    extern __shared__ int16_t moved[];   // [k][Q]: a replica's neighbour | the direction left to move one level up << 8, or -1
    for (int i = threadIdx.x; i < F.k * Q; i += blockDim.x) {
        const int j = i / Q;
        int d = i - j * Q, t = 0, w = 1, up = 0, w3 = 1;
        for (int a = 0; a < DIM; ++a) {
            const int q = F.off[j][a] + d % 3 - 1, b = q < 0 ? -1 : (q >= F.s ? 1 : 0);
            t += (q - b * F.s) * w;
            up += (b + 1) * w3;
            w *= F.s;
            w3 *= 3;
            d /= 3;
        }
        moved[i] = F.hinv[t] < 0 ? (int16_t)-1 : (int16_t)(F.hinv[t] | up << 8);
    }
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 32 * NG; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t T = i, base = 0;
        bool live = T < NT;
        if (groups) {   // a batch: the tile's place in its instance, whose tiles start at group group0
            const SliceGroup s = groups[i >> 5];
            live = (i & 31) < s.nt;
            T = s.tile0 + (i & 31);
            base = 32 * (int64_t)s.group0;
            levels = s.levels;
        }
        for (int d = 0; d < ND; ++d) {
            int dir = live ? (d < ND / 2 ? d : d + 1) : -1;
            uint32_t rest = (uint32_t)T, below = 0, w = 1;
            for (int l = 0; l < levels && dir >= 0 && dir != Q / 2; ++l) {
                const uint32_t q = divu(F.kdiv, rest);
                const int e = moved[(rest - q * (uint32_t)F.k) * Q + dir];
                below += (uint32_t)(e & 0xff) * w;
                w *= (uint32_t)F.k;
                rest = q;
                dir = e >> 8;
            }
            // (a move left over at the top leaves the box)
            out[((i >> 5) * ND + d) * 32 + (i & 31)] = dir == Q / 2 ? (int32_t)(base + below + rest * w) : -1;
        }
    }
}

// ---------------------------------------------------------------- plan

static int64_t pw(int64_t b, int e)
{
    int64_t v = 1;
    for (int i = 0; i < e; ++i) v *= b;
    return v;
}

// Neighbours of the cells of an m-level box: entry [l][q] (q = (dx + 1) + 3
// (dy + 1) + 9 (dz + 1), Q = 9 or 27 of them) is the neighbour's number in the
// box that holds it | that box's direction << 24 (Q / 2: the same box), or -1
// where the fractal has none.
using SliceNbrs = std::vector<int32_t>;

// One level more: level 0 digits move as `first` says, and where they leave
// their block the rest moves as it does with m - 1 levels.
static SliceNbrs slice_deepen(const SliceNbrs &first, const SliceNbrs &rest, int k, int Q)
{
    const size_t n = rest.size() / Q;
    SliceNbrs out(n * k * Q);
    for (size_t r = 0; r < n; ++r)
        for (int j = 0; j < k; ++j)
            for (int d = 0; d < Q; ++d) {
                const int32_t a = first[(size_t)j * Q + d];
                int32_t v = -1;
                if (a >= 0) {
                    const int32_t b = (a >> 24) == Q / 2 ? (int32_t)r | (Q / 2) << 24 : rest[r * Q + (a >> 24)];
                    if (b >= 0) v = ((b & 0xffffff) * k + (a & 0xffffff)) | (b & ~0xffffff);
                }
                out[(r * k + j) * Q + d] = v;
            }
    return out;
}

// The neighbours in a single block of s^dim digits.
static SliceNbrs slice_first(const fractal *f)
{
    const int Q = f->dim == 3 ? 27 : 9;
    SliceNbrs out((size_t)f->k * Q, -1);
    for (int j = 0; j < f->k; ++j)
        for (int d = 0; d < Q; ++d) {
            const int m[3] = {d % 3 - 1, (d / 3) % 3 - 1, d / 9 - 1};
            int t = 0, w = 1, box = 0, b3 = 1;
            for (int i = 0; i < f->dim; ++i) {
                int q = f->offsets[(size_t)f->dim * j + i] + m[i];
                const int b = q < 0 ? -1 : (q >= f->s ? 1 : 0);
                t += (q - b * f->s) * w;
                w *= f->s;
                box += (b + 1) * b3;
                b3 *= 3;
            }
            const int h = f->dev.hinv[t];
            if (h >= 0) out[(size_t)j * Q + d] = h | box << 24;
        }
    return out;
}

struct SliceTables {
    int KL = 0, H = 0, D = 0;
    int zero = 0;                   // the first of 32 zero words in a group's array
    SliceNbrs nb;
    int Q = 9;                      // directions and the centre
    std::vector<int32_t> hidx;      // [Q][KL]: word of a halo cell (by its box's direction), -1 = none
    std::vector<uint32_t> jobs;     // halo words: export word | direction slot << 8
    std::vector<uint16_t> xlist;    // [XW][32] cells of the export words
    std::vector<uint32_t> cells;    // halo cells: cell of the neighbouring tile, word index | direction slot << 16
    int XW() const { return (int)xlist.size() / 32; }
};

static SliceTables slice_tables(SliceNbrs &&nbrs, int Q)
{
    SliceTables t;
    t.Q = Q;
    t.nb = std::move(nbrs);
    t.KL = (int)(t.nb.size() / Q);
    const int KL = t.KL, KLp = (KL + 31) / 32 * 32;
    t.hidx.assign((size_t)Q * KL, -1);
    for (int l = 0; l < KL; ++l) {
        int n = 0;
        for (int d = 0; d < Q; ++d) {
            const int32_t v = d == Q / 2 ? -1 : t.nb[(size_t)l * Q + d];
            if (v < 0) continue;
            ++n;
            if ((v >> 24) != Q / 2) t.hidx[(size_t)(v >> 24) * KL + (v & 0xffffff)] = 0;
        }
        t.D = std::max(t.D, n);
    }
    // export words: the directions with the most border cells first, their
    // cells in runs of 32; a run whose cells all lie in an earlier word uses
    // that one (a corner cell is in its sides' words)
    std::vector<int> cells[27];
    std::vector<int> order;
    for (int d = 0; d < Q; ++d)
        if (d != Q / 2) order.push_back(d);
    for (int d : order)
        for (int l = 0; l < KL; ++l)
            if (t.hidx[(size_t)d * KL + l] >= 0) cells[d].push_back(l);
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cells[x].size() > cells[y].size(); });
    std::vector<std::vector<int>> words;
    for (int d : order)
        for (size_t i = 0; i < cells[d].size(); i += 32) {
            const std::vector<int> run(cells[d].begin() + i, cells[d].begin() + std::min(i + 32, cells[d].size()));
            int w = -1;
            for (int x = 0; x < (int)words.size() && w < 0; ++x)
                if (words[x].size() >= run.size() && words[x].front() <= run.front() && words[x].back() >= run.back() &&
                    std::includes(words[x].begin(), words[x].end(), run.begin(), run.end())) w = x;
            if (w < 0) {
                w = (int)words.size();
                words.push_back(run);
            }
            const uint32_t slot = (uint32_t)(d < Q / 2 ? d : d - 1);
            for (int l : run) {
                const int at = KLp + 32 * (int)t.jobs.size() +
                               (int)(std::lower_bound(words[w].begin(), words[w].end(), l) - words[w].begin());
                t.hidx[(size_t)d * KL + l] = at;
                t.cells.push_back((uint32_t)l);
                t.cells.push_back((uint32_t)at | slot << 16);
            }
            t.jobs.push_back((uint32_t)w | slot << 8);
            t.H += (int)run.size();
        }
    for (const auto &w : words)
        for (int i = 0; i < 32; ++i) t.xlist.push_back((uint16_t)w[std::min<size_t>(i, w.size() - 1)]);
    t.zero = KLp + std::max(32 * (int)t.jobs.size(), 64);
    return t;
}

// The neighbour table (byte offsets): the 32 cells of a chunk are
// added by 32 lanes, one neighbour per lane and load, and the order of a
// cell's neighbours is free; each goes to the load that has the fewest words
// in its bank so far (triangle: 9.4 -> 6.0 shared-memory wavefronts per chunk,
// carpet 14.6 -> 8.6).  The loads a cell has no neighbour for read a zero word
// from the emptiest bank.
static void slice_neighbour_table(const SliceTables &t, int D, uint16_t *tab)
{
    const int KLp = (t.KL + 31) / 32 * 32, Q = t.Q;
    const uint32_t all = (1u << D) - 1u;
    // entry k of cell i is at col[k] + i * step[k]: columns of 8, the last of 4 or 2 (see SliceRow)
    const int entries = D <= 8 ? 8 : D;
    size_t col[26], step[26];
    for (int k = 0; k < entries; ++k) {
        step[k] = D > 8 && k / 8 == (D - 1) / 8 ? (D == 20 ? 4 : 2) : 8;
        col[k] = (size_t)(k / 8) * 8 * KLp + k % 8;
    }
    std::vector<uint32_t> loaded((size_t)t.zero + 32, 0);   // per word: the loads of this chunk that read it
    for (int c = 0; c < KLp; c += 32) {
        // [bank][x]: the loads that read x words of the bank, as a bit set; per load: the banks it reads
        uint32_t with[32][33], used[26] = {};
        int v[32][26], put[32][26], n[32], top[32];
        for (int b = 0; b < 32; ++b) {
            with[b][0] = all;
            top[b] = 0;
        }
        int by_count[27][32], many[27] = {};
        for (int i = 0; i < 32; ++i) {
            n[i] = 0;
            if (c + i < t.KL) {
                const int32_t *nb = &t.nb[(size_t)(c + i) * Q];
                for (int d = 0; d < Q; ++d)
                    if (nb[d] >= 0 && d != Q / 2)
                        v[i][n[i]++] = (nb[d] >> 24) == Q / 2 ? nb[d] & 0xffffff
                                                              : t.hidx[(size_t)(nb[d] >> 24) * t.KL + (nb[d] & 0xffffff)];
            }
            by_count[n[i]][many[n[i]]++] = i;
        }
        for (int want = D; want >= 1; --want)   // cells with the most neighbours first
            for (int m = 0; m < many[want]; ++m) {
                const int i = by_count[want][m];
                uint32_t open = all;
                for (int e = 0; e < want; ++e) {
                    const int w = v[i][e], b = w & 31;
                    uint32_t pick = open & loaded[w];
                    if (!pick) {
                        int x = 0;
                        while (!(pick = open & with[b][x])) ++x;
                        pick &= 0u - pick;
                        if (x == top[b]) with[b][++top[b]] = 0u;
                        with[b][x] &= ~pick;
                        with[b][x + 1] |= pick;
                        loaded[w] |= pick;
                    }
                    pick &= 0u - pick;
                    open &= ~pick;
                    put[i][e] = __builtin_ctz(pick);
                    used[put[i][e]] |= 1u << b;
                }
            }
        for (int k = 0; k < entries; ++k) {
            // the zero word in a bank the load does not read, where there is one
            const uint32_t free = k < D ? ~used[k] : ~0u;
            const uint16_t z = (uint16_t)(4 * (t.zero + (free ? (__builtin_ctz(free) - t.zero) & 31 : 0)));
            uint16_t *p = tab + col[k] + (size_t)c * step[k];
            for (int i = 0; i < 32; ++i) p[i * step[k]] = z;
        }
        for (int i = 0; i < 32; ++i)
            for (int e = 0; e < n[i]; ++e) {
                tab[col[put[i][e]] + (size_t)(c + i) * step[put[i][e]]] = (uint16_t)(4 * v[i][e]);
                loaded[v[i][e]] = 0;
            }
    }
}

// The tables of a transition table at a tile depth, and their device layout.
struct SliceImage {
    SliceTables t;
    std::once_flag once;
    std::vector<uint16_t> tab;   // neighbour table, made when first wanted
    size_t bytes = 0;
    const std::vector<uint16_t> &neighbours(int D)
    {
        std::call_once(once, [&]() {
            tab.resize((size_t)((t.KL + 31) / 32 * 32) * (D <= 8 ? 8 : (D == 20 ? 20 : 26)));
            slice_neighbour_table(t, D, tab.data());
        });
        return tab;
    }
};

// They depend on the transition table alone, take milliseconds to make in 3D
// and serve every handle of that fractal at any level: the most recently used
// ones are kept (at most kSliceImageBytes of them), and handles that are being
// planned hold what they use themselves.
constexpr size_t kSliceImageBytes = (size_t)32 << 20;
static std::mutex g_image_mu;
static std::list<std::pair<std::string, std::shared_ptr<SliceImage>>> g_images;   // the latest first

static std::shared_ptr<SliceImage> slice_image(const fractal *f, int L)
{
    std::string key = std::to_string(f->dim) + "," + std::to_string(f->s) + "," + std::to_string(L) + "|";
    for (int32_t v : f->offsets) key += std::to_string(v) + ",";
    {
        std::lock_guard<std::mutex> lk(g_image_mu);
        for (auto it = g_images.begin(); it != g_images.end(); ++it)
            if (it->first == key) {
                g_images.splice(g_images.begin(), g_images, it);
                return it->second;
            }
    }
    const int Q = f->dim == 3 ? 27 : 9;
    SliceNbrs nbrs = slice_first(f);
    if (L > 1) nbrs = slice_deepen(nbrs, slice_image(f, L - 1)->t.nb, f->k, Q);
    auto img = std::make_shared<SliceImage>();
    img->t = slice_tables(std::move(nbrs), Q);
    img->bytes = (size_t)img->t.KL * (Q * 8 + 52) + 4096;
    std::lock_guard<std::mutex> lk(g_image_mu);
    g_images.emplace_front(key, img);
    size_t total = 0;
    for (auto it = g_images.begin(); it != g_images.end();) {
        total += it->second->bytes;
        if (total > kSliceImageBytes && it != g_images.begin()) it = g_images.erase(it);
        else ++it;
    }
    return img;
}

void free_slice_plan(SlicePlan &p)
{
    cudaFree(p.arena);
    for (uint8_t *m : p.packed) cudaFree(m);
    p = SlicePlan();
}

using StepFn = void (*)(SliceArgs, const uint32_t *, uint32_t *, uint8_t *, int);

template <int D>
static StepFn step_fn_d(bool life, bool bytes)
{
    if (bytes) return life ? slice_step_kernel<D, true, true> : slice_step_kernel<D, false, true>;
    return life ? slice_step_kernel<D, true, false> : slice_step_kernel<D, false, false>;
}

static StepFn step_fn(int D, bool life, bool bytes)
{
    switch (D) {
        case 4: return step_fn_d<4>(life, bytes);
        case 6: return step_fn_d<6>(life, bytes);
        case 7: return step_fn_d<7>(life, bytes);
        case 8: return step_fn_d<8>(life, bytes);
        case 20: return step_fn_d<20>(life, bytes);
        default: return step_fn_d<26>(life, bytes);
    }
}

using SingleFn = void (*)(SliceArgs, const uint8_t *, uint8_t *);

static SingleFn single_fn(int D, bool life)
{
    switch (D) {
        case 4: return life ? slice_single_kernel<4, true> : slice_single_kernel<4, false>;
        case 6: return life ? slice_single_kernel<6, true> : slice_single_kernel<6, false>;
        case 7: return life ? slice_single_kernel<7, true> : slice_single_kernel<7, false>;
        default: return life ? slice_single_kernel<8, true> : slice_single_kernel<8, false>;
    }
}

using ResidentFn = void (*)(SliceArgs, const uint8_t *, uint8_t *, uint32_t *, uint32_t *, int, int64_t);

// rounds: 32-cell chunks per warp
template <int D, bool LIFE>
static ResidentFn resident_fn_d(const SlicePlan &s)
{
    if (s.groups) return s.rounds <= 8 ? slice_resident_kernel<D, LIFE, false, 8, true> : slice_resident_kernel<D, LIFE, false, kSliceRounds, true>;
    if (s.grid_resident == 1)
        return s.rounds <= 1 ? slice_resident_kernel<D, LIFE, true, 1, false> : slice_resident_kernel<D, LIFE, true, 8, false>;
    if (s.rounds <= 8) return slice_resident_kernel<D, LIFE, false, 8, false>;
    if (s.rounds <= 20) return slice_resident_kernel<D, LIFE, false, 20, false>;
    return slice_resident_kernel<D, LIFE, false, kSliceRounds, false>;
}

static ResidentFn resident_fn(const SlicePlan &s, bool life)
{
    switch (s.geo.D) {
        case 4: return life ? resident_fn_d<4, true>(s) : resident_fn_d<4, false>(s);
        case 6: return life ? resident_fn_d<6, true>(s) : resident_fn_d<6, false>(s);
        case 7: return life ? resident_fn_d<7, true>(s) : resident_fn_d<7, false>(s);
        default: return life ? resident_fn_d<8, true>(s) : resident_fn_d<8, false>(s);
    }
}

static bool slice_fractal_ok(const fractal *f) { return !f->mixed && f->k >= 2 && f->r >= 1; }

// Whether the rule is the one the kernels have a closed form for: B3/S23, in 3D B5/S45.
static bool slice_life(const fractal *f, uint32_t birth, uint32_t survive)
{
    if (f->dim == 3) return (birth & 0x7ffffffu) == 0x20u && (survive & 0x7ffffffu) == 0x30u;
    return (birth & 0x1ffu) == 0x8u && (survive & 0x1ffu) == 0xcu;
}

// The resident kernels of the plan may use its shared memory, a block per SM.
static cudaError_t resident_ready(const SlicePlan &s)
{
    cudaError_t e = cudaSuccess;
    for (int life = 0; life < 2 && e == cudaSuccess; ++life) {
        ResidentFn fn = resident_fn(s, life);
        int per_sm = 0;
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSliceSmem);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, s.block_resident, s.smem_resident);
        if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
    }
    return e;
}

static int launch_resident(const SlicePlan &s, const SliceArgs &a, bool life, const uint8_t *in, uint8_t *out, int64_t steps,
                           cudaStream_t st)
{
    ResidentFn fn = resident_fn(s, life);
    uint32_t *e0 = steps == 1 ? s.ex[2] : s.ex[0], *e1 = s.ex[1];   // (one generation writes e0 alone)
    int per_block = s.per_block;
    void *args[] = {(void *)&a, &in, &out, &e0, &e1, &per_block, &steps};
    if (s.grid_resident > 1)
        FR_CUDA(cudaLaunchCooperativeKernel((const void *)fn, dim3(s.grid_resident), dim3(s.block_resident), args, s.smem_resident, st));
    else
        FR_CUDA(cudaLaunchKernel((const void *)fn, dim3(1), dim3(s.block_resident), args, s.smem_resident, st));
    return FR_OK;
}

// Geometry of the tables of one tile depth.
static SliceGeo slice_geo(const fractal *f, int L, const SliceTables &t)
{
    SliceGeo p;
    p.L = L;
    p.KL = t.KL;
    p.NC = (t.KL + 31) / 32;
    p.KLp = 32 * p.NC;
    p.NJ = (int)t.jobs.size();
    p.XW = t.XW();
    p.H = t.H;
    p.ND = t.Q - 1;
    p.D = t.Q == 27 ? (t.D <= 20 ? 20 : 26) : (t.D <= 4 ? 4 : (t.D <= 6 ? 6 : t.D));
    p.NT = pw(f->k, f->r - L);
    p.NG = (p.NT + 31) / 32;
    p.AW = p.KLp + std::max(32 * p.NJ, 64) + 32;   // at least a group's bit strings
    // tiles of 2, 4, 8, ... words: the rows of 32 lanes would share banks
    p.BP = p.KL >= 64 && (p.KL & (p.KL - 1)) == 0 ? p.KL / 32 + 1 : 0;
    p.RP = (p.NC + 1) | 1;
    return p;
}
static int string_words(const SliceGeo &p) { return p.BP ? 32 * p.BP : p.KLp + 1; }

constexpr int kSliceMaxKL = 4096, kSliceMaxKL3 = 8192;
constexpr int kSliceWave = 760, kSliceWave3 = 304;

// Blocks, groups per block and threads of the resident kernel, and its
// estimated cycles per generation; false when the state does not fit.
static bool slice_resident_shape(const SliceGeo &p, int num_sms, bool batch, SlicePlan *s, double *cost)
{
    if (p.D > 8) return false;   // 3D: the neighbour table alone is larger than shared memory
    // one block where that takes no more than 8 chunks per warp, else as many as there are SMs
    for (int64_t grid : {(int64_t)1, std::min<int64_t>(num_sms, p.NG)}) {
        if (grid == 1 && batch && p.NG > 1) continue;   // (batches: no kernel for a single block's exports)
        const int64_t per = (p.NG + grid - 1) / grid, chunks = per * p.NC;
        const int64_t rounds = (chunks + 31) / 32;
        if (rounds > (grid == 1 ? 8 : kSliceRounds)) continue;
        const int64_t exw = grid == 1 ? 2 * p.NG * p.XW * 32 : 0;
        const int64_t smem = 4 * (4 * p.KLp + exw + 16 * p.XW + per * (32 * p.NJ + 1 + p.AW));
        if (smem > kSliceSmem) continue;
        // `n` warp-sized items of `instr` instructions: at least a chain of
        // latencies per round, else the SM's issue rate
        auto cycles = [](double n, double instr) {
            return std::ceil(n / 32) * std::max(170.0, std::min(n, 32.0) * instr / 2.8);
        };
        const double c = (grid > 1 ? 3000 : 100) + cycles((double)chunks, 55) + cycles((double)per * p.NJ, 35) +
                         cycles((double)per * p.XW, 35);
        if (s->resident && c >= *cost) continue;
        *cost = c;
        s->resident = true;
        s->per_block = (int)per;
        s->grid_resident = (int)grid;
        s->smem_resident = (int)smem;
        s->rounds = (int)rounds;
        s->block_resident = (int)std::min<int64_t>(1024, std::max<int64_t>(128, (chunks + 3) / 4 * 128));
    }
    return s->resident;
}

// Tables for the tile depth that costs least per generation: the resident
// kernel's where the state fits in shared memory, else the streaming one's (a
// group of 32 tiles adds its cells' neighbours, about 45 instructions per 32
// cells, makes and takes its halo words, about 30 each, and pays its loops
// and barriers, about 400; kSliceWave groups run at a time).
static int slice_levels(const fractal *f, SlicePlan *plan, std::shared_ptr<SliceImage> *image)
{
    int best = 0;
    double cost = 0;
    const bool d3 = f->dim == 3;
    // 3D: the deepest tiles with a group per SM, where there are such, without a look at the others
    int only = 0;
    for (int L = 1; d3 && L <= f->r && pw(f->k, L) <= kSliceMaxKL3; ++L)
        if ((double)pw(f->k, f->r - L) < 2147483648.0 && (pw(f->k, f->r - L) + 31) / 32 >= f->num_sms) only = L;
    for (int L = 1; L <= f->r && pw(f->k, L) <= (d3 ? kSliceMaxKL3 : kSliceMaxKL); ++L) {
        if ((only && L != only) || (double)pw(f->k, f->r - L) >= 2147483648.0) continue;
        const std::shared_ptr<SliceImage> img = slice_image(f, L);
        const SliceTables &t = img->t;
        const SliceGeo p = slice_geo(f, L, t);
        if (p.AW * 4 > 65535 || p.XW > 255) continue;
        SlicePlan s;
        double c;
        if (!slice_resident_shape(p, f->num_sms, false, &s, &c)) {
            const int wave = d3 ? kSliceWave3 : kSliceWave;
            const int64_t waves = (p.NG + wave - 1) / wave;
            c = (double)waves * (p.NC * (d3 ? 110 : 45) + 30.0 * (p.NJ + p.XW) + 400);
        }
        if (best && plan->resident && !s.resident) continue;
        if (!best || (s.resident && !plan->resident) || c < cost) {
            best = L;
            cost = c;
            *plan = s;
            plan->geo = p;
            *image = img;
        }
    }
    return best;
}

// Bytes of a packed state and its exports, and the states of one kind of call
// (one of single generations, two of several) at `mem`.
static size_t slice_packed_bytes(const SliceGeo &p)
{
    return ((size_t)p.NG * (p.KLp + 32 * p.XW) * sizeof(uint32_t) + 255) / 256 * 256;
}
static void slice_set_packed(SlicePlan &s, int states, uint8_t *mem)
{
    for (int i = 0; i < states; ++i)
        s.bits[states == 1 ? 2 : i] = reinterpret_cast<uint32_t *>(mem + i * slice_packed_bytes(s.geo));
}

// One allocation: the tables (copied from the host in one piece), the grid
// barrier's zeros, the neighbouring tiles, the resident exports and `packed`
// packed states.  `img` becomes the host's piece: the copy may read it until
// `st` has been waited for (a runtime that reads pageable memory in place does
// not stage it first), so the caller keeps it until then.
static cudaError_t slice_upload(SliceGeo &p, SliceImage &image, SlicePlan &s, const std::vector<SliceGroup> &groups,
                                int packed, std::vector<uint8_t> &img, cudaStream_t st)
{
    const SliceTables &t = image.t;
    const std::vector<uint16_t> &nb = image.neighbours(p.D);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t o_tab = take(nb.size() * 2), o_jobs = take(t.jobs.size() * 4), o_xl = take(t.xlist.size() * 2),
                 o_cells = take(t.cells.size() * 4), o_bar = take(16), o_groups = take(groups.size() * sizeof(SliceGroup)), host = off;
    const size_t o_nbr = take((size_t)p.NG * p.ND * 32 * sizeof(int32_t)),
                 exb = s.resident ? (size_t)p.NG * p.XW * 128 : 0, o_ex0 = take(exb), o_ex1 = take(exb),
                 o_ex2 = take(groups.empty() ? exb : 0), o_bits = take((size_t)packed * slice_packed_bytes(p));
    img.assign(host, 0);
    memcpy(img.data() + o_tab, nb.data(), nb.size() * 2);
    memcpy(img.data() + o_jobs, t.jobs.data(), t.jobs.size() * 4);
    memcpy(img.data() + o_xl, t.xlist.data(), t.xlist.size() * 2);
    memcpy(img.data() + o_cells, t.cells.data(), t.cells.size() * 4);
    if (!groups.empty()) memcpy(img.data() + o_groups, groups.data(), groups.size() * sizeof(SliceGroup));
    cudaError_t e = cudaMalloc(&s.arena, off);
    if (e == cudaSuccess) e = cudaMemcpyAsync(s.arena, img.data(), host, cudaMemcpyHostToDevice, st);
    p.tab = reinterpret_cast<uint4 *>(s.arena + o_tab);
    p.jobs = reinterpret_cast<uint32_t *>(s.arena + o_jobs);
    p.xlist = reinterpret_cast<uint16_t *>(s.arena + o_xl);
    p.cells = reinterpret_cast<uint2 *>(s.arena + o_cells);
    p.nbr = reinterpret_cast<int32_t *>(s.arena + o_nbr);
    s.bar = reinterpret_cast<uint32_t *>(s.arena + o_bar);
    s.groups = groups.empty() ? nullptr : s.arena + o_groups;
    s.ex[0] = reinterpret_cast<uint32_t *>(s.arena + o_ex0);
    s.ex[1] = reinterpret_cast<uint32_t *>(s.arena + o_ex1);
    s.ex[2] = reinterpret_cast<uint32_t *>(s.arena + o_ex2);
    if (packed) slice_set_packed(s, packed, s.arena + o_bits);
    return e;
}

// The plan, on the host alone: the tile depth and the shared memory.
static bool plan_slice(fractal *f)
{
    SlicePlan s;
    std::shared_ptr<SliceImage> img;
    if (slice_levels(f, &s, &img) < 1) return false;
    const SliceGeo &p = s.geo;
    s.single = f->slice.single;
    s.block = f->dim == 3 ? kSliceBlock3 : kSliceBlock;
    const int ring = 16 * kSliceBatch * s.block, arrays = f->dim == 3 ? 1 : 2;
    s.smem_pack = ring + 4 * string_words(p);
    s.smem_single = ring + 4 * (p.AW + std::max(string_words(p), 32 * p.RP + 1));
    s.smem_step = 4 * arrays * p.AW;
    s.smem_bytes = 4 * (arrays * p.AW + 32 * p.RP + 1);
    f->slice = s;
    return std::max(std::max(s.smem_pack, s.smem_single), std::max(s.smem_step, s.smem_bytes)) <= kSliceMost;
}

// Blocks of a kernel that fill the GPU, once its shared memory is allowed.
template <class Fn>
static cudaError_t slice_grid(Fn fn, int block, int smem, int num_sms, int64_t groups, int *grid)
{
    int per_sm = 0;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSliceMost);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, block, smem);
    if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
    *grid = (int)std::min<int64_t>((int64_t)per_sm * num_sms, groups);
    return e;
}

// Makes what a call still lacks: the tables, and with `packed` the packed
// states of its kind.  The kernels of the routes that need no packed state
// are set up with the tables (a later call may be captured), the others with
// the first packed state.
static int slice_prepare(fractal *f, bool packed, int64_t steps, cudaStream_t st)
{
    const bool tables = f->slice.state < 2;
    SlicePlan s = f->slice;   // (the handle's changes only when everything is there)
    SliceGeo &p = s.geo;
    const int states = !packed ? 0 : (steps == 1 ? 1 : 2);
    std::vector<uint8_t> host;
    uint8_t *mem = nullptr;
    cudaError_t e = cudaSuccess;
    if (tables) {
        e = slice_upload(p, *slice_image(f, p.L), s, {}, states, host, st);
        mem = s.arena;
        if (e == cudaSuccess) {
            const unsigned blocks = (unsigned)std::min<int64_t>((32 * p.NG + 255) / 256, (int64_t)f->num_sms * 16);
            const int moves = f->k * (p.ND + 1) * (int)sizeof(int16_t);
            if (f->dim == 3) slice_nbr_kernel<3><<<blocks, 256, moves, st>>>(f->dev, p.NT, p.NG, f->r - p.L, nullptr, p.nbr);
            else slice_nbr_kernel<2><<<blocks, 256, moves, st>>>(f->dev, p.NT, p.NG, f->r - p.L, nullptr, p.nbr);
            e = cudaGetLastError();
        }
        // the kernels while the tables are on their way
        if (e == cudaSuccess && s.resident) e = resident_ready(s);
        for (int life = 0; life < 2 && p.D <= 8 && p.H <= kSliceSingleHalo && e == cudaSuccess; ++life)
            e = slice_grid(single_fn(p.D, life), kSliceBlock, s.smem_single, f->num_sms, p.NG, &s.grid_single[life]);
    } else if (states) {
        e = cudaMalloc(&mem, states * slice_packed_bytes(p));
        if (e == cudaSuccess) slice_set_packed(s, states, s.packed[states == 1] = mem);
    }
    if (packed && s.grid_pack == 0 && e == cudaSuccess) {
        auto pack = f->dim == 3 ? slice_pack_kernel<kSliceBlock3> : slice_pack_kernel<kSliceBlock>;
        e = slice_grid(pack, s.block, s.smem_pack, f->num_sms, p.NG, &s.grid_pack);
        for (int life = 0; life < 2 && e == cudaSuccess; ++life) {
            e = slice_grid(step_fn(p.D, life, false), s.block, s.smem_step, f->num_sms, p.NG, &s.grid_step[life]);
            if (e == cudaSuccess) e = slice_grid(step_fn(p.D, life, true), s.block, s.smem_bytes, f->num_sms, p.NG, &s.grid_bytes[life]);
        }
    }
    if (tables && mem) {
        const cudaError_t landed = cudaStreamSynchronize(st);   // the tables serve calls on any stream from here on
        if (e == cudaSuccess) e = landed;
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        cudaFree(mem);
        return e == cudaErrorMemoryAllocation ? FR_ENOMEM : (e == cudaErrorInvalidConfiguration ? FR_EINVAL : FR_ECUDA);
    }
    s.state = 2;
    f->slice = s;
    return FR_OK;
}

// Whether a single generation is faster in the tile kernels (one launch, no
// packing).  Measured per launch in a graph, tiles -> sliced: single pass
// (few halo cells) triangle r = 10 4.6 -> 10 us, r = 12 4.8 -> 3.3, r = 15
// 10.4 -> 9.6; others H-fractal r = 7 (0.8 million cells) 6.4 -> 6.5, r = 8
// 18 -> 8.3; carpet r = 7 (2.1 million) 5.7 -> 6.3, r = 8 19 -> 15; Vicsek
// r = 11 21.5 -> 22, r = 12 96 -> 101.
// (halo_cells < 0: not known yet; only what holds for any)
static bool slice_one_generation_by_tiles(const fractal *f, int halo_cells)
{
    const int preset = rows_preset_of(f);
    if (preset == 1 || f->cells < (1 << 17)) return true;
    if (f->dim == 3) return f->cells < (1 << 22);
    if (halo_cells < 0) return false;
    if (halo_cells <= kSliceSingleHalo) return false;
    return f->cells < (preset == 0 ? 4 << 20 : 1 << 20);
}

// Whether a few generations of a small state are faster in the tile kernels,
// a launch each, than in the sliced step's launches and grid barriers.  Per
// call, tiles -> sliced: 2D, two generations, more than a chunk per warp: the
// triangle r = 10 12.4 -> 13.4 us, Vicsek r = 7 12.5 -> 15.8, r = 10 18.7 ->
// 20.1 (three generations of all of them are faster sliced).  3D: two
// generations of Menger r = 2 11.7 -> 16.4 us, k = 4, s = 2, r = 8 two, four
// and ten generations 12.6 -> 22.7, 24.8 -> 33.0, 61.7 -> 66.7, and the full
// cube with s = 2, r = 6 two and six 20.6 -> 29.0, 61.7 -> 64.7.  The sliced
// step's times there: three launches, and per generation a group's work, the
// barrier once there are several groups, more groups than two per SM.
static bool slice_few_generations_by_tiles(const fractal *f, const SlicePlan &s, int64_t steps)
{
    if (steps < 2 || steps > 64) return false;
    const double tiles = (double)steps * short_generation_us(f, f->plan.NT);
    if (f->dim == 2) {
        if (steps != 2 || (s.resident && s.grid_resident == 1 && s.rounds == 1)) return false;
        return tiles > 0.0 || (rows_preset_of(f) == 1 && f->plan.NT <= 5 * (int64_t)f->num_sms);
    }
    const double n = (double)steps, waves = (double)((s.geo.NG + 2 * f->num_sms - 1) / (2 * f->num_sms));
    const double sliced = s.geo.NG == 1 ? 11.5 + 2.0 * n : (s.geo.NG <= f->num_sms ? 8.0 + 4.1 * n : 11.0 + (2.6 + 1.5 * waves) * n);
    return tiles > 0.0 && tiles < sliced;
}

// Whether `steps` generations run in the resident kernel.  A single
// generation of a state with many groups is faster as streaming launches.
static bool slice_use_resident(const SlicePlan &s, int64_t steps, int num_sms)
{
    if (steps == 1 && s.geo.H <= kSliceSingleHalo) return false;
    return s.resident && (steps > 1 || s.geo.NG <= num_sms);
}

static SliceArgs slice_args(const SliceGeo &p, uint32_t birth, uint32_t survive, uint32_t *bar, int *status)
{
    SliceArgs a;
    a.NT = p.NT;
    a.NG = p.NG;
    a.KL = p.KL;
    a.KLp = p.KLp;
    a.NC = p.NC;
    a.NJ = p.NJ;
    a.BP = p.BP;
    a.RP = p.RP;
    a.AW = p.AW;
    a.A_zero = p.AW - 32;
    a.XW = p.XW;
    a.ND = p.ND;
    a.birth = birth & 0x7ffffffu;
    a.survive = survive & 0x7ffffffu;
    a.ex = p.NG * p.KLp;
    a.kdiv = make_div((uint32_t)p.KL);
    a.cdiv = make_div((uint32_t)std::max(2, p.NC));
    a.jdiv = make_div((uint32_t)std::max(2, p.NJ));
    a.xdiv = make_div((uint32_t)std::max(2, p.XW));
    a.bsh = 30;
    if (p.BP)
        for (a.bsh = 0; (32 << a.bsh) < p.KL;) ++a.bsh;
    a.lane_bits = p.BP ? 32u * (uint32_t)p.BP : (uint32_t)p.KL;
    for (int c = 0; c < 9; ++c) {
        a.mb[c] = (birth >> c) & 1u ? 0xffffffffu : 0u;
        a.ms[c] = (survive >> c) & 1u ? 0xffffffffu : 0u;
    }
    a.tab = p.tab;
    a.jobs = p.jobs;
    a.xlist = p.xlist;
    a.cells = p.cells;
    a.H = p.H;
    a.nbr = p.nbr;
    a.groups = nullptr;
    a.bar = bar;
    a.status = status;
    return a;
}

// Bytes -> packed state, the generations but the last on packed states, the last one to bytes.
static int run_packed(fractal *f, const SliceArgs &a, bool life, const uint8_t *in, uint8_t *out, int64_t steps, cudaStream_t st)
{
    const SlicePlan &s = f->slice;
    int cur = steps == 1 ? 2 : 0;
    if (f->dim == 3) slice_pack_kernel<kSliceBlock3><<<s.grid_pack, kSliceBlock3, s.smem_pack, st>>>(a, in, s.bits[cur]);
    else slice_pack_kernel<kSliceBlock><<<s.grid_pack, kSliceBlock, s.smem_pack, st>>>(a, in, s.bits[cur]);
    FR_CUDA(cudaGetLastError());
    int64_t left = steps - 1;   // generations before the one that writes bytes
    StepFn fn = step_fn(s.geo.D, life, false);
    while (left > 0) {
        int gens = (int)std::min<int64_t>(left, 1 << 20);
        const uint32_t *src = s.bits[cur];
        uint32_t *dst = s.bits[cur ^ 1];
        uint8_t *none = nullptr;
        void *args[] = {(void *)&a, &src, &dst, &none, &gens};
        if (s.grid_step[life] > 1 && gens > 1)
            FR_CUDA(cudaLaunchCooperativeKernel((const void *)fn, dim3(s.grid_step[life]), dim3(s.block), args, s.smem_step, st));
        else
            FR_CUDA(cudaLaunchKernel((const void *)fn, dim3(s.grid_step[life]), dim3(s.block), args, s.smem_step, st));
        left -= gens;
        if (gens & 1) cur ^= 1;
    }
    {
        StepFn fb = step_fn(s.geo.D, life, true);
        const uint32_t *src = s.bits[cur];
        uint32_t *none = nullptr;
        int one = 1;
        void *args[] = {(void *)&a, &src, &none, &out, &one};
        FR_CUDA(cudaLaunchKernel((const void *)fb, dim3(s.grid_bytes[life]), dim3(s.block), args, s.smem_bytes, st));
    }
    return FR_OK;
}

int try_slice_step(fractal *f, const uint8_t *in, uint8_t *out, int64_t steps, uint32_t birth, uint32_t survive,
                   cudaStream_t st, bool *done)
{
    *done = false;
    if (!slice_fractal_ok(f) || steps < 1) return FR_OK;
    SlicePlan &s = f->slice;
    if (s.state < 0) return FR_OK;
    if (steps == 1 && slice_one_generation_by_tiles(f, s.state > 0 ? s.geo.H : -1)) return FR_OK;
    const bool captured = capturing(st);
    if (s.state == 0) {
        if (captured) return FR_OK;
        s.state = plan_slice(f) ? 1 : -1;
        if (s.state < 0 || (steps == 1 && slice_one_generation_by_tiles(f, s.geo.H))) return FR_OK;
    }
    // (a captured call takes what exists: its handle may have no scratch for the tile kernels)
    if (!captured && slice_few_generations_by_tiles(f, s, steps)) return FR_OK;
    // how the call will run: in one resident or single-pass launch, or with packed states between launches
    const bool res = slice_use_resident(s, steps, f->num_sms);
    const bool packed = !res && !(steps == 1 && s.geo.D <= 8 && s.geo.H <= kSliceSingleHalo);
    // a handle's first single generation (of those that use packed states:
    // they run on the tile kernels under capture in any case) does not pay for
    // the tables, unless the state is large: first call of the H-fractal at
    // r = 8 with them 314 us, without 212, the next ones 8 against 18; Menger
    // r = 6 677 and 575, then 51 and 104; r = 7 1436 and 2150
    if (steps == 1 && (res || packed) && s.state == 1 && !captured && !s.single && f->cells < (f->dim == 3 ? 1 << 27 : 1 << 30)) {
        s.single = true;
        return FR_OK;
    }
    // under capture nothing is allocated, and a single generation leaves the
    // packed state alone (its replays may run beside other calls): the tile kernels run there
    PackedTurn &turn = f->step_turn[steps == 1];
    if (steps == 1 && (res || packed) && !captured && packed_busy(turn, st)) return FR_OK;
    const bool ready = s.state > 1 && (!packed || (steps == 1 ? s.bits[2] != nullptr : s.bits[0] && s.bits[1]));
    if (captured && (!ready || (steps == 1 && (res || packed)))) return FR_OK;
    int rc;
    if (!ready) {
        // after a refused allocation a number of calls go to the tile kernels before the next try
        if (s.memory.skip()) return FR_OK;
        rc = ensure_status(f);
        if (rc) return rc;
        rc = slice_prepare(f, packed, steps, st);
        if (rc == FR_EINVAL) s.state = -1;   // (what the handle has stays until it is destroyed)
        else if (rc) s.memory.refused();
        if (rc) return FR_OK;
        s.memory.granted();
    }
    const SliceGeo &p = s.geo;
    const SliceArgs a = slice_args(p, birth, survive, steps == 1 ? s.bar + 2 : s.bar, f->status);
    const bool life = slice_life(f, birth, survive);
    // fractal_test_arm_timeout: calls without a grid barrier are the tile kernels'
    const bool armed = f->test_extra_tx != 0;
    if (armed && !(res ? s.grid_resident > 1 : packed && steps > 2 && s.grid_step[life] > 1)) return FR_OK;
    *done = true;
    s.several |= steps > 1;
    if (!res && !packed) {
        single_fn(p.D, life)<<<s.grid_single[life], kSliceBlock, s.smem_single, st>>>(a, in, out);
        FR_CUDA(cudaGetLastError());
        return FR_OK;
    }
    rc = packed_enter(turn, st, captured);
    if (armed && !rc) {
        // the barrier's count starts one short, so its first wait runs out (a
        // limit and a target among the kernels' arguments cost every
        // generation 0.1 us); the last block to leave resets it as ever
        FR_CUDA(cudaMemsetAsync(a.bar, 0xff, sizeof(uint32_t), st));
        f->test_extra_tx = f->test_wait_limit = 0;
    }
    if (!rc) rc = res ? launch_resident(s, a, life, in, out, steps, st) : run_packed(f, a, life, in, out, steps, st);
    return rc ? rc : packed_leave(turn, st, captured);
}

// ---------------------------------------------------------------- batches

// Many instances of one fractal in resident launches: their groups stand in
// one list (an instance starts a group of its own; the neighbour table keeps
// them apart) and run as if they were one state.  Instances of few
// generations come last in every block's share and drop out on the way.
// Instances whose packed words do not fit the SMs' shared memory together run
// in several launches, one after the other, each through all of its
// generations; levels below a launch's tile depth have launches of their own.
struct SliceBatch {
    struct Launch {
        SlicePlan plan;
        SliceArgs args;
        bool life;
        int64_t steps;
    };
    std::vector<Launch> launches;
};

void free_slice_batch(SliceBatch *b)
{
    if (!b) return;
    for (auto &l : b->launches) free_slice_plan(l.plan);
    delete b;
}

int slice_batch_launches(const SliceBatch *b) { return (int)b->launches.size(); }

int run_slice_batch(const SliceBatch *b, cudaStream_t st)
{
    for (const auto &l : b->launches) {
        const int rc = launch_resident(l.plan, l.args, l.life, nullptr, nullptr, l.steps, st);
        if (rc) return rc;
    }
    return FR_OK;
}

bool slice_batch_takes(const fractal *f, int64_t steps)
{
    return f->dim == 2 && slice_fractal_ok(f) && steps >= 2 && steps < (1 << 30) && f->cells <= kSliceBatchCells && slice_settings(f, steps);
}

// Groups that fit one launch at this tile depth (0: none), and its cycles per generation.
static int64_t slice_batch_fit(SliceGeo p, int num_sms, int64_t groups, double *cost)
{
    for (int n = 1; n <= 256; ++n) {
        p.NG = (groups + n - 1) / n;
        SlicePlan s;
        double c = 0;
        if (slice_resident_shape(p, num_sms, true, &s, &c)) {
            *cost = n * c;
            return p.NG;
        }
    }
    return 0;
}

int build_slice_batch(const std::vector<SliceBatchItem> &items, uint32_t birth, uint32_t survive, cudaStream_t st, SliceBatch **out)
{
    *out = nullptr;
    fractal *rep = items[0].f;
    int rc = ensure_status(rep);
    if (rc) return rc;
    int rmax = 0;
    for (const auto &i : items) rmax = std::max(rmax, i.f->r);
    // tables by tile depth
    std::vector<std::shared_ptr<SliceImage>> tabs(1);
    std::vector<SliceGeo> geos(1);
    for (int L = 1; L <= rmax && pw(rep->k, L) <= kSliceMaxKL; ++L) {
        tabs.push_back(slice_image(rep, L));
        geos.push_back(slice_geo(rep, L, tabs.back()->t));
    }
    const int lmax = (int)tabs.size() - 1;
    auto groups_of = [&](const SliceBatchItem &i, int L) { return (pw(rep->k, i.f->r - L) + 31) / 32; };
    // best[b]: tile depth and cost of all instances of fewer than b levels
    struct Choice { int L = 0; int64_t cap = 0; double cost = 0; };
    std::vector<Choice> best(rmax + 2);
    for (int b = 2; b <= rmax + 1; ++b) {
        bool any = false;
        for (const auto &i : items) any = any || i.f->r < b;
        if (!any) continue;
        Choice pick;
        for (int L = 1; L <= std::min(lmax, b - 1); ++L) {
            if (geos[L].AW * 4 > 65535 || geos[L].XW > 255) continue;
            int64_t groups = 0, largest = 0;
            for (const auto &i : items)
                if (i.f->r < b && i.f->r >= L) {
                    groups += groups_of(i, L);
                    largest = std::max(largest, groups_of(i, L));
                }
            double c = 0;
            int64_t cap = 0;
            if (groups) {
                cap = slice_batch_fit(geos[L], rep->num_sms, groups, &c);
                if (cap < largest) {   // as few launches as the largest instance allows
                    double one = 0;
                    cap = slice_batch_fit(geos[L], rep->num_sms, largest, &one);
                    if (cap < largest) continue;
                    c = one * std::ceil((double)groups / (double)cap);
                }
            }
            bool rest = false;
            for (const auto &i : items) rest = rest || i.f->r < L;
            if (rest && best[L].L == 0) continue;
            c += rest ? best[L].cost : 0.0;
            if (pick.L == 0 || c < pick.cost) {
                pick.L = L;
                pick.cap = cap;
                pick.cost = c;
            }
        }
        best[b] = pick;
    }
    if (best[rmax + 1].L == 0) return FR_EINVAL;
    SliceBatch *batch = new (std::nothrow) SliceBatch();
    if (!batch) return FR_ENOMEM;
    const bool life = slice_life(rep, birth, survive);
    for (int b = rmax + 1; b > 1 && best[b].L > 0; b = best[b].L) {
        const int L = best[b].L;
        std::vector<const SliceBatchItem *> in;
        for (const auto &i : items)
            if (i.f->r < b && i.f->r >= L) in.push_back(&i);
        std::stable_sort(in.begin(), in.end(), [](const SliceBatchItem *x, const SliceBatchItem *y) { return x->steps > y->steps; });
        for (size_t i0 = 0; i0 < in.size();) {
            std::vector<SliceGroup> groups;
            size_t i = i0;
            for (; i < in.size() && (i == i0 || (int64_t)groups.size() + groups_of(*in[i], L) <= best[b].cap); ++i) {
                const SliceBatchItem &it = *in[i];
                const int64_t NT = pw(rep->k, it.f->r - L), n = groups_of(it, L);
                const int32_t g0 = (int32_t)groups.size(), levels = it.f->r - L;
                for (int64_t g = 0; g < n; ++g)
                    groups.push_back(SliceGroup{it.in + 32 * g * geos[L].KL, it.out + 32 * g * geos[L].KL,
                                                (int32_t)std::min<int64_t>(32, NT - 32 * g), (int32_t)(32 * g), levels, g0,
                                                (int32_t)it.steps});
            }
            batch->launches.emplace_back();
            SliceBatch::Launch &l = batch->launches.back();
            l.life = life;
            l.steps = in[i0]->steps;
            l.plan.geo = geos[L];
            SliceGeo &p = l.plan.geo;
            p.NG = (int64_t)groups.size();
            p.NT = 32 * p.NG;
            double c = 0;
            cudaError_t e = slice_resident_shape(p, rep->num_sms, true, &l.plan, &c) ? cudaSuccess : cudaErrorInvalidConfiguration;
            std::vector<uint8_t> host;
            if (e == cudaSuccess) e = slice_upload(p, *tabs[L], l.plan, groups, 0, host, st);
            if (e == cudaSuccess) {
                const int64_t blocks = std::min<int64_t>((32 * p.NG + 255) / 256, (int64_t)rep->num_sms * 16);
                slice_nbr_kernel<2><<<(unsigned)blocks, 256, rep->k * 9 * (int)sizeof(int16_t), st>>>(
                    rep->dev, p.NT, p.NG, 0, reinterpret_cast<const SliceGroup *>(l.plan.groups), p.nbr);
                e = cudaGetLastError();
                const cudaError_t landed = cudaStreamSynchronize(st);
                if (e == cudaSuccess) e = landed;
            }
            if (e == cudaSuccess) e = resident_ready(l.plan);
            if (e != cudaSuccess) {
                cudaGetLastError();
                free_slice_batch(batch);
                return e == cudaErrorMemoryAllocation ? FR_ENOMEM : FR_ECUDA;
            }
            l.args = slice_args(p, birth, survive, l.plan.bar, rep->status);
            l.args.groups = reinterpret_cast<const SliceGroup *>(l.plan.groups);
            i0 = i;
        }
    }
    *out = batch;
    return FR_OK;
}

}  // namespace fr
