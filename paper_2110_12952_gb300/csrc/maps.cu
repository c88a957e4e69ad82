// maps.cu -- the thread maps lambda and nu over arrays (Sec. 3, Sec. 3.1),
// the paper's multi-dimensional compact coordinate (Eqs. 6-8), compact <->
// box views, and the seeded Bernoulli initial state.
//
// Large arrays go through tables of several levels at once: lambda and nu are
// sums over the levels, so a table over the digits of m levels (built by each
// block in shared memory) replaces m digit steps by one look-up, and the
// triangle's 20 levels by three or four.  The digit loops they replace read
// the transition tables from constant memory at a different address per lane,
// which the hardware serialises (one pass per distinct address); they remain
// for short arrays, where building a table would cost more, and for fractals
// with a different table per level.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "handle.h"

namespace fr {

static int grid_for(int64_t n, int block, int num_sms)
{
    int64_t g = (n + block - 1) / block;
    int64_t cap = (int64_t)num_sms * 16;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

__global__ void lambda_kernel(FracDev F, const int64_t *__restrict__ omega, int64_t count,
                              int64_t cells, int32_t *__restrict__ coords)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t w = omega[e];
        int32_t p[3] = {-1, -1, -1};
        if (w >= 0 && w < cells) lambda64(F, (uint64_t)w, F.r, p);
        for (int i = 0; i < F.dim; ++i) coords[e * F.dim + i] = p[i];
    }
}

// Unsigned division of x < 2^63 by a constant (DivU32's method with 64 bits).
struct DivU64 {
    uint64_t m;
    uint32_t sh;
};

static DivU64 make_div64(uint64_t d)
{
    uint32_t l = 1;
    while ((1ull << l) < d) ++l;
    // ceil(2^(63 + l) / d), below 2^64 because d > 2^(l - 1)
    const unsigned __int128 num = (unsigned __int128)1 << (63 + l);
    return DivU64{(uint64_t)((num + d - 1) / d), l - 1};
}

constexpr int kMapTable = 4096;     // most entries of a table
constexpr int kMapGroups = 16;      // most groups of levels
constexpr int kMapBlock = 512;
constexpr int kMapBlocksPerSM = 4;
constexpr int64_t kMapLong = 20000000;  // points x levels x replicas from which arrays go through tables
// Cells from which the box views go by tiles.  Scatter and gather, cell by
// cell -> by tiles: 160,000 cells (Menger r = 4) 10.4 -> 11.9 and 7.4 -> 7.5 us,
// 262,144 (carpet r = 6) 10.4 -> 12.0 and 7.1 -> 7.5, 390,625 (Vicsek r = 8)
// 22.7 -> 24.7 and 8.4 -> 10.1, 531,441 (triangle r = 12) 16.5 -> 16.5 and 10.4
// -> 10.4, 823,543 (H-fractal r = 7) 18.5 -> 14.5 and 14.4 -> 10.4.
constexpr int64_t kViewLong = 1 << 19;
constexpr int64_t kMapBuild = 8;        // a block's points take at least this many times the digit steps of its tables

// lambda through tables: entry i holds the coordinates of i over m levels
// (16 bits each in 2D, 10 in 3D); omega's base-k^m digits pick the entries.
struct LambdaTab {
    int m, groups, n;        // levels per group, groups, entries (k^m)
    int m_last, n_last;      // the same of the last group, whose table follows (n_last = n: the same table)
    int last;                // where the last group's table starts
    int wide;                // groups before which the number may reach 2^31
    int32_t start[kMapGroups];    // where a group's table starts
    uint32_t scale[kMapGroups];   // s^(m g)
    DivU64 div64;            // by k^m
    DivU32 div32;
};

template <int DIM>
__device__ __forceinline__ void lambda_table(const FracDev &F, const LambdaTab &L, uint32_t *tab)
{
    const int all = L.n + (L.n_last == L.n ? 0 : L.n_last);
    for (int i = threadIdx.x; i < all; i += blockDim.x) {
        int32_t p[3];
        lambda32(F, (uint32_t)(i < L.n ? i : i - L.n), i < L.n ? L.m : L.m_last, p);
        tab[i] = DIM == 2 ? (uint32_t)p[0] | (uint32_t)p[1] << 16
                          : (uint32_t)p[0] | (uint32_t)p[1] << 10 | (uint32_t)p[2] << 20;
    }
}

template <int DIM>
__device__ __forceinline__ void lambda_lookup(const LambdaTab &L, const uint32_t *tab, uint64_t w, int32_t *p)
{
    uint32_t x = 0, y = 0, z = 0, v = (uint32_t)w;
    // (the loop is unrolled and left at a group count that is the same for all)
#pragma unroll
    for (int g = 0; g < kMapGroups; ++g) {
        if (g == L.groups) break;
        uint32_t q;
        if (g < L.wide) {   // the number may still reach 2^31
            w = __umul64hi(w, L.div64.m) >> L.div64.sh;
            q = (uint32_t)w;
        } else {
            q = divu(L.div32, v);
        }
        const uint32_t e = tab[v - q * (uint32_t)L.n + (uint32_t)L.start[g]];
        v = q;
        if (DIM == 2) {
            x += L.scale[g] * (e & 0xffffu);
            y += L.scale[g] * (e >> 16);
        } else {
            x += L.scale[g] * (e & 0x3ffu);
            y += L.scale[g] * ((e >> 10) & 0x3ffu);
            z += L.scale[g] * (e >> 20);
        }
    }
    p[0] = (int32_t)x;
    p[1] = (int32_t)y;
    if (DIM == 3) p[2] = (int32_t)z;
}

// 2^25 points of the triangle at r = 20: 1447 us with the digit loop (its
// constant loads serialised), 155 us here (3.4 TB/s; issue slots and latency)
template <int DIM, bool VEC>
__global__ void __launch_bounds__(kMapBlock) lambda_tab_kernel(FracDev F, LambdaTab L, const int64_t *__restrict__ omega,
                                                               int64_t count, int64_t cells, int32_t *__restrict__ coords)
{
    __shared__ uint32_t tab[2 * kMapTable];
    lambda_table<DIM>(F, L, tab);
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * blockDim.x, t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (VEC) {
        // two points per 16-byte load; their coordinates as 16 bytes (2D)
        const int64_t pairs = count / 2;
#pragma unroll 4
        for (int64_t e = t0; e < pairs; e += step) {
            const longlong2 w = __ldcs(reinterpret_cast<const longlong2 *>(omega) + e);
            int32_t p[2 * DIM];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t v = h ? w.y : w.x;
                const bool ok = v >= 0 && v < cells;
                lambda_lookup<DIM>(L, tab, ok ? (uint64_t)v : 0u, p + DIM * h);
                for (int i = 0; i < DIM; ++i) p[DIM * h + i] = ok ? p[DIM * h + i] : -1;
            }
            if (DIM == 2) __stcs(reinterpret_cast<int4 *>(coords) + e, make_int4(p[0], p[1], p[2], p[3]));
            else
                for (int i = 0; i < 3; ++i) __stcs(reinterpret_cast<int2 *>(coords) + 3 * e + i, make_int2(p[2 * i], p[2 * i + 1]));
        }
    }
    for (int64_t e = (VEC ? count / 2 * 2 : 0) + t0; e < count; e += step) {
        const int64_t v = omega[e];
        int32_t p[3] = {-1, -1, -1};
        if (v >= 0 && v < cells) lambda_lookup<DIM>(L, tab, (uint64_t)v, p);
        for (int i = 0; i < DIM; ++i) coords[e * DIM + i] = p[i];
    }
}

// nu through tables: entry x + s^m (y + s^m z) holds the replica digits of m
// levels as a number (base k), or -1 where some level's digits are no
// replica.  With COMPACT it holds the compact coordinate of the m levels
// instead, 16 bits per component in 2D, 10 in 3D, in a table for each axis
// that a group's first level may fall on.
struct NuTab {
    int m, groups, n;        // levels per group, groups, entries (s^(m dim))
    int m_last, n_last;      // the same of the last group, whose table follows (n_last = n: the same table)
    int last;                // where the last group's table starts
    int phases;              // tables by the axis of a group's first level (compact coordinate)
    uint32_t sm;             // s^m
    int shift;               // log2 of s^m, or -1
    DivU32 div;              // by s^m
    int32_t start[kMapGroups];   // where a group's table starts
    int64_t scale[kMapGroups];   // k^(m g); compact coordinate: k^floor(m g / dim)
};

template <int DIM, bool COMPACT>
__device__ __forceinline__ void nu_table(const FracDev &F, const NuTab &N, uint32_t *tab)
{
    const int whole = N.n * N.phases, all = whole + (N.last == 0 ? 0 : N.n_last);
    for (int i = threadIdx.x; i < all; i += blockDim.x) {
        // (the last group's digits run over s^m_last only, but are laid out
        // like the others': entries in between are never read)
        const int part = i < whole ? i / N.n : (N.groups - 1) * N.m % DIM;
        uint32_t c[3] = {0, 0, 0}, v = (uint32_t)(i < whole ? i - part * N.n : i - whole);
        const int m = i < whole ? N.m : N.m_last;
        // the group of a whole table starts at axis (m part) mod dim, the last one at its own
        int axis = COMPACT ? (i < whole ? part * N.m % DIM : part) : 0;
        for (int a = 0; a < DIM; ++a) {
            const uint32_t q = divu(N.div, v);
            c[a] = v - q * N.sm;
            v = q;
        }
        uint32_t acc[3] = {0, 0, 0}, w = 1;
        bool ok = true;
        for (int mu = 0; mu < m; ++mu) {
            uint32_t t = 0, base = 1;
            for (int a = 0; a < DIM; ++a) {
                const uint32_t q = divu(F.sdiv, c[a]);
                t += (c[a] - q * F.s) * base;
                base *= F.s;
                c[a] = q;
            }
            const int h = F.hinv[t];
            ok = ok && h >= 0;
            acc[axis] += (uint32_t)h * w;
            if (!COMPACT) w *= F.k;
            else if (++axis == DIM) {
                axis = 0;
                w *= F.k;
            }
        }
        tab[i] = !ok ? 0xffffffffu
                     : (!COMPACT ? acc[0] : (DIM == 2 ? acc[0] | acc[1] << 16 : acc[0] | acc[1] << 10 | acc[2] << 20));
    }
}

// POW2: s^m is a power of two.
template <int DIM, bool COMPACT, bool POW2>
__device__ __forceinline__ void nu_lookup(const NuTab &N, const uint32_t *tab, int32_t side, const int32_t *c, int64_t *out)
{
    constexpr int NC = COMPACT ? DIM : 1;
    uint32_t v[3] = {(uint32_t)c[0], (uint32_t)c[1], DIM == 3 ? (uint32_t)c[2] : 0u};
    // (a negative coordinate is a large unsigned one)
    bool ok = v[0] < (uint32_t)side && v[1] < (uint32_t)side && v[2] < (uint32_t)side;
#pragma unroll
    for (int a = 0; a < DIM; ++a) v[a] = ok ? v[a] : 0u;
    int64_t acc[3] = {0, 0, 0};
#pragma unroll
    for (int g = 0; g < kMapGroups; ++g) {
        if (g == N.groups) break;
        uint32_t i = (uint32_t)N.start[g], w = 1;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            const uint32_t q = POW2 ? v[a] >> N.shift : divu(N.div, v[a]);
            const uint32_t d = POW2 ? v[a] & (N.sm - 1u) : v[a] - q * N.sm;
            i += POW2 ? d << (a * N.shift) : d * w;
            w *= N.sm;
            v[a] = q;
        }
        const uint32_t e = tab[i];
        ok = ok && e != 0xffffffffu;
        if (!COMPACT) acc[0] += N.scale[g] * (int64_t)e;
        else if (DIM == 2) {
            acc[0] += N.scale[g] * (int64_t)(e & 0xffffu);
            acc[1] += N.scale[g] * (int64_t)(e >> 16);
        } else {
            acc[0] += N.scale[g] * (int64_t)(e & 0x3ffu);
            acc[1] += N.scale[g] * (int64_t)((e >> 10) & 0x3ffu);
            acc[2] += N.scale[g] * (int64_t)(e >> 20);
        }
    }
    for (int i = 0; i < NC; ++i) out[i] = ok ? acc[i] : -1;
}

// 2^25 points of the triangle at r = 20: nu 957 -> 145 us, compact coordinate
// 1094 -> 185 us
template <int DIM, bool COMPACT, bool VEC, bool POW2>
__global__ void __launch_bounds__(kMapBlock) nu_tab_kernel(FracDev F, NuTab N, int32_t side, const int32_t *__restrict__ coords,
                                                           int64_t count, int64_t *__restrict__ out)
{
    constexpr int NC = COMPACT ? DIM : 1;
    __shared__ uint32_t tab[2 * kMapTable];
    nu_table<DIM, COMPACT>(F, N, tab);
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * blockDim.x, t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (VEC) {
        // 2D: two points per 16-byte load
        const int64_t pairs = count / 2;
#pragma unroll 4
        for (int64_t e = t0; e < pairs; e += step) {
            const int4 v = __ldcs(reinterpret_cast<const int4 *>(coords) + e);
            const int32_t c[4] = {v.x, v.y, v.z, v.w};
            int64_t r[2 * NC];
            nu_lookup<2, COMPACT, POW2>(N, tab, side, c, r);
            nu_lookup<2, COMPACT, POW2>(N, tab, side, c + 2, r + NC);
            for (int i = 0; i < NC; ++i)
                __stcs(reinterpret_cast<longlong2 *>(out) + NC * e + i, make_longlong2(r[2 * i], r[2 * i + 1]));
        }
    }
    for (int64_t e = (VEC ? count / 2 * 2 : 0) + t0; e < count; e += step) {
        int32_t c[3] = {0, 0, 0};
        for (int i = 0; i < DIM; ++i) c[i] = coords[e * DIM + i];
        int64_t r[3];
        nu_lookup<DIM, COMPACT, POW2>(N, tab, side, c, r);
        for (int i = 0; i < NC; ++i) out[e * NC + i] = r[i];
    }
}

// Whether tables pay for an array: the digit loops take longer with more
// levels and, their constant loads being serialised, with more replicas.  The
// triangle at r = 11, 504,289 points, lambda, nu and compact coordinate with a
// cold cache: digit loops 48 us, tables 53; at r = 20 with a warm one 64 and 25.
static bool map_long(const fractal *f, int64_t count)
{
    return (double)count * f->r * f->k >= (double)kMapLong;
}

static int map_grid(const fractal *f, int64_t count)
{
    return (int)std::min<int64_t>((int64_t)f->num_sms * kMapBlocksPerSM, (count + kMapBlock - 1) / kMapBlock);
}

// Most entries x levels of a block's tables: building an entry costs what a
// point of that many levels costs in the digit loops.  504,289 points of the
// triangle at r = 11, cold: largest tables at any length 81 us, by this rule
// 53.  At 3 instead of 8 arrays of 2 and 8 million points take up to 60 %
// longer; at 24 some take up to 30 % less and others (Menger r = 7, compact
// coordinate) 30 % more.
static int64_t map_budget(const fractal *f, int64_t count)
{
    return count / map_grid(f, count) * f->r / kMapBuild;
}

static bool lambda_tab(const fractal *f, int64_t count, LambdaTab *L)
{
    if (f->mixed || f->k < 2 || f->r < 1) return false;
    const int64_t most = f->dim == 2 ? 65536 : 1024, budget = map_budget(f, count);
    int64_t n = f->k, sm = f->s;
    int m = 1;
    while (m < f->r && n * f->k <= kMapTable && sm * f->s <= most && n * f->k * (m + 1) <= budget) {
        n *= f->k;
        sm *= f->s;
        ++m;
    }
    const int groups = (f->r + m - 1) / m, m_last = f->r - m * (groups - 1);
    int64_t n_last = 1;
    for (int i = 0; i < m_last; ++i) n_last *= f->k;
    if (groups > kMapGroups) return false;
    L->m = m;
    L->groups = groups;
    L->n = (int)n;
    L->m_last = m_last;
    L->n_last = (int)n_last;
    L->last = n_last == n ? 0 : (int)n;
    for (int g = 0; g < kMapGroups; ++g) L->start[g] = g == groups - 1 ? L->last : 0;
    L->wide = 0;
    for (int64_t c = f->cells - 1; c >> 31; c /= n) ++L->wide;
    uint32_t scale = 1;
    for (int g = 0; g < kMapGroups; ++g, scale *= (uint32_t)sm) L->scale[g] = scale;
    L->div64 = make_div64((uint64_t)n);
    L->div32 = make_div((uint32_t)n);
    return true;
}

static bool nu_tab(const fractal *f, bool compact, int64_t count, NuTab *N)
{
    if (f->mixed || f->r < 1) return false;
    const int dim = f->dim;
    // components are stored in 16 or 10 bits, nu in 31
    const int64_t budget = map_budget(f, count);
    const int64_t most = !compact ? (int64_t)1 << 31 : (dim == 2 ? 65535 : 1024);
    int64_t block = 1;
    for (int i = 0; i < dim; ++i) block *= f->s;
    int m = 0, phases = 1;
    int64_t n = 1, sm = 1;
    for (int t = 1; t <= f->r; ++t) {
        int64_t nt = 1, st = 1, kc = 1;
        for (int i = 0; i < t; ++i) {
            nt *= block;
            st *= f->s;
            if (nt > kMapTable) break;
        }
        // (a group's components have at most ceil(t / dim) digits, wherever it starts: t levels alternate the axes)
        for (int i = 0; i < (compact ? (t + dim - 1) / dim : t); ++i) kc = kc > most ? kc : kc * f->k;
        const int ph = !compact || t % dim == 0 ? 1 : dim;   // (dim is 2 or 3: prime)
        if (nt > kMapTable) break;
        if (kc > most || nt * ph > kMapTable || (m > 0 && nt * ph * t > budget)) continue;
        m = t;
        n = nt;
        sm = st;
        phases = ph;
    }
    if (m == 0) return false;
    const int groups = (f->r + m - 1) / m, m_last = f->r - m * (groups - 1);
    // the last group's largest index + 1: its coordinates stay below s^m_last, in steps of s^m
    int64_t sl = 1, n_last = 0, row = 1;
    for (int i = 0; i < m_last; ++i) sl *= f->s;
    for (int i = 0; i < dim; ++i, row *= sm) n_last += (sl - 1) * row;
    if (groups > kMapGroups) return false;
    N->m = m;
    N->groups = groups;
    N->n = (int)n;
    N->m_last = m_last;
    N->n_last = m_last == m ? (int)n : (int)n_last + 1;
    N->phases = phases;
    N->last = m_last == m ? 0 : (int)n * phases;
    N->sm = (uint32_t)sm;
    N->shift = -1;
    if ((sm & (sm - 1)) == 0)
        for (N->shift = 0; (1ll << N->shift) < sm;) ++N->shift;
    N->div = make_div((uint32_t)sm);
    for (int g = 0; g < kMapGroups; ++g) N->start[g] = g == groups - 1 && N->last ? N->last : g % phases * (int)n;
    for (int g = 0; g < kMapGroups; ++g) {   // (past the last group it may wrap: never read)
        uint64_t scale = 1;
        for (int i = 0; i < (compact ? m * g / dim : m * g); ++i) scale *= (uint64_t)f->k;
        N->scale[g] = (int64_t)scale;
    }
    return true;
}

template <bool COMPACT>
static int launch_nu_tab(const fractal *f, const NuTab &N, const int32_t *coords, int64_t count, int64_t *out, cudaStream_t st)
{
    const bool vec = f->dim == 2 && ((uintptr_t)coords & 15) == 0 && ((uintptr_t)out & 15) == 0;
    const int grid = map_grid(f, count), side = (int32_t)f->side;
    if (f->dim == 3) nu_tab_kernel<3, COMPACT, false, false><<<grid, kMapBlock, 0, st>>>(f->dev, N, side, coords, count, out);
    else if (vec && N.shift >= 0) nu_tab_kernel<2, COMPACT, true, true><<<grid, kMapBlock, 0, st>>>(f->dev, N, side, coords, count, out);
    else if (vec) nu_tab_kernel<2, COMPACT, true, false><<<grid, kMapBlock, 0, st>>>(f->dev, N, side, coords, count, out);
    else nu_tab_kernel<2, COMPACT, false, false><<<grid, kMapBlock, 0, st>>>(f->dev, N, side, coords, count, out);
    FR_CUDA(cudaGetLastError());
    return FR_OK;
}

__device__ __forceinline__ bool in_box(const FracDev &F, int32_t side, const int32_t *c)
{
    for (int i = 0; i < F.dim; ++i)
        if (c[i] < 0 || c[i] >= side) return false;
    return true;
}

__global__ void nu_kernel(FracDev F, int32_t side, const int32_t *__restrict__ coords,
                          int64_t count, int64_t *__restrict__ omega)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count;
         e += (int64_t)gridDim.x * blockDim.x) {
        int32_t c[3] = {0, 0, 0};
        for (int i = 0; i < F.dim; ++i) c[i] = coords[e * F.dim + i];
        omega[e] = in_box(F, side, c) ? nu_levels(F, c[0], c[1], c[2], F.r) : -1;
    }
}

// Eqs. 6-8: component (mu mod dim) gains H_mu * k^floor(mu/dim).
__global__ void nu2d_kernel(FracDev F, int32_t side, const int32_t *__restrict__ coords,
                            int64_t count, int64_t *__restrict__ out)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count;
         e += (int64_t)gridDim.x * blockDim.x) {
        int32_t c[3] = {0, 0, 0};
        for (int i = 0; i < F.dim; ++i) c[i] = coords[e * F.dim + i];
        int64_t acc[3] = {0, 0, 0};
        bool inside = in_box(F, side, c);
        uint32_t x = c[0], y = c[1], z = c[2];
        int64_t w = 1;
        int axis = 0;
        if (F.mix) {
            // per-level tables: level mu's replica ID, weighted by the replica
            // counts of the earlier levels of the same axis
            int64_t wa[3] = {1, 1, 1};
            for (int mu = 0; inside && mu < F.r; ++mu) {
                const MixLevel &M = F.mix[mu];
                const uint32_t qx = divu(F.sdiv, x), qy = divu(F.sdiv, y);
                uint32_t t = (x - qx * F.s) + (uint32_t)F.s * (y - qy * F.s);
                x = qx;
                y = qy;
                if (F.dim == 3) {
                    const uint32_t qz = divu(F.sdiv, z);
                    t += (uint32_t)(F.s * F.s) * (z - qz * F.s);
                    z = qz;
                }
                const int h = M.hinv[t];
                if (h < 0) inside = false;
                const int a = mu % F.dim;
                acc[a] += (int64_t)h * wa[a];
                wa[a] *= M.k;
            }
            for (int i = 0; i < F.dim; ++i) out[e * F.dim + i] = inside ? acc[i] : -1;
            continue;
        }
        for (int mu = 0; inside && mu < F.r; ++mu) {
            uint32_t qx = divu(F.sdiv, x), qy = divu(F.sdiv, y);
            uint32_t t = (x - qx * F.s) + (uint32_t)F.s * (y - qy * F.s);
            x = qx;
            y = qy;
            if (F.dim == 3) {
                uint32_t qz = divu(F.sdiv, z);
                t += (uint32_t)(F.s * F.s) * (z - qz * F.s);
                z = qz;
            }
            int h = F.hinv[t];
            if (h < 0) inside = false;
            acc[axis] += (int64_t)h * w;
            if (++axis == F.dim) {
                axis = 0;
                w *= F.k;
            }
        }
        for (int i = 0; i < F.dim; ++i) out[e * F.dim + i] = inside ? acc[i] : -1;
    }
}

// SplitMix64 (Steele, Lea & Flood, OOPSLA 2014): the omega-th output for a
// seed is mix(seed + (omega + 1) * gamma).
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t i)
{
    uint64_t z = seed + (i + 1) * 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// 16 cells per thread and per iteration, written as one 16-byte store when
// the destination is aligned.
__global__ void init_kernel(uint8_t *__restrict__ state, int64_t cells, uint64_t seed,
                            uint64_t thr)
{
    const int64_t head = (16 - ((uintptr_t)state & 15)) & 15;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;; c += (int64_t)gridDim.x * blockDim.x) {
        int64_t w0 = (c == 0) ? 0 : head + (c - 1) * 16;
        if (w0 >= cells) break;
        int64_t w1 = (c == 0) ? (head < cells ? head : cells) : (w0 + 16 < cells ? w0 + 16 : cells);
        if (c > 0 && w1 - w0 == 16) {
            uint32_t v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t word = 0;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    uint64_t x = splitmix64_at(seed, (uint64_t)(w0 + q * 4 + b));
                    word |= (uint32_t)((x >> 11) < thr) << (8 * b);
                }
                v[q] = word;
            }
            *reinterpret_cast<uint4 *>(state + w0) = make_uint4(v[0], v[1], v[2], v[3]);
        } else {
            for (int64_t w = w0; w < w1; ++w)
                state[w] = (splitmix64_at(seed, (uint64_t)w) >> 11) < thr;
        }
    }
}

__global__ void scatter_kernel(FracDev F, int64_t cells, int64_t side,
                               const uint8_t *__restrict__ compact, uint8_t *__restrict__ box)
{
    for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < cells;
         w += (int64_t)gridDim.x * blockDim.x) {
        int32_t p[3] = {0, 0, 0};
        lambda64(F, (uint64_t)w, F.r, p);
        int64_t idx = p[0] + side * (p[1] + side * (int64_t)p[2]);
        box[idx] = compact[w] != 0;
    }
}

__global__ void gather_kernel(FracDev F, int64_t cells, int64_t side,
                              const uint8_t *__restrict__ box, uint8_t *__restrict__ compact)
{
    for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < cells;
         w += (int64_t)gridDim.x * blockDim.x) {
        int32_t p[3] = {0, 0, 0};
        lambda64(F, (uint64_t)w, F.r, p);
        int64_t idx = p[0] + side * (p[1] + side * (int64_t)p[2]);
        compact[w] = box[idx] != 0;
    }
}

// Compact <-> box by tiles of m levels (k^m <= kMapTable cells): the place of
// a tile's cells relative to the tile's own is the same for all tiles, so each
// block builds that table once in shared memory and walks runs of up to 32
// tiles, whose places its first warp computes with lambda.  A cell then costs one
// table look-up; what bounds it is the byte-wise access to the box (rows of a
// few cells).  Menger r = 6: scatter
// 1140 -> 273 us (and 57 us of memset), gather 1148 -> 88 us.
template <bool SCATTER>
__global__ void __launch_bounds__(256) box_tiles_kernel(FracDev F, int64_t NT, int m, int KL, DivU32 kldiv, int run, uint32_t side,
                                                        const uint8_t *__restrict__ src, uint8_t *__restrict__ dst)
{
    __shared__ uint32_t tab[kMapTable];
    __shared__ int64_t place[32];
    for (int l = threadIdx.x; l < KL; l += blockDim.x) {
        int32_t p[3];
        lambda32(F, (uint32_t)l, m, p);
        tab[l] = (uint32_t)p[0] + side * ((uint32_t)p[1] + side * (uint32_t)p[2]);
    }
    int64_t sm = 1;
    for (int i = 0; i < m; ++i) sm *= F.s;
    for (int64_t t0 = run * (int64_t)blockIdx.x; t0 < NT; t0 += run * (int64_t)gridDim.x) {
        const int nt = (int)min((int64_t)run, NT - t0);
        __syncthreads();
        if ((int)threadIdx.x < nt) {
            int32_t p[3];
            lambda64(F, (uint64_t)(t0 + threadIdx.x), F.r - m, p);
            place[threadIdx.x] = sm * (p[0] + (int64_t)side * (p[1] + (int64_t)side * p[2]));
        }
        __syncthreads();
        const int64_t w0 = t0 * KL;
        if (SCATTER) {   // tile by tile: the stores to a tile's rows stay close together
            for (int t = 0; t < nt; ++t) {
                uint8_t *b = dst + place[t];
#pragma unroll 4
                for (int l = threadIdx.x; l < KL; l += 256) b[tab[l]] = src[w0 + (int64_t)t * KL + l] != 0;
            }
        } else {
#pragma unroll 4
            for (int i = threadIdx.x; i < nt * KL; i += 256) {
                const int t = (int)divu(kldiv, (uint32_t)i);
                dst[w0 + i] = src[place[t] + tab[i - t * KL]] != 0;
            }
        }
    }
}

__global__ void copy_normalise_kernel(const uint8_t *__restrict__ in, uint8_t *__restrict__ out,
                                      int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = in[i] != 0;
}

int launch_copy_normalise(const uint8_t *in, uint8_t *out, int64_t n, int num_sms, cudaStream_t st)
{
    if (n == 0) return FR_OK;
    copy_normalise_kernel<<<grid_for(n, 256, num_sms), 256, 0, st>>>(in, out, n);
    FR_CUDA(cudaGetLastError());
    return FR_OK;
}

// Loads the copy kernel's module now, so that a first launch inside a stream
// capture does not have to.
int preload_copy_kernel()
{
    cudaFuncAttributes fa;
    FR_CUDA(cudaFuncGetAttributes(&fa, copy_normalise_kernel));
    return FR_OK;
}

}  // namespace fr

using namespace fr;

// Whether the views go by tiles, and the tile depth: the deepest with at most
// kMapTable cells whose places fit in 32 bits, and with four tiles per SM
// where the state has as many (of 128 cells or more).
static int box_tile_levels(const fractal *f)
{
    if (f->mixed || f->k < 2 || f->cells < kViewLong) return 0;
    int m = 0;
    int64_t kl = f->k, sm = f->s;
    for (; m < f->r && kl <= kMapTable; ++m, kl *= f->k, sm *= f->s) {
        const double most = (double)(sm - 1) * (1.0 + (double)f->side + (f->dim == 3 ? (double)f->side * f->side : 0.0));
        if (most >= 4294967296.0 || (kl / f->k >= 128 && f->cells / kl < 4 * f->num_sms)) break;
    }
    return m;
}

template <bool SCATTER>
static int launch_box_tiles(const fractal *f, int m, const uint8_t *src, uint8_t *dst, cudaStream_t st)
{
    int64_t KL = 1;
    for (int i = 0; i < m; ++i) KL *= f->k;
    const int64_t NT = f->cells / KL;
    const int64_t blocks = (int64_t)f->num_sms * 8;
    const int run = (int)std::max<int64_t>(1, std::min<int64_t>(32, NT / blocks));
    const int grid = (int)std::min<int64_t>((NT + run - 1) / run, blocks);
    box_tiles_kernel<SCATTER><<<grid, 256, 0, st>>>(f->dev, NT, m, (int)KL, make_div((uint32_t)KL), run, (uint32_t)f->side, src, dst);
    FR_CUDA(cudaGetLastError());
    return FR_OK;
}

static int fail_null(const char *what)
{
    set_error(FR_EINVAL, std::string(what) + ": NULL argument");
    return FR_EINVAL;
}

extern "C" int fractal_lambda(const fractal_t *f, const int64_t *omega, int64_t count,
                              int32_t *coords, void *stream)
{
    if (!f || (count > 0 && (!omega || !coords))) return fail_null("fractal_lambda");
    if (count < 0) return fail_null("fractal_lambda (count < 0)");
    if (count == 0) return FR_OK;
    LambdaTab L;
    if (map_long(f, count) && lambda_tab(f, count, &L)) {
        const bool vec = ((uintptr_t)omega & 15) == 0 && ((uintptr_t)coords & 15) == 0;
        const int grid = map_grid(f, count);
        cudaStream_t st = (cudaStream_t)stream;
        if (f->dim == 3 && vec) lambda_tab_kernel<3, true><<<grid, kMapBlock, 0, st>>>(f->dev, L, omega, count, f->cells, coords);
        else if (f->dim == 3) lambda_tab_kernel<3, false><<<grid, kMapBlock, 0, st>>>(f->dev, L, omega, count, f->cells, coords);
        else if (vec) lambda_tab_kernel<2, true><<<grid, kMapBlock, 0, st>>>(f->dev, L, omega, count, f->cells, coords);
        else lambda_tab_kernel<2, false><<<grid, kMapBlock, 0, st>>>(f->dev, L, omega, count, f->cells, coords);
        FR_CUDA(cudaGetLastError());
        return FR_OK;
    }
    lambda_kernel<<<grid_for(count, 256, f->num_sms), 256, 0, (cudaStream_t)stream>>>(
        f->dev, omega, count, f->cells, coords);
    FR_CUDA(cudaGetLastError());
    return FR_OK;
}

extern "C" int fractal_nu(const fractal_t *f, const int32_t *coords, int64_t count,
                          int64_t *omega, void *stream)
{
    if (!f || (count > 0 && (!omega || !coords))) return fail_null("fractal_nu");
    if (count < 0) return fail_null("fractal_nu (count < 0)");
    if (count == 0) return FR_OK;
    NuTab N;
    if (map_long(f, count) && nu_tab(f, false, count, &N)) return launch_nu_tab<false>(f, N, coords, count, omega, (cudaStream_t)stream);
    nu_kernel<<<grid_for(count, 256, f->num_sms), 256, 0, (cudaStream_t)stream>>>(
        f->dev, (int32_t)f->side, coords, count, omega);
    FR_CUDA(cudaGetLastError());
    return FR_OK;
}

extern "C" int fractal_nu2d(const fractal_t *f, const int32_t *coords, int64_t count,
                            int64_t *out, void *stream)
{
    if (!f || (count > 0 && (!out || !coords))) return fail_null("fractal_nu2d");
    if (count < 0) return fail_null("fractal_nu2d (count < 0)");
    if (count == 0) return FR_OK;
    NuTab N;
    if (map_long(f, count) && nu_tab(f, true, count, &N)) return launch_nu_tab<true>(f, N, coords, count, out, (cudaStream_t)stream);
    nu2d_kernel<<<grid_for(count, 256, f->num_sms), 256, 0, (cudaStream_t)stream>>>(
        f->dev, (int32_t)f->side, coords, count, out);
    FR_CUDA(cudaGetLastError());
    return FR_OK;
}

extern "C" int fractal_init_bernoulli(const fractal_t *f, uint8_t *state, uint64_t seed,
                                      double p, void *stream)
{
    if (!f || !state) return fail_null("fractal_init_bernoulli");
    uint64_t thr;
    if (!(p > 0.0)) thr = 0;
    else if (p >= 1.0) thr = 1ull << 53;
    else thr = (uint64_t)(p * 9007199254740992.0);  // floor(p * 2^53), exact scaling
    int64_t chunks = f->cells / 16 + 2;
    init_kernel<<<grid_for(chunks, 256, f->num_sms), 256, 0, (cudaStream_t)stream>>>(
        state, f->cells, seed, thr);
    FR_CUDA(cudaGetLastError());
    return FR_OK;
}

extern "C" int fractal_scatter_to_box(const fractal_t *f, const uint8_t *compact, uint8_t *box,
                                      void *stream)
{
    if (!f || !compact || !box) return fail_null("fractal_scatter_to_box");
    if (f->box_cells < 0) {
        set_error(FR_EOVERFLOW, "fractal_scatter_to_box: n^dim overflows");
        return FR_EOVERFLOW;
    }
    cudaStream_t st = (cudaStream_t)stream;
    FR_CUDA(cudaMemsetAsync(box, 0, (size_t)f->box_cells, st));
    if (const int m = box_tile_levels(f)) return launch_box_tiles<true>(f, m, compact, box, st);
    scatter_kernel<<<grid_for(f->cells, 256, f->num_sms), 256, 0, st>>>(
        f->dev, f->cells, f->side, compact, box);
    FR_CUDA(cudaGetLastError());
    return FR_OK;
}

extern "C" int fractal_gather_from_box(const fractal_t *f, const uint8_t *box, uint8_t *compact,
                                       void *stream)
{
    if (!f || !compact || !box) return fail_null("fractal_gather_from_box");
    if (const int m = box_tile_levels(f)) return launch_box_tiles<false>(f, m, box, compact, (cudaStream_t)stream);
    gather_kernel<<<grid_for(f->cells, 256, f->num_sms), 256, 0, (cudaStream_t)stream>>>(
        f->dev, f->cells, f->side, box, compact);
    FR_CUDA(cudaGetLastError());
    return FR_OK;
}
