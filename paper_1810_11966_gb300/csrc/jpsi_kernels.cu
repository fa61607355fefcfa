// Kernels of the J/psi first-level selection (arXiv:1810.11966, Sec. 3.2) on
// sm_103a.  Work unit: one event (on the block tile in CHAIN mode, one of its
// stations).  Four paths, chosen per event, give bit-identical results:
//
//   k_light    one warp per event.  Each station's hits are read once from HBM
//              (coalesced) and kept as slopes (s_x, s_y) in shared memory, in
//              the order of the hits.  A sieve of two bit maps of the slope
//              plane leaves the few hits that can be part of a passing triplet;
//              pairs and triples of those are tested, and the survivors of an
//              event's stations get the exact FP32 fit (P1) together.  CHAIN
//              mode keeps the passing trigger triplets' slopes in the tile
//              and holds the other stations' passing triplets against them
//              (P2).
//              Limits: 192 hits per layer, 384 per station, 32 passing trigger
//              triplets.
//   k_medium   the same sieve, with larger maps and one more pass, on 4-warp
//              blocks (384 hits per layer, 960 per station) for the events
//              k_light passes on.
//   k_heavy, k_heavy_units, k_heavy_final
//              8-warp blocks on the block tile (2048 hits per layer, 5632 per
//              station, 32 x 64 cells), the warps taking L0 rounds and
//              trigger-slope searches from a shared counter.  k_sort_heavy
//              orders these events largest first; k_heavy runs each one's
//              trigger station and, in CHAIN mode, hands the other stations
//              to k_heavy_units (one block per station, trigger slopes in a
//              batch-wide pool) and k_heavy_final (alive slopes left per
//              event).
//   k_generic  one block per event, unpruned where the pruning bound is not
//              finite (extreme coordinates) and no size limit: reads hits
//              straight from global memory.
//   k_accept   accept bits from track counts (ballot per 32 events).
//   k_scan*    exclusive scan of per-unit counts into int64 trip_off.
//   k_scatter  moves the triplets recorded by the counting pass to their rows
//              trip_off[unit] + rank; when the record overflowed, the emit
//              variants of the enumeration kernels re-enumerate instead.
//
// Every kernel takes the run's Job by value (a __grid_constant__ parameter).
// Pruning only skips triples that provably fail P1 (see jpsi_device.cuh), and
// P1/P2 are the same correctly rounded FP32 expressions everywhere.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "jpsi.h"
#include "jpsi_device.cuh"
#include "jpsi_internal.h"

// The file is compiled twice: JPSI_STREAM = 0 gives the event kernels
// (namespace jpsi::basek), JPSI_STREAM = 1 the same kernels with the time
// tests of free-streaming windows (jpsi::streamk); `if constexpr (kStream)`
// keeps those tests, and their registers, out of the event build.
#ifndef JPSI_STREAM
#define JPSI_STREAM 0
#endif
namespace jpsi {
#if JPSI_STREAM
namespace streamk {
#else
namespace basek {
#endif

constexpr bool kStream = JPSI_STREAM != 0;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kQCap = 128;                // pair queue entries per warp

// warp path: size limits of an event on it
constexpr int kTCap = 64;                 // passing trigger triplets per event on the medium tile (CHAIN)
struct SmallCfg {
    static constexpr int LAYER_CAP = 192;           // hits per layer
    static constexpr int HCAP = 384;                // hits per station
    static constexpr int TCAP = 32;                 // passing trigger triplets kept (CHAIN)
    static constexpr uint8_t CLS = kClsLight;       // event class of this path
};
// the size limits of the medium path (MediumTile below)
struct MediumCfg {
    static constexpr int LAYER_CAP = 384, HCAP = 960;
    static constexpr uint8_t CLS = kClsMedium;
};

// block-tile path: a block of THREADS threads stages a station (each thread
// up to RMAX hits per layer) into NY x NX cells per layer, and its warps
// share the station's enumeration rounds and trigger-slope searches
template <int THREADS_, int RMAX_, int HCAP_, int NX_, int NY_, uint8_t CLS_>
struct BCfg {
    static constexpr int THREADS = THREADS_, WARPS = THREADS_ / 32;
    static constexpr int RMAX = RMAX_;                   // hits per thread per layer
    static constexpr int LAYER_CAP = THREADS_ * RMAX_;   // hits per layer
    static constexpr int HCAP = HCAP_;                   // hits per station tile
    static constexpr int NX = NX_, NY = NY_, NC = NX_ * NY_;
    static constexpr uint8_t CLS = CLS_;                 // event class of this path
};
// the block tile proper: 8 warps, 2048 hits per layer, 5632 per station, 32 x 64 cells
using HeavyCfg = BCfg<256, 8, 5632, 64, 32, kClsHeavy>;
constexpr int kHThreads = HeavyCfg::THREADS;
constexpr int kHLayerCap = HeavyCfg::LAYER_CAP;
constexpr int kHHCap = HeavyCfg::HCAP;

struct LayerMeta {
    float lox, scx, loy, scy;  // cell map: column = bin of s_x, row = bin of s_y
    float bmax;                // largest pruning bound b of the layer
    float rmax, smax;          // largest r ~ 1/z and |s_x| + |s_y| (pair bounds)
    int32_t base;              // global index of the layer's first hit
    int32_t pbase;             // tile position of the layer's first stored hit
    int32_t nlive;             // stored hits (finite coordinates)
};

// One station staged in shared memory: hit slopes (s_x, s_y) and layer-local
// indices, sorted by layer then cell; cell starts and per-layer metadata.
template <int NX_, int NY_>
struct TileView {
    static constexpr int NX = NX_, NY = NY_, NC = NX_ * NY_;
    float2* P;
    uint16_t* idx;
    uint16_t* bst;  // [3 * NC + 1] tile positions: layer l, cell k at l * NC + k
    LayerMeta* meta;
};

// The warp path's memory: one station's hit slopes in the order of the hits,
// two maps of the slope plane, the hits that the sieve leaves of layers 0 and
// 2, triples that wait for their fit, and the event's trigger slopes.
constexpr int kMapRows = 128;             // a map has 128 rows (s_y) of 64 columns (s_x), both modulo
constexpr int kMapWords = 2 * kMapRows;   // word 2 y + (x >> 5), bit x
struct LayerMax {
    float r, s;                           // largest 1/z and |slope| of a layer's live hits
};
struct WarpTile {
    static constexpr int TCAP = SmallCfg::TCAP;
    static constexpr uint8_t CLS = kClsLight;
    float2 P[SmallCfg::HCAP + 32];        // (s_x, s_y); reads run up to 31 places past the last hit
    alignas(16) uint32_t map[2][kMapWords];
    uint32_t pend[64];                    // triples: station << 27 | i << 18 | j << 9 | k
    uint8_t left[2][SmallCfg::LAYER_CAP]; // layer-local indices of the hits that the sieve leaves
    int32_t off[3 * kMaxStations + 1];    // the event's offsets
    int32_t sh[kStream ? 3 * kMaxStations : 1];  // and shifts (free-streaming windows)
    int32_t count[kMaxStations];          // passing triplets per station
    float2 T[SmallCfg::TCAP];             // trigger triplet slopes
    using Slopes = uint32_t;              // one bit for each
    Slopes partners[kMaxStations];        // those that have a compatible triplet in the station (CHAIN)
    union {
        unsigned long long Tijk[SmallCfg::TCAP];  // their packed hits (distinct_hits)
        float2 Tt[SmallCfg::TCAP];                // or their (min t, max t) (free-streaming windows)
    };
    uint8_t alive[SmallCfg::TCAP];        // in every station (distinct_hits)
    LayerMax lay[3];                      // of an uneven station
    static_assert(SmallCfg::LAYER_CAP <= 256, "8-bit indices");
};

// The same for the four warps of a medium block (384 hits per layer, 960 per
// station): maps of 128 columns, what is left of all three layers, and pending
// triples for each warp.
struct MediumTile {
    static constexpr int THREADS = 128, WARPS = THREADS / 32, BLOCKS = 8, TCAP = kTCap;
    static constexpr uint8_t CLS = kClsMedium;
    float2 P[MediumCfg::HCAP + THREADS];
    alignas(16) uint32_t map[2][4 * kMapRows];  // word 4 y + (x >> 5), bit x
    uint32_t pend[WARPS][64];
    uint16_t left[3][MediumCfg::LAYER_CAP];
    int n_left[3];
    int32_t off[3 * kMaxStations + 1];
    int32_t sh[kStream ? 3 * kMaxStations : 1];
    int32_t count[kMaxStations];
    int red[WARPS][3];                          // largest |slope|, largest and smallest 1/z (bit patterns)
    int s_gi, s_flag;
    float2 T[TCAP];
    using Slopes = unsigned long long;
    Slopes partners[kMaxStations];
    union {
        unsigned long long Tijk[TCAP];
        float2 Tt[TCAP];
    };
    uint8_t alive[TCAP];
    LayerMax lay[3];                            // of an uneven station
    static_assert(MediumCfg::LAYER_CAP <= 512, "9-bit indices in pend");
};

template <class B>
struct BlockSmem {
    float2 P[B::HCAP];
    uint16_t idx[B::HCAP];
    uint32_t queue[B::WARPS][kQCap];
    uint32_t pend_pair[B::WARPS][32];        // triples that wait for their fit: i | j << 16 (tile positions)
    uint16_t pend_k[B::WARPS][32];           //   and k
    alignas(4) uint16_t bst[3 * B::NC + 1];  // cell starts (cell counts while a layer is staged)
    LayerMeta meta[3];
    int32_t off[3 * kMaxStations + 1];
    int32_t sh[kStream ? 3 * kMaxStations : 1];  // shifts (free-streaming windows)
    int32_t wsum[B::WARPS];
    int red_i[B::WARPS][2];
    int red_k[B::WARPS][7];
    unsigned long long s_pool;
    long long s_item;
    int s_gi, s_rank, s_nT, s_cand, s_hx, s_hy, s_next;
};
using HeavySmem = BlockSmem<HeavyCfg>;

// The kernels of a run are launched one behind the other with programmatic
// serialization.  chain_wait, the first statement of each: its work starts when the
// kernel before it is complete.  chain_next: the next kernel's blocks may be set
// up (and wait) once all blocks of this grid have come here or ended; small
// kernels say so at once, the persistent ones when they run out of work (earlier,
// the waiting blocks would keep shared memory from other streams' kernels:
// twelve timeslices over three serving slots 3.01 -> 3.17 ms).  Both are no-ops in
// a launch without the attribute.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;"); }

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// distinct_hits: do the candidates ijk[0, n) (those with alive set, when
// alive is given) hold two that use no common hit?  The warp walks the pair
// matrix in 32 x 32 tiles (candidate b of a tile comes by shuffle) and stops
// at the first tile with such a pair; warp-uniform result.  Block version:
// the warps take the rows of tiles in turn and stop at a block-shared flag.
__device__ __forceinline__ bool pair_tile_rows(const unsigned long long* ijk, const uint8_t* alive, int n, int a0,
                                               int lane) {
    const int a = a0 + lane;
    const bool va = a < n && (!alive || alive[a]);
    const unsigned long long ca = va ? ijk[a] : 0ull;
    for (int b0 = a0; b0 < n; b0 += 32) {
        const int b = b0 + lane;
        const bool vb = b < n && (!alive || alive[b]);
        const unsigned long long cb = vb ? ijk[b] : 0ull;
        bool f = false;
        for (int q = 0; q < 32; ++q) {
            const unsigned long long cq = __shfl_sync(0xffffffffu, cb, q);
            const bool vq = __shfl_sync(0xffffffffu, vb, q);
            f |= va & vq & (b0 + q > a) && ijk_disjoint(ca, cq);
        }
        if (__any_sync(0xffffffffu, f)) return true;
    }
    return false;
}

__device__ bool warp_disjoint_pair(const unsigned long long* ijk, const uint8_t* alive, int n, int lane) {
    for (int a0 = 0; a0 < n; a0 += 32)
        if (pair_tile_rows(ijk, alive, n, a0, lane)) return true;
    return false;
}

// All threads of the block call it; sh_flag is block-shared scratch.
template <int THREADS>
__device__ bool block_disjoint_pair(const unsigned long long* ijk, const uint8_t* alive, int n, int* sh_flag) {
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    if (threadIdx.x == 0) *sh_flag = 0;
    __syncthreads();
    for (int a0 = 32 * wp; a0 < n; a0 += THREADS) {
        if (__any_sync(0xffffffffu, *(volatile int*)sh_flag)) break;  // warp-uniform
        if (pair_tile_rows(ijk, alive, n, a0, lane)) {
            if (lane == 0) *(volatile int*)sh_flag = 1;
            break;
        }
    }
    return __syncthreads_or(*(volatile int*)sh_flag);
}

// Min/max of non-NaN floats through the integer reduction unit: the map is
// strictly increasing on floats ordered by value.
__device__ __forceinline__ int f2key(float f) {
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float key2f(int k) { return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff); }

__device__ __forceinline__ int warp_incl_scan(int v, int lane) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(kFull, v, d);
        if (lane >= d) v += o;
    }
    return v;
}

// Pulls the hit lines [h0, h1) of x, y, z into L2 (addresses stay inside the
// arrays: the first line starts at or after index h0 & ~31 >= 0).  At most
// 32 * 31 hits: one line of each array per lane.
__device__ __forceinline__ void prefetch_hits_l2(const Job& j, int32_t h0, int32_t h1, int lane) {
    const int32_t a = (h0 & ~31) + 32 * lane;
    if (a < h1) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(j.x + a));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(j.y + a));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(j.z + a));
    }
}

// The lines of station s of the event with these offsets (and shifts).
__device__ __forceinline__ void prefetch_station(const Job& j, const int32_t* off, const int32_t* sh, int s, int lane) {
    if (j.host_hits) return;
    if constexpr (kStream) {
#pragma unroll
        for (int l = 0; l < 3; ++l)
            prefetch_hits_l2(j, off[3 * s + l] + sh[3 * s + l], off[3 * s + l + 1] + sh[3 * s + l], lane);
    } else {
        prefetch_hits_l2(j, off[3 * s], off[3 * s + 3], lane);
    }
}

__device__ __forceinline__ int station_of(int si, int trig) { return si == 0 ? trig : (si - 1 < trig ? si - 1 : si); }

// Free-streaming windows: are the times a, b, c coincident (max t <=
// fl32(min t + dt))?  Also returns min and max.
__device__ __forceinline__ bool coincident3(float a, float b, float c, float dt, float& tmin, float& tmax) {
    tmin = fminf(fminf(a, b), c);
    tmax = fmaxf(fmaxf(a, b), c);
    return tmax <= __fadd_rn(tmin, dt);
}

// A partner triplet with times (pmin, pmax) of a trigger triplet with times
// T = (min, max): itself coincident, and the six hits together.
__device__ __forceinline__ bool partner_coincident(float pmin, float pmax, float2 T, float dt) {
    return pmax <= __fadd_rn(pmin, dt) && fmaxf(pmax, T.y) <= __fadd_rn(fminf(pmin, T.x), dt);
}

// Where a station's hits lie in the hit arrays: layer l at the station's own
// offsets plus shift[l].  Events lie there in CSR order (no shift); the windows of a
// timeslice are ranges of its layer groups, so their offsets only count hits.
struct Shift3 {
    int32_t a, b, c;
    __device__ __forceinline__ int32_t of(int l) const { return l == 0 ? a : l == 1 ? b : c; }
    // of the hit at place p of the station, whose layers 1 and 2 start at s1 and s2
    __device__ __forceinline__ int32_t at(int p, int s1, int s2) const {
        return !kStream ? 0 : p < s1 ? a : p < s2 ? b : c;
    }
};
__device__ __forceinline__ Shift3 shift3(const int32_t* sh, int s) {
    return kStream ? Shift3{sh[3 * s], sh[3 * s + 1], sh[3 * s + 2]} : Shift3{0, 0, 0};
}
constexpr int kShifts = kStream ? 3 * kMaxStations : 1;  // entries of an event's shifts in shared memory

// Cell histogram of the layer being staged on a block tile, kept in place in
// the layer's own cell-start array: two 16-bit counters per 32-bit word (a
// count never exceeds the layer's hit capacity, < 2^16, so no carry crosses
// into the neighbour).  Returns the hit's rank in its cell.
__device__ __forceinline__ int cell_count_add(uint16_t* cnt, int cell) {
    uint32_t* wd = reinterpret_cast<uint32_t*>(cnt) + (cell >> 1);
    const int sh = (cell & 1) << 4;
    return (int)((atomicAdd(wd, 1u << sh) >> sh) & 0xffffu);
}

// ------------------------------------------------------ block staging

// Block version of the staging (block-tile paths).
template <class B>
__device__ int stage_layer_block(const Job& j, BlockSmem<B>& sm, int l, int32_t base, int32_t n, int32_t pbase,
                                 int& nlive) {
    constexpr int CPT = B::NC / B::THREADS;  // cells per thread
    static_assert(B::NC % B::THREADS == 0, "cells per layer");
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    float sx[B::RMAX], sy[B::RMAX];
    int key[B::RMAX];  // cell << 16 | rank in the cell once binned; -1: not stored
    static_assert(CPT % 2 == 0, "two 16-bit cell counters per word");
    float lox = INFINITY, hix = -INFINITY, loy = INFINITY, hiy = -INFINITY, bmax = 0.0f, rmax = 0.0f, smax = 0.0f;
    bool zbad = false, wild = false;
    uint16_t* bst = sm.bst + l * B::NC;  // the end of layer l is the start of layer l + 1
#pragma unroll
    for (int q = 0; q < CPT / 2; ++q) reinterpret_cast<uint32_t*>(bst)[CPT / 2 * tid + q] = 0;
#pragma unroll
    for (int r = 0; r < B::RMAX; ++r) {
        key[r] = -1;
        sx[r] = sy[r] = 0.0f;
    }
#pragma unroll
    for (int r = 0; r < B::RMAX; ++r) {
        if (B::THREADS * r >= n) break;  // block-uniform
        const int h = tid + B::THREADS * r;
        const bool in = h < n;
        const int hc = in ? h : n - 1;
        const HitPrep p = hit_prep(__ldg(j.x + base + hc), __ldg(j.y + base + hc), __ldg(j.z + base + hc), j.K);
        zbad |= in & p.zbad;
        wild |= in & p.wild;
        const bool live = in & p.live & !p.wild;
        key[r] = live ? 0 : -1;
        sx[r] = p.sx;
        sy[r] = p.sy;
        lox = live ? fminf(lox, p.sx) : lox;
        hix = live ? fmaxf(hix, p.sx) : hix;
        loy = live ? fminf(loy, p.sy) : loy;
        hiy = live ? fmaxf(hiy, p.sy) : hiy;
        bmax = live ? fmaxf(bmax, p.b) : bmax;
        rmax = live ? fmaxf(rmax, p.r) : rmax;
        smax = live ? fmaxf(smax, p.l1) : smax;
    }
    // block-wide ranges, bounds and flags: a warp reduction of order-
    // preserving integer keys (the bounds and their parts are >= 0, so their
    // bit patterns already order like the values), one slot per warp, then
    // each warp reduces the slots itself
    int kv[7] = {f2key(lox), -f2key(hix), f2key(loy), -f2key(hiy), -__float_as_int(bmax), -__float_as_int(rmax),
                 -__float_as_int(smax)};  // minima (maxima negated; keys of finite values never overflow)
#pragma unroll
    for (int q = 0; q < 7; ++q) kv[q] = __reduce_min_sync(kFull, kv[q]);
    const int fz = __any_sync(kFull, zbad), fw = __any_sync(kFull, wild);
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 7; ++q) sm.red_k[wp][q] = kv[q];
        sm.red_i[wp][0] = fz;
        sm.red_i[wp][1] = fw;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 7; ++q) kv[q] = __reduce_min_sync(kFull, lane < B::WARPS ? sm.red_k[lane][q] : INT_MAX);
    const int anyz = __any_sync(kFull, lane < B::WARPS && sm.red_i[lane][0]);
    const int anyw = __any_sync(kFull, lane < B::WARPS && sm.red_i[lane][1]);
    lox = key2f(kv[0]);
    hix = key2f(-kv[1]);
    loy = key2f(kv[2]);
    hiy = key2f(-kv[3]);
    bmax = __int_as_float(-kv[4]);
    rmax = __int_as_float(-kv[5]);
    smax = __int_as_float(-kv[6]);
    // (red_k / red_i are written again only in the next layer, behind the
    // three barriers below)
    if (anyz) return 1;
    if (anyw) return 2;
    const float scx = bin_scale(lox, hix, B::NX), scy = bin_scale(loy, hiy, B::NY);
#pragma unroll
    for (int r = 0; r < B::RMAX; ++r) {
        if (B::THREADS * r >= n) break;
        if (key[r] >= 0) {
            const int cell = slope_bin<B::NY>(sy[r], loy, scy) * B::NX + slope_bin<B::NX>(sx[r], lox, scx);
            key[r] = JPSI_IN(j.ctrl, cell >= 0 && cell < B::NC) ? (cell << 16) | cell_count_add(bst, cell) : -1;
        }
    }
    __syncthreads();
    // block exclusive scan of the cell counts, CPT consecutive cells per thread
    int cs[CPT];
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < CPT; ++q) {
        cs[q] = (int)bst[CPT * tid + q];
        cnt += cs[q];
    }
    const int incl = warp_incl_scan(cnt, lane);
    if (lane == 31) sm.wsum[wp] = incl;
    __syncthreads();
    int woff = 0, total = 0;
    {  // the warps' offsets by a scan over the lanes
        const int ws = lane < B::WARPS ? sm.wsum[lane] : 0;
        const int wi = warp_incl_scan(ws, lane);
        woff = __shfl_sync(kFull, wi - ws, wp);
        total = __shfl_sync(kFull, wi, B::WARPS - 1);
    }
    int run = pbase + woff + incl - cnt;
#pragma unroll
    for (int q = 0; q < CPT; ++q) {
        bst[CPT * tid + q] = (uint16_t)run;
        run += cs[q];
    }
    if (tid == B::THREADS - 1) bst[B::NC] = (uint16_t)(pbase + total);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < B::RMAX; ++r) {
        if (B::THREADS * r >= n) break;
        if (key[r] >= 0) {
            const int pos = bst[key[r] >> 16] + (key[r] & 0xffff);
            if (JPSI_IN(j.ctrl, pos >= 0 && pos < B::HCAP)) {
                sm.P[pos] = make_float2(sx[r], sy[r]);
                sm.idx[pos] = (uint16_t)(tid + B::THREADS * r);
            }
        }
    }
    if (tid == 0) {
        LayerMeta m;
        m.lox = lox;
        m.scx = scx;
        m.loy = loy;
        m.scy = scy;
        m.bmax = bmax;
        m.rmax = rmax;
        m.smax = smax;
        m.base = base;
        m.pbase = pbase;
        m.nlive = total;
        sm.meta[l] = m;
    }
    // no barrier here: the next layer works on its own cells and tile
    // positions, and the caller synchronises before the tile is read
    nlive = total;
    return 0;
}

// Cell window of a query: columns [x0, x1] around c_x +- W_x, rows [y0, y1]
// around c_y +- W_y, each padded as in query_bins.  An intersection of
// windows may be empty (x0 > x1 or y0 > y1).
struct Win {
    int x0, x1, y0, y1;
};

template <class TV>
__device__ __forceinline__ Win cell_window(const TV& t, int l, float cx, float cy, float Wx, float Wy) {
    const LayerMeta& m = t.meta[l];
    Win w;
    query_bins<TV::NX>(cx, Wx, m.lox, m.scx, w.x0, w.x1);
    query_bins<TV::NY>(cy, Wy, m.loy, m.scy, w.y0, w.y1);
    return w;
}

__device__ __forceinline__ Win win_meet(const Win& a, const Win& b) {
    return Win{max(a.x0, b.x0), min(a.x1, b.x1), max(a.y0, b.y0), min(a.y1, b.y1)};
}

// Tile positions of window w in layer l as two runs: its first row
// [a, a + n0), and the positions from its second row's first column to its
// last row's last column [a2, a2 + n1) (every cell in between included, a
// superset when the window spans more than two rows; empty for one row).
template <class TV>
__device__ __forceinline__ void win_runs(const TV& t, int l, const Win& w, int& a, int& n0, int& a2, int& n1) {
    a = n0 = a2 = n1 = 0;
    if (w.x0 > w.x1 || w.y0 > w.y1) return;
    const uint16_t* b = t.bst + l * TV::NC;
    a = b[w.y0 * TV::NX + w.x0];
    n0 = b[w.y0 * TV::NX + w.x1 + 1] - a;
    if (w.y1 > w.y0) {
        a2 = b[(w.y0 + 1) * TV::NX + w.x0];
        n1 = b[w.y1 * TV::NX + w.x1 + 1] - a2;
    }
}

// ---------------------------------------------------------- enumeration

// Pair bound of the staged layers a and b (pair_bound in jpsi_device.cuh).
template <class TV>
__device__ __forceinline__ float layer_pair_bound(const TV& t, int a, int b, float K) {
    const LayerMeta &ma = t.meta[a], &mb = t.meta[b];
    return pair_bound(ma.rmax, ma.smax, mb.rmax, mb.smax, K);
}

// Where passing trigger triplets' slopes go (CHAIN mode, trigger station).
struct TSink {
    bool on;
    float2* T;
    int cap;
    int* sh_n;  // their number (block-shared)
    bool norec = false;  // a repeated enumeration: record no triplet entries
    unsigned long long* ijk = nullptr;  // distinct_hits: the triplets' packed hits beside T
    float2* tt = nullptr;               // free-streaming windows: their (min t, max t) beside T
};

// Triples that passed all pair tests and wait for their exact fit (block
// paths): the warp's m entries in shared memory.  The fits (and the global
// loads of their hits) then run 32 at a time.
struct Pending {
    uint32_t* pair;
    uint16_t* k;
    int m;
};

// P1 on the triples of the lanes with `has` (layer-local hits ii, jj, kk of
// the layers that start at base0, base1, base2) and what follows from a pass:
// the triplet's rank in its unit (from the block-shared counter), its row (emit pass), its slopes for the
// trigger sink (CHAIN) and its entry in the scatter record.  All lanes call it.
template <bool EMIT>
__device__ __forceinline__ void fit_and_record(const Job& j, int lane, const Cuts& c, bool has, int32_t base0,
                                               int32_t base1, int32_t base2, int ii, int jj, int kk, TSink& ts,
                                               int32_t* rows, int limit, int64_t unit, int* sh_rank, int tag) {
    bool ok = false;
    float mx = 0.f, my = 0.f;
    float2 tt = make_float2(0.f, 0.f);
    if (has) {
        const float xs[3] = {__ldg(j.x + base0 + ii), __ldg(j.x + base1 + jj), __ldg(j.x + base2 + kk)};
        const float ys[3] = {__ldg(j.y + base0 + ii), __ldg(j.y + base1 + jj), __ldg(j.y + base2 + kk)};
        const float zs[3] = {__ldg(j.z + base0 + ii), __ldg(j.z + base1 + jj), __ldg(j.z + base2 + kk)};
        ok = fit_pass(xs, ys, zs, c, mx, my);
        if constexpr (kStream) {  // coincident, and owned by this window
            const int64_t e = unit / j.S;
            ok = ok && coincident3(__ldg(j.t + base0 + ii), __ldg(j.t + base1 + jj), __ldg(j.t + base2 + kk), j.dt,
                                   tt.x, tt.y) &&
                 tt.x >= __ldg(j.wb + e) && tt.x < __ldg(j.wb + e + 1);
        }
    }
    const unsigned mask = __ballot_sync(kFull, ok);
    if (mask) {
        const int rk = __popc(mask & lanemask_lt()), np = __popc(mask);
        int base = 0;
        if (lane == 0) base = atomicAdd(sh_rank, np);
        base = __shfl_sync(kFull, base, 0);
        if (EMIT && ok && base + rk < limit &&  // never past the unit's rows
            JPSI_IN(j.ctrl, (rows - j.triplets) / 3 + base + rk < j.trip_cap)) {
            int32_t* r = rows + 3 * (int64_t)(base + rk);
            r[0] = ii;
            r[1] = jj;
            r[2] = kk;
        }
        if (ts.on) {
            int tb = 0;
            if (lane == 0) tb = atomicAdd(ts.sh_n, np);
            tb = __shfl_sync(kFull, tb, 0);
            if (ok && tb + rk < ts.cap) {
                ts.T[tb + rk] = make_float2(mx, my);
                if (ts.ijk) ts.ijk[tb + rk] = pack_ijk(ii, jj, kk);
                if (ts.tt) ts.tt[tb + rk] = tt;
            }
        }
        if (!EMIT && j.tscr && !ts.norec) {  // record for the scatter pass
            unsigned long long b = 0;
            if (lane == 0) b = atomicAdd(&j.ctrl->scratch_n, (unsigned long long)np);
            b = __shfl_sync(kFull, b, 0) + rk;
            if (ok && b < (unsigned long long)j.tscr_cap) {
                TripEntry te;
                te.unit = (int32_t)unit;
                te.rank = base + rk;
                te.ijk = (unsigned long long)ii | ((unsigned long long)jj << 20) | ((unsigned long long)kk << 40) |
                         ((unsigned long long)tag << kTagShift);
                j.tscr[b] = te;
            }
        }
    }
}

// The same on tile positions pi, pj, pk of a staged block tile.
template <bool EMIT, class TV>
__device__ __forceinline__ void fit_tile(const Job& j, const TV& t, int lane, const Cuts& c, bool has, int pi, int pj,
                                         int pk, TSink& ts, int32_t* rows, int limit, int64_t unit, int* sh_rank, int tag) {
    int ii = 0, jj = 0, kk = 0;
    if (has) {
        ii = t.idx[pi];
        jj = t.idx[pj];
        kk = t.idx[pk];
    }
    fit_and_record<EMIT>(j, lane, c, has, t.meta[0].base, t.meta[1].base, t.meta[2].base, ii, jj, kk, ts, rows, limit,
                         unit, sh_rank, tag);
}

// Drains a pair queue: every (i, j) against the L2 hits in the meet of both
// cell windows.  Each lane walks the window of its own pair (both runs), as long
// as the longest of the 32: pairs of one queue come from neighbouring hits, so
// their windows are alike, and a step costs a load, two pair tests and a vote.
// Triples that pass all pair tests join the pending ones, which are fitted 32 at
// a time.  (Spreading the items of all windows evenly over the lanes cost an
// owner search of five shuffles a step and two searches for the n-th set bit per
// vote: 2 000 dense events 12.06 -> 11.40 ms without them, the block tiles of
// 100 000 free-streaming collisions 2.21 -> 2.00 ms, of a 55 000-event log-normal
// timeslice 0.946 -> 0.913 ms.)
template <bool EMIT, class TV>
__device__ void drain(const Job& j, const TV& t, const uint32_t* queue, int lane, const Cuts& c, int qn,
                      TSink& ts, int32_t* rows, int limit, int64_t unit, int* sh_rank, int tag, Pending& pd) {
    const float B02 = layer_pair_bound(t, 0, 2, c.K), B12 = layer_pair_bound(t, 1, 2, c.K);
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll 1
    for (int q0 = 0; q0 < qn; q0 += 32) {
        const uint32_t en = queue[min(q0 + lane, qn - 1)];
        const float2 Pi = t.P[en & 0xffffu], Pj = t.P[en >> 16];
        int a = 0, m0 = 0, a2 = 0, m1 = 0;
        if (q0 + lane < qn) {
            const Win w = win_meet(cell_window(t, 2, Pi.x, Pi.y, B02, B02), cell_window(t, 2, Pj.x, Pj.y, B12, B12));
            win_runs(t, 2, w, a, m0, a2, m1);
        }
        const int len = m0 + m1, nmax = __reduce_max_sync(kFull, len);
#pragma unroll 1
        for (int k = 0; k < nmax; ++k) {
            const int pk = k < m0 ? a + k : a2 + (k - m0);
            const float2 Pk = t.P[k < len ? pk : 0];
            const bool cand = (k < len) & pair_ok(Pi.x, Pi.y, Pk.x, Pk.y, B02) & pair_ok(Pj.x, Pj.y, Pk.x, Pk.y, B12);
            const unsigned mask = __ballot_sync(kFull, cand);
            if (!mask) continue;
            const int at = pd.m + __popc(mask & lt);
            if (cand && at < 32) {
                pd.pair[at] = en;
                pd.k[at] = (uint16_t)pk;
            }
            pd.m += __popc(mask);
            if (pd.m >= 32) {
                __syncwarp();
                const uint32_t pe = pd.pair[lane];
                fit_tile<EMIT>(j, t, lane, c, true, (int)(pe & 0xffffu), (int)(pe >> 16), pd.k[lane], ts, rows, limit,
                               unit, sh_rank, tag);
                __syncwarp();
                if (cand && at >= 32) {
                    pd.pair[at - 32] = en;
                    pd.k[at - 32] = (uint16_t)pk;
                }
                pd.m -= 32;
            }
        }
    }
    __syncwarp();
}

// The pending triples of a block-path warp, at the end of its station.
template <bool EMIT, class TV>
__device__ __forceinline__ void flush_pending(const Job& j, const TV& t, int lane, const Cuts& c, TSink& ts,
                                              int32_t* rows, int limit, int64_t unit, int* sh_rank, int tag, Pending& pd) {
    if (pd.m > 0) {
        const uint32_t pe = pd.pair[min(lane, pd.m - 1)];
        fit_tile<EMIT>(j, t, lane, c, lane < pd.m, (int)(pe & 0xffffu), (int)(pe >> 16), pd.k[min(lane, pd.m - 1)], ts,
                       rows, limit, unit, sh_rank, tag);
    }
    pd.m = 0;
}

template <class TV>
__device__ bool road_warp(const Job& j, const TV& t, const Cuts& c, float mx, float my, float2 Tt, int lane);

// CHAIN-mode trigger slopes a block searches for while it enumerates a
// station (block path): item n_rounds + i of the block-shared counter is
// slope i; a slope with no compatible triplet in the station loses its flag.
struct RoadItems {
    const float2* T;
    uint8_t* alive;
    int n;
    const float2* Tt = nullptr;  // free-streaming windows: the slopes' (min t, max t)
};

// All passing triplets of the staged station (Sec. 3.2 steps 1-2) found by
// this warp: rounds of 32 L0 hits, taken from a counter that the warps of the
// block share.  Each lane walks its own hit's L1 window.  Pairs that may belong to
// a passing triplet are queued and drained against L2.
template <bool EMIT, class TV>
__device__ void enum_station(const Job& j, const TV& t, uint32_t* queue, Pending pd, int lane, const Cuts& c,
                            TSink& ts, int32_t* rows, int limit, int64_t unit, int* sh_rank, int tag, int* sh_next,
                            const RoadItems* rd) {
    const int n0 = t.meta[0].nlive, n1 = t.meta[1].nlive, n2 = t.meta[2].nlive;
    if (n0 == 0 || n1 == 0 || n2 == 0) return;
    const int n_rounds = (n0 + 31) >> 5;
    const int p0 = t.meta[0].pbase;
    const float B01 = layer_pair_bound(t, 0, 1, c.K);
    int qn = 0;
    // each warp takes the next round from the block-shared counter; items past
    // the rounds are trigger slopes to search for (CHAIN)
    auto next_round = [&]() {
        int g = 0;
        if (lane == 0) g = atomicAdd(sh_next, 1);
        return 32 * __shfl_sync(kFull, g, 0);
    };
    auto next_work = [&]() {
        int i0 = next_round();
        while (rd && i0 >= n0 && (i0 >> 5) - n_rounds < rd->n) {
            const int ti = (i0 >> 5) - n_rounds;
            if (rd->alive[ti]) {
                const float2 m = rd->T[ti];
                const bool found = road_warp(j, t, c, m.x, m.y, rd->Tt ? rd->Tt[ti] : make_float2(0.f, 0.f), lane);
                if (lane == 0 && !found) rd->alive[ti] = 0;
            }
            i0 = next_round();
        }
        return i0;
    };
    for (;;) {
        const int i0 = next_work();
        if (i0 >= n0) break;
        const bool has = i0 + lane < n0;
        const float2 Pi = t.P[p0 + (has ? i0 + lane : 0)];
        int a = 0, m0 = 0, a2 = 0, m1 = 0;
        if (has) win_runs(t, 1, cell_window(t, 1, Pi.x, Pi.y, B01, B01), a, m0, a2, m1);
        // each lane walks its own hit's window (both runs), as long as the
        // warp's longest: the 32 L0 hits of a round are neighbours in the cell
        // order, so their windows are alike
        const int len = m0 + m1;
        const int nmax = __reduce_max_sync(kFull, len);
#pragma unroll 1
        for (int k = 0; k < nmax; ++k) {
            const bool in = k < len;
            const int pj = k < m0 ? a + k : a2 + (k - m0);
            const float2 Pj = t.P[in ? pj : p0];
            const bool pass = in & pair_ok(Pi.x, Pi.y, Pj.x, Pj.y, B01);
            const unsigned mask = __ballot_sync(kFull, pass);
            if (!mask) continue;
            const int qi = qn + __popc(mask & lanemask_lt());
            if (pass && JPSI_IN(j.ctrl, qi < kQCap)) queue[qi] = (uint32_t)(p0 + i0 + lane) | ((uint32_t)pj << 16);
            qn += __popc(mask);
            if (qn > kQCap - 32) {
                __syncwarp();
                drain<EMIT>(j, t, queue, lane, c, qn, ts, rows, limit, unit, sh_rank, tag, pd);
                qn = 0;
            }
        }
    }
    __syncwarp();
    drain<EMIT>(j, t, queue, lane, c, qn, ts, rows, limit, unit, sh_rank, tag, pd);
    flush_pending<EMIT>(j, t, lane, c, ts, rows, limit, unit, sh_rank, tag, pd);
}

// Tile positions of a cell window, row by row: the first row's run [a, e)
// is given; windows of more than one row continue on the next rows (each
// row's columns [x0, x1] are one run of positions).
template <int NX>
struct WinIter {
    int p, end, row, y1, x0, x1;
    const uint16_t* bs;
    __device__ __forceinline__ WinIter(int a, int e, const uint16_t* b, const Win& w)
        : p(a), end(e), row(w.y0), y1(w.y1), x0(w.x0), x1(w.x1), bs(b) {
        settle();
    }
    __device__ __forceinline__ void settle() {
        while (p >= end && row < y1) {
            ++row;
            p = bs[row * NX + x0];
            end = bs[row * NX + x1 + 1];
        }
    }
    __device__ __forceinline__ bool valid() const { return p < end; }
    __device__ __forceinline__ void next() {
        ++p;
        settle();
    }
};

// Does the staged station hold a passing triplet compatible with the
// trigger slopes (mx, my)?  Per-thread search through each layer's cells
// inside the tube, row by row.
template <class TV>
__device__ bool road(const Job& j, const TV& t, const Cuts& c, float mx, float my, float2 Tt) {
    Win w[3];
    int a[3], e[3];  // first-row runs
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const float b = t.meta[l].bmax;
        w[l] = cell_window(t, l, mx, my, __fadd_rn(b, __fmul_rn(2.0f * kKappa, fabsf(mx))),
                           __fadd_rn(b, __fmul_rn(2.0f * kKappa, fabsf(my))));
        const uint16_t* bs = t.bst + l * TV::NC;
        a[l] = bs[w[l].y0 * TV::NX + w[l].x0];
        e[l] = bs[w[l].y0 * TV::NX + w[l].x1 + 1];
    }
    const uint16_t *bs0 = t.bst, *bs1 = t.bst + TV::NC, *bs2 = t.bst + 2 * TV::NC;
    const int32_t base0 = t.meta[0].base, base1 = t.meta[1].base, base2 = t.meta[2].base;
    const float b0 = t.meta[0].bmax, b1 = t.meta[1].bmax, b2 = t.meta[2].bmax;
    for (WinIter<TV::NX> i0(a[0], e[0], bs0, w[0]); i0.valid(); i0.next()) {
        const int p0 = i0.p;
        const float2 P0 = t.P[p0];
        if (!tube_ok(P0.x, P0.y, b0, mx, my)) continue;
        const int h0 = base0 + t.idx[p0];
        const float x0 = __ldg(j.x + h0), y0 = __ldg(j.y + h0), z0 = __ldg(j.z + h0);
        if (!tube_pass(x0, y0, z0, mx, my, c)) continue;
        for (WinIter<TV::NX> i1(a[1], e[1], bs1, w[1]); i1.valid(); i1.next()) {
            const int p1 = i1.p;
            const float2 P1 = t.P[p1];
            if (!tube_ok(P1.x, P1.y, b1, mx, my)) continue;
            const int h1 = base1 + t.idx[p1];
            const float x1 = __ldg(j.x + h1), y1 = __ldg(j.y + h1), z1 = __ldg(j.z + h1);
            if (!tube_pass(x1, y1, z1, mx, my, c)) continue;
            for (WinIter<TV::NX> i2(a[2], e[2], bs2, w[2]); i2.valid(); i2.next()) {
                const int p2 = i2.p;
                const float2 P2 = t.P[p2];
                if (!tube_ok(P2.x, P2.y, b2, mx, my)) continue;
                const int h2 = base2 + t.idx[p2];
                const float xs[3] = {x0, x1, __ldg(j.x + h2)};
                const float ys[3] = {y0, y1, __ldg(j.y + h2)};
                const float zs[3] = {z0, z1, __ldg(j.z + h2)};
                float fx, fy;
                if (fit_pass(xs, ys, zs, c, fx, fy) && chain_pass(xs, ys, zs, mx, my, c)) {
                    if constexpr (!kStream) return true;
                    float pmin, pmax;
                    coincident3(__ldg(j.t + h0), __ldg(j.t + h1), __ldg(j.t + h2), j.dt, pmin, pmax);
                    if (partner_coincident(pmin, pmax, Tt, j.dt)) return true;
                }
            }
        }
    }
    return false;
}

// Warp-cooperative road(): the 32 lanes search together for one trigger
// slope (mx, my warp-uniform).  For each layer they test the tube on the
// window's tile positions, row by row, 32 at a time, and keep the hits that
// pass tube_pass: the k-th kept hit of layer l sits in lane k's registers.
// Every combination of one kept hit per layer then gets P1 and P2.  A layer
// with more than 32 kept hits hands the slope to road() on one lane (no such
// limit).  Same answer as road(), warp-uniform.
template <class TV>
__device__ bool road_warp(const Job& j, const TV& t, const Cuts& c, float mx, float my, float2 Tt, int lane) {
    float hx[3] = {0.f, 0.f, 0.f}, hy[3] = {0.f, 0.f, 0.f}, hz[3] = {0.f, 0.f, 0.f}, ht[3] = {0.f, 0.f, 0.f};
    int nk[3] = {0, 0, 0};
    bool over = false;
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const float b = t.meta[l].bmax;
        const Win w = cell_window(t, l, mx, my, __fadd_rn(b, __fmul_rn(2.0f * kKappa, fabsf(mx))),
                                  __fadd_rn(b, __fmul_rn(2.0f * kKappa, fabsf(my))));
        const uint16_t* bs = t.bst + l * TV::NC;
        const int32_t base = t.meta[l].base;
        for (int row = w.y0; row <= w.y1 && !over; ++row) {
            const int a = bs[row * TV::NX + w.x0], e = bs[row * TV::NX + w.x1 + 1];
            for (int p0 = a; p0 < e; p0 += 32) {
                const int p = p0 + lane;
                bool keep = false;
                float x = 0.f, y = 0.f, z = 0.f, tm = 0.f;
                if (p < e) {
                    const float2 P = t.P[p];
                    if (tube_ok(P.x, P.y, b, mx, my)) {
                        const int h = base + t.idx[p];
                        x = __ldg(j.x + h);
                        y = __ldg(j.y + h);
                        z = __ldg(j.z + h);
                        if constexpr (kStream) tm = __ldg(j.t + h);
                        keep = tube_pass(x, y, z, mx, my, c);
                    }
                }
                unsigned m = __ballot_sync(kFull, keep);
                if (nk[l] + __popc(m) > 32) {
                    over = true;
                    break;
                }
                while (m) {  // the kept hits go to lanes nk, nk + 1, ...
                    const int src = __ffs(m) - 1;
                    m &= m - 1;
                    const float vx = __shfl_sync(kFull, x, src), vy = __shfl_sync(kFull, y, src),
                                vz = __shfl_sync(kFull, z, src), vt = __shfl_sync(kFull, tm, src);
                    if (lane == nk[l]) {
                        hx[l] = vx;
                        hy[l] = vy;
                        hz[l] = vz;
                        ht[l] = vt;
                    }
                    ++nk[l];
                }
            }
        }
        if (over) break;
        if (nk[l] == 0) return false;
    }
    if (over) {
        bool f = false;
        if (lane == 0) f = road(j, t, c, mx, my, Tt);
        return __shfl_sync(kFull, f, 0);
    }
    const int n01 = nk[0] * nk[1], total = n01 * nk[2];
    for (int it0 = 0; it0 < total; it0 += 32) {
        const int it = min(it0 + lane, total - 1);
        const int i2 = it / n01, r = it - i2 * n01, i1 = r / nk[0], i0 = r - i1 * nk[0];
        const float xs[3] = {__shfl_sync(kFull, hx[0], i0), __shfl_sync(kFull, hx[1], i1),
                             __shfl_sync(kFull, hx[2], i2)};
        const float ys[3] = {__shfl_sync(kFull, hy[0], i0), __shfl_sync(kFull, hy[1], i1),
                             __shfl_sync(kFull, hy[2], i2)};
        const float zs[3] = {__shfl_sync(kFull, hz[0], i0), __shfl_sync(kFull, hz[1], i1),
                             __shfl_sync(kFull, hz[2], i2)};
        float fx, fy;
        bool ok = fit_pass(xs, ys, zs, c, fx, fy) && chain_pass(xs, ys, zs, mx, my, c);
        if constexpr (kStream) {
            float pmin, pmax;
            coincident3(__shfl_sync(kFull, ht[0], i0), __shfl_sync(kFull, ht[1], i1), __shfl_sync(kFull, ht[2], i2),
                        j.dt, pmin, pmax);
            ok = ok && partner_coincident(pmin, pmax, Tt, j.dt);
        }
        if (__any_sync(kFull, ok)) return true;
    }
    return false;
}

// ------------------------------------------------------------ warp path

// A warp-uniform value in a uniform register: branches and addresses that come
// from it need no divergence handling (the compiler does not know that the
// result of a shuffle or of a load is uniform; that of a reduction is).
__device__ __forceinline__ int uniform(int v) { return __reduce_max_sync(kFull, v); }

// Largest |v| seen so far, NaN if any value was NaN.
__device__ __forceinline__ float max3_abs_nan(float m, float a, float b) {
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ float rcp_approx(float v) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// What the warp knows of the station it staged: the pair bound of any two of
// its hits, and the sieve's cells per unit of slope.
struct StationBounds {
    float B, inv;
};

// The bounds from the largest 1/z and |slope| of the station's hits.
__device__ __forceinline__ StationBounds station_bounds(float rmax, float smax, float K) {
    StationBounds sb;
    sb.B = station_pair_bound(rmax, smax, K);
    sb.inv = __fmul_rn(0.998f, rcp_approx(sb.B));
    return sb;
}

// One bound serves a station whose hits are alike.  A single hit at a small z
// or a huge slope would make it so wide that every triple of the station came to a
// fit (one such hit in every other event of 100 hits per layer: 0.2 -> 45 ms); such
// an uneven station gets a bound for each pair of its layers instead, as only the
// two pairs with that hit's layer are then wide.  Alike: 1/z within a factor of
// four, and slopes that add no more than a quarter to the bound (or below 8).
__device__ __forceinline__ bool even_hits(int rmax_bits, int rmin_bits, float rmax, float smax, float K) {
    return rmax_bits <= rmin_bits + (2 << 23) && smax <= fmaxf(8.0f, __fmul_rn(11585.0f * K, rmax));
}

// The bounds of the three pairs of layers.
struct PairBounds {
    float b01, b02, b12;
};
__device__ __forceinline__ bool uneven_bounds(const PairBounds& b, float B) {
    return fminf(fminf(b.b01, b.b02), b.b12) < 0.5f * B;
}
__device__ __forceinline__ PairBounds pair_bounds(const LayerMax* lay, float K) {
    const float b[3] = {lay[0].r, lay[1].r, lay[2].r}, m[3] = {lay[0].s, lay[1].s, lay[2].s};
    return {station_pair_bound(fmaxf(b[0], b[1]), fmaxf(m[0], m[1]), K),
            station_pair_bound(fmaxf(b[0], b[2]), fmaxf(m[0], m[2]), K),
            station_pair_bound(fmaxf(b[1], b[2]), fmaxf(m[1], m[2]), K)};
}

// Exact classification of the station's hits (n places from o0 on), for stations
// with an odd coordinate or uneven hits: their slopes to P, (Inf, Inf) for a hit
// with a non-finite coordinate (it passes no finite bound, and no fit in any case),
// and each layer's maxima to `lay`.  Returns 0, 1 (z <= 0) or 2 (a hit whose
// pruning bound is not finite).
__device__ __forceinline__ int sieve_classify(const Job& j, float2* P, int lane, int32_t o0, int s1, int s2, int n,
                                              const Shift3& sh, LayerMax* lay, float& rmax, float& smax) {
    bool zbad = false, wild = false;
    rmax = smax = 0.0f;
    __syncwarp();  // (the slopes written so far)
#pragma unroll 1
    for (int l = 0; l < 3; ++l) {
        float r = 0.0f, sl = 0.0f;
        const int end = l == 0 ? s1 : l == 1 ? s2 : n;
#pragma unroll 1
        for (int p = (l == 0 ? 0 : l == 1 ? s1 : s2) + lane; p < end; p += 32) {
            const int32_t g = o0 + p + (kStream ? sh.of(l) : 0);
            const HitPrep h = hit_prep(__ldg(j.x + g), __ldg(j.y + g), __ldg(j.z + g), j.K);
            zbad |= h.zbad;
            wild |= h.wild;
            const bool live = h.live & !h.wild;
            P[p] = live ? make_float2(h.sx, h.sy) : make_float2(INFINITY, INFINITY);
            if (live) {
                sl = fmaxf(sl, fmaxf(fabsf(h.sx), fabsf(h.sy)));
                r = fmaxf(r, h.r);
            }
        }
        sl = __int_as_float(__reduce_max_sync(kFull, __float_as_int(sl)));
        r = __int_as_float(__reduce_max_sync(kFull, __float_as_int(r)));
        if (lane == 0) lay[l] = LayerMax{r, sl};
        smax = fmaxf(smax, sl);
        rmax = fmaxf(rmax, r);
    }
    __syncwarp();
    return __any_sync(kFull, zbad) ? 1 : __any_sync(kFull, wild) ? 2 : 0;
}

// The cell of a slope: the nearest integer of s * inv, modulo the map's size
// when it is used.  A bound is at least 2 kappa times the largest |s| that it is
// used on, so |s * inv| <= 2^16 (1 + 2^-20), and the sum with 1.5 * 2^23 holds that
// integer in its low mantissa bits (one rounding).  Hits of one passing
// triplet lie within B (1 - 5e-5) of each other (jpsi_device.cuh) and inv <=
// 0.998 (1 + 2^-22) / B, so their s * inv differ by less than 1 and their
// cells by at most 1.
__device__ __forceinline__ int sieve_cell(float s, float inv) { return __float_as_int(__fmaf_rn(s, inv, 12582912.0f)); }
struct SieveBit {
    int word;
    uint32_t bit;
};
__device__ __forceinline__ SieveBit sieve_bit(float2 s, float inv) {
    const int cx = sieve_cell(s.x, inv), cy = sieve_cell(s.y, inv);
    return {((cy & (kMapRows - 1)) << 1) + ((cx >> 5) & 1), __funnelshift_l(0u, 1u, cx)};  // (1 << (cx & 31))
}

// Dilates the map by one cell to all sides (rows and columns are rings) and,
// with MEET, keeps only the cells of `other`.  Lane l has the rows 4 l .. 4 l + 3.
template <bool MEET>
__device__ __forceinline__ void sieve_dilate(uint32_t* map, const uint32_t* other, int lane) {
    __syncwarp();
    const uint4 a = reinterpret_cast<const uint4*>(map)[2 * lane], b = reinterpret_cast<const uint4*>(map)[2 * lane + 1];
    uint32_t r[12] = {0u, 0u, a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, 0u, 0u};
    r[0] = __shfl_sync(kFull, b.z, lane + 31);  // (source lane modulo 32)
    r[1] = __shfl_sync(kFull, b.w, lane + 31);
    r[10] = __shfl_sync(kFull, a.x, lane + 1);
    r[11] = __shfl_sync(kFull, a.y, lane + 1);
    uint4 oa = make_uint4(~0u, ~0u, ~0u, ~0u), ob = oa;
    if (MEET) {
        oa = reinterpret_cast<const uint4*>(other)[2 * lane];
        ob = reinterpret_cast<const uint4*>(other)[2 * lane + 1];
    }
    const uint32_t o[8] = {oa.x, oa.y, oa.z, oa.w, ob.x, ob.y, ob.z, ob.w};
    uint32_t d[8];
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
        const uint32_t lo = r[q] | r[q + 2] | r[q + 4], hi = r[q + 1] | r[q + 3] | r[q + 5];
        d[q] = (lo | __funnelshift_l(hi, lo, 1) | __funnelshift_r(lo, hi, 1)) & o[q];
        d[q + 1] = (hi | __funnelshift_l(lo, hi, 1) | __funnelshift_r(hi, lo, 1)) & o[q + 1];
    }
    __syncwarp();
    reinterpret_cast<uint4*>(map)[2 * lane] = make_uint4(d[0], d[1], d[2], d[3]);
    reinterpret_cast<uint4*>(map)[2 * lane + 1] = make_uint4(d[4], d[5], d[6], d[7]);
    __syncwarp();
}

// P1 on the warp's pending triples, 32 at a time, until at most `keep` of its np
// are left (their number is returned), and what follows from a pass: the
// triplet's rank in its unit (from the station's count), its row (emit pass),
// its slopes if it is a trigger triplet and the event keeps them (`sink`), the nT
// trigger slopes that it is compatible with (P2; nT is 0 until they are all known),
// and its entry in the scatter record.
//   The search finds every triplet of a station that passes P1, so the compatible
// ones are among these, and P2 costs some 30 instructions per slope for 32 of them.
// (A search of the station's hits for each slope, in turn, cost events with many
// tracks more than all else: 20 000 events of 20 tracks and 5 other hits per layer
// 600 us, 232 now (287 with one slope per lane on the cell-sorted tile); of 30
// tracks and 60 hits 1 070, 554 (794).)
template <bool EMIT, class W>
__device__ __forceinline__ int light_fit(const Job& j, W& w, const uint32_t* pend, int lane, const Cuts& c, int64_t e,
                                         bool sink, int nT, int np, int keep) {
    __syncwarp();
#pragma unroll 1
    while (np > keep) {
        const int n = min(np, 32), first = np - n;
        np = first;
        bool ok = false;
        float mx = 0.f, my = 0.f;
        float2 tt = make_float2(0.f, 0.f);
        int st = 0, ii = 0, jj = 0, kk = 0;
        if (lane < n) {
            const uint32_t en = pend[first + lane];
            st = en >> 27;
            ii = (en >> 18) & 511;
            jj = (en >> 9) & 511;
            kk = en & 511;
            const Shift3 sh = shift3(w.sh, st);
            const int32_t h0 = w.off[3 * st] + ii + sh.a, h1 = w.off[3 * st + 1] + jj + sh.b,
                          h2 = w.off[3 * st + 2] + kk + sh.c;
            const float xs[3] = {__ldg(j.x + h0), __ldg(j.x + h1), __ldg(j.x + h2)};
            const float ys[3] = {__ldg(j.y + h0), __ldg(j.y + h1), __ldg(j.y + h2)};
            const float zs[3] = {__ldg(j.z + h0), __ldg(j.z + h1), __ldg(j.z + h2)};
            ok = fit_pass(xs, ys, zs, c, mx, my);
            if constexpr (kStream)
                ok = ok && coincident3(__ldg(j.t + h0), __ldg(j.t + h1), __ldg(j.t + h2), j.dt, tt.x, tt.y);
            if (!EMIT && ok) {
                typename W::Slopes with = 0;
#pragma unroll 1
                for (int ti = 0; ti < nT; ++ti) {
                    const float2 m = w.T[ti];
                    if (chain_pass(xs, ys, zs, m.x, m.y, c) &&
                        (!kStream || partner_coincident(tt.x, tt.y, w.Tt[ti], j.dt)))
                        with |= (typename W::Slopes)1 << ti;
                }
                if (with) atomicOr(&w.partners[st], with);
            }
            // (free-streaming windows: a triplet counts where it is owned, a partner anywhere)
            if constexpr (kStream) ok = ok && tt.x >= __ldg(j.wb + e) && tt.x < __ldg(j.wb + e + 1);
        }
        int rank = 0;
        if (ok) {
            rank = atomicAdd(&w.count[st], 1);
            if (sink && st == j.trig && rank < W::TCAP) {
                w.T[rank] = make_float2(mx, my);
                if (j.distinct) w.Tijk[rank] = pack_ijk(ii, jj, kk);
                if (kStream) w.Tt[rank] = tt;
            }
        }
        if (EMIT) {
            const int64_t u = e * j.S + st;
            if (ok && rank < j.unit_counts[u]) {  // never past the unit's rows
                const int64_t row = j.trip_off[u] + rank;
                if (JPSI_IN(j.ctrl, row >= 0 && row < j.trip_cap)) {
                    int32_t* r = j.triplets + 3 * row;
                    r[0] = ii;
                    r[1] = jj;
                    r[2] = kk;
                }
            }
        } else if (j.tscr) {  // record for the scatter pass
            const unsigned mask = __ballot_sync(kFull, ok);
            if (mask) {
                unsigned long long b = 0;
                if (lane == 0) b = atomicAdd(&j.ctrl->scratch_n, (unsigned long long)__popc(mask));
                b = __shfl_sync(kFull, b, 0) + __popc(mask & ((1u << lane) - 1u));
                if (ok && b < (unsigned long long)j.tscr_cap) {
                    TripEntry te;
                    te.unit = (int32_t)(e * j.S + st);
                    te.rank = rank;
                    te.ijk = (unsigned long long)ii | ((unsigned long long)jj << 20) | ((unsigned long long)kk << 40) |
                             ((unsigned long long)W::CLS << kTagShift);
                    j.tscr[b] = te;
                }
            }
        }
        __syncwarp();
    }
    return np;
}

// The slopes of a station's hits [o0, o0 + n0 + n1 + n2) (its three layers in
// turn, each of at most 32 R hits) to P, in the order of the hits, and the largest
// 1/z and |slope|.  Returns false, P then incomplete, for hits that want
// sieve_classify: NaN, an infinity or 1/z outside (2^-126, 2^126) among the hits
// read, uneven hits (even_hits), or a station so close to the end of the hit arrays that the lanes past
// the end of a layer, which read on into the hits behind it, would leave them.
template <int R>
__device__ __forceinline__ bool sieve_stage(const Job& j, WarpTile& w, int lane, int32_t o0, int n0, int n1, int n2,
                                            const Shift3& sh, float& rmax, float& smax) {
    const int nl[3] = {n0, n1, n2}, sl[3] = {0, n0, n0 + n1};
    rmax = smax = 0.0f;
    // hits read over the host link: none that is not needed (200 000 events of 20
    // hits per layer, PAPER: 1.69 ms with full rounds, 1.11 without)
    if (j.host_hits) return false;
    if constexpr (kStream) {
        if ((int64_t)o0 + max(max(sh.a, sl[1] + sh.b), sl[2] + sh.c) + 32 * R > j.n_src) return false;
    } else if ((int64_t)o0 + sl[2] + 32 * R > j.n_src) {
        return false;
    }
    float rmin = INFINITY;
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const int32_t hs = kStream ? sh.of(l) : 0;
        const float *px = j.x + o0 + sl[l] + hs + lane, *py = j.y + o0 + sl[l] + hs + lane,
                    *pz = j.z + o0 + sl[l] + hs + lane;
        float x[R], y[R], z[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            x[r] = __ldg(px + 32 * r);
            y[r] = __ldg(py + 32 * r);
            z[r] = __ldg(pz + 32 * r);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float iz = rcp_approx(z[r]);
            const float2 v = make_float2(__fmul_rn(x[r], iz), __fmul_rn(y[r], iz));
            smax = max3_abs_nan(smax, v.x, v.y);
            if (32 * r + lane < nl[l]) w.P[sl[l] + lane + 32 * r] = v;
            z[r] = iz;
        }
#pragma unroll
        for (int r = 0; r < R; r += 2) {
            rmin = fminf(fminf(z[r], z[r + 1]), rmin);
            // (the hits behind layer 2 may be another event's, at half the z)
            const bool a = l < 2 || 32 * r + lane < n2, b = l < 2 || 32 * r + 32 + lane < n2;
            rmax = max3_abs_nan(rmax, a ? z[r] : 0.0f, b ? z[r + 1] : 0.0f);
        }
    }
    // floats >= 0 (and the NaN of the maxima) order like their bit patterns; a
    // negative 1/z has a negative pattern
    const int si = __reduce_max_sync(kFull, __float_as_int(smax)), ri = __reduce_max_sync(kFull, __float_as_int(rmax)),
              ni = __reduce_min_sync(kFull, __float_as_int(rmin));
    smax = __int_as_float(si);
    rmax = __int_as_float(ri);
    return si < 0x7f800000 && ri < 0x7e800000 && ni > 0x00800000 && even_hits(ri, ni, rmax, smax, j.K);
}

// The sieve of the staged station: which hits of layers 0 and 2 can be part of a
// triple whose pairs are all close enough to pass.  Their layer-local indices go
// to left[0][0, m0) and left[1][0, m2).
//   A station of about 100 hits per layer holds about 0.3 such triples, so the
// work is to find the few hits that can be part of one, in maps of the slope
// plane whose cells are as wide as the pair bound: hits set their cells, a map
// is dilated by one cell, and a hit of another layer is close to one of them
// only if its cell is set.  First layer 0 is held against layer 1, then layer 2
// against what is left of layer 0 and against layer 1.  Of 100 hits per layer of
// the 10^6-event workload 14 to 20 of layer 0 and 2 to 4 of layer 2 are left.
// Cells repeat every 64 columns and 128 rows, which only lets more through.
//   Instructions bound this code, so it is straight-line: R rounds of a layer,
// predicates instead of branches, the loads of all rounds before what depends on
// them.
template <int R>
__device__ __forceinline__ void sieve_layers(const Job& j, WarpTile& w, int lane, int n0, int n1, int n2, float inv,
                                             int& m0, int& m2) {
    const int nl[3] = {n0, n1, n2}, sl[3] = {0, n0, n0 + n1};
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t *ma = w.map[0], *mb = w.map[1];
    // slope of place sl[l] + 32 r + lane; past the end of the layer whatever the tile holds there
    static_assert(sizeof(WarpTile) >= (2 * SmallCfg::LAYER_CAP + 32 * R) * sizeof(float2), "reads stay in the tile");
    auto slope = [&](int l, int r) { return reinterpret_cast<const float2*>(&w)[sl[l] + lane + 32 * r]; };
#pragma unroll
    for (int q = 0; q < 4; ++q) reinterpret_cast<uint4*>(w.map)[32 * q + lane] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    {   // layer 1 sets its cells
        SieveBit b[R];
#pragma unroll
        for (int r = 0; r < R; ++r) b[r] = sieve_bit(slope(1, r), inv);
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (32 * r + lane < n1) atomicOr(&ma[b[r].word], b[r].bit);
    }
    sieve_dilate<false>(ma, nullptr, lane);
    // the hits of layer l whose cells are set in `map`: their indices to `left`, their cells to `mark`
    auto pass = [&](int l, const uint32_t* map, uint32_t* mark, uint8_t* left) {
        SieveBit b[R];
        uint32_t word[R];
        int m = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            b[r] = sieve_bit(slope(l, r), inv);
            word[r] = map[b[r].word];
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const bool in = (32 * r + lane < nl[l]) & ((word[r] & b[r].bit) != 0);
            const unsigned mask = __ballot_sync(kFull, in);
            const int at = m + __popc(mask & lt);
            if (mark && in) atomicOr(&mark[b[r].word], b[r].bit);
            if (in && JPSI_IN(j.ctrl, at < SmallCfg::LAYER_CAP)) left[at] = (uint8_t)(32 * r + lane);
            m += __popc(mask);
        }
        return uniform(m);
    };
    m2 = 0;
    m0 = pass(0, ma, mb, w.left[0]);
    if (m0 > 0) {
        sieve_dilate<true>(mb, ma, lane);
        m2 = pass(2, mb, nullptr, w.left[1]);
    }
    __syncwarp();
}

// Crowded stations (wide windows: the maps let most hits through).  Trying every
// hit that is left with every other grows with the square of the hits, so there two
// of the layers are put in the order of their cells' rows, and a hit looks at three
// rows of them.  The hits of the outer layer find partners in the middle one (the
// pair of layers with the tightest bound), those pairs find theirs in the last:
// layers 2, 1 and 0 unless the hits are uneven.
// Bound by instruction issue: two passes over the hits make the lists, then a step
// of a walk is two loads, the pair test and a vote for 32 hits.
//   The lists, and what a search keeps from one fit to the next, take the maps'
// memory, which is free by then: in registers they cost the stations that never come
// here 9 %.  Loops run to uniform() ends: one that the compiler cannot show to be
// the same for all lanes makes it prepare every vote and reduction of the kernel for
// diverged warps, which is half as much code again (k_light 58 -> 91 KB) and then a
// wait for instructions (10^6 events 4.61 -> 5.5 to 6.4 ms).
//   L: the type of the indices; MAX: hits per layer; Q: warps.
constexpr int kRowQueue = 64;
struct RowState {
    // outer hits from `due` on have not looked, the next 32 of them from step t of
    // their rows on; pairs waiting in the queue and, behind them, looking for
    // partners, from step u of their rows on.  Kept as due | t << 10 | waiting << 20
    // and looking | u << 8.
    int due, t, waiting, looking, u;
    __device__ __forceinline__ explicit RowState(const int2& p) {
        const int a = uniform(p.x), b = uniform(p.y);
        due = a & 1023;
        t = a >> 10 & 1023;
        waiting = a >> 20;
        looking = b & 255;
        u = b >> 8;
    }
    __device__ __forceinline__ int2 packed() const {
        return make_int2(due | t << 10 | waiting << 20, looking | u << 8);
    }
};
template <class L, int MAX, int Q>
struct RowLists {
    uint32_t end[2][kMapRows];     // where each row's hits end (middle, last layer)
    L order[2][MAX];               // layer-local indices by row
    uint32_t queue[Q][kRowQueue];  // pairs, as they stand in the pending triples
    int2 state[Q];                 // RowState, packed
    int n_out, start[3], shift[3];  // hits of the outer layer; places and index shifts of outer, middle and last
    float b, b_out, b_mid;          // bounds of the pairs outer - middle, outer - last, middle - last
    float inv[2];                   // cells per unit of slope of middle and last
    bool from_out;                  // partners in the last layer are looked for around the outer hit
};

// The row of a hit's cell.
__device__ __forceinline__ int sieve_row(float2 s, float inv) { return sieve_cell(s.y, inv) & (kMapRows - 1); }

// Fills the lists from m0, m1, m2 hits of the layers, whose indices are in `left` from
// 0, f1 and f2 on (all of layer 1 when f1 < 0) and whose slopes start at places 0, s1
// and s2.  All T threads (a warp or a block) call it.
template <int T, class R, class L>
__device__ __forceinline__ void row_lists(const Job& j, R& r, const float2* P, int tid, const PairBounds& pb,
                                          const L* left, int m0, int f1, int m1, int f2, int m2, int s1, int s2) {
    auto sync = [] {
        if constexpr (T == 32)
            __syncwarp();
        else
            __syncthreads();
    };
    const int lane = tid & 31;
    const bool from0 = pb.b01 < pb.b12 && pb.b01 <= pb.b02, over1 = pb.b02 < pb.b12 && pb.b02 < pb.b01;
    const int f_mid = over1 ? 0 : f1, f_last = over1 ? f1 : from0 ? f2 : 0;
    const int n_mid = over1 ? m0 : m1, n_last = over1 ? m1 : from0 ? m2 : m0;
    const int p_mid = over1 ? 0 : s1, p_last = over1 ? s1 : from0 ? s2 : 0;
    sync();  // the maps are done with
    for (int q = tid; q < 2 * kMapRows; q += T) r.end[0][q] = 0u;
    if (tid < T / 32) r.state[tid] = make_int2(tid, 0);
    if (tid == 0) {
        r.n_out = from0 ? m0 : m2;
        const int out_l = from0 ? 0 : 2, mid_l = over1 ? 0 : 1, last_l = 3 - out_l - mid_l;
        r.start[0] = from0 ? 0 : s2;
        r.start[1] = p_mid;
        r.start[2] = p_last;
        r.shift[0] = 18 - 9 * out_l;
        r.shift[1] = 18 - 9 * mid_l;
        r.shift[2] = 18 - 9 * last_l;
        r.b = over1 ? pb.b02 : from0 ? pb.b01 : pb.b12;
        r.b_out = over1 ? pb.b12 : pb.b02;
        r.b_mid = over1 || !from0 ? pb.b01 : pb.b12;
        r.from_out = r.b_out < r.b_mid;
        r.inv[0] = __fmul_rn(0.998f, rcp_approx(r.b));
        r.inv[1] = __fmul_rn(0.998f, rcp_approx(fminf(r.b_out, r.b_mid)));
    }
    sync();
    // twice over the hits: each row's size, then their places (which turn the rows'
    // starts into their ends)
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
        for (int w = 0; w < 2; ++w) {
            const int f = w ? f_last : f_mid, n = uniform(w ? n_last : n_mid);
            const float2* slopes = P + (w ? p_last : p_mid);
            const float inv = r.inv[w];
#pragma unroll 1
            for (int q0 = 0; q0 < n; q0 += T) {
                const int q = q0 + tid;
                if (q >= n) continue;
                const int h = f >= 0 ? (int)left[f + q] : q;
                const uint32_t at = atomicAdd(&r.end[w][sieve_row(slopes[h], inv)], 1u);
                if (pass && JPSI_IN(j.ctrl, at < sizeof(r.order[0]) / sizeof(L))) r.order[w][at] = (L)h;
            }
        }
        sync();
        if (!pass && (T == 32 || tid < 32)) {  // four rows a lane
#pragma unroll
            for (int w = 0; w < 2; ++w) {
                uint4* p = reinterpret_cast<uint4*>(r.end[w]) + lane;
                const uint4 c = *p;
                const uint32_t sum = c.x + c.y + c.z + c.w, b = (uint32_t)warp_incl_scan((int)sum, lane) - sum;
                *p = make_uint4(b, b + c.x, b + c.x + c.y, b + c.x + c.y + c.z);
            }
        }
        if (!pass) sync();
    }
}

// The hits of a row and of the rows beside it (a ring): up to two runs of the order.
struct RowRuns {
    int a, n, a2, len;  // the first run [a, a + n), the second from a2; hits of both
    __device__ __forceinline__ int at(int t) const { return t < n ? a + t : a2 + (t - n); }
};
__device__ __forceinline__ RowRuns row_runs(const uint32_t* end, int row) {
    constexpr int kLast = kMapRows - 1;
    RowRuns w;
    w.a = row > 1 ? (int)end[row - 2] : 0;
    w.n = (int)end[min(row + 1, kLast)] - w.a;
    w.a2 = row == 0 ? (int)end[kLast - 1] : 0;
    w.len = w.n + (row == 0 ? (int)(end[kLast] - end[kLast - 1]) : row == kLast ? (int)end[0] : 0);
    return w;
}

// Searches on until more than 32 triples (np) are pending or, then returning false,
// to the end: 32 hits of the outer layer at a time (this warp's are wp + k_step (32 b +
// lane)) look for partners in their rows, and 32 of the pairs found for theirs, each
// lane walking its own runs.
template <class R, class L>
__device__ __forceinline__ bool row_search(const Job& j, const float2* P, uint32_t* pend, R& r, int wp, int k_step,
                                           uint32_t station, const L* l0, const L* l2, int lane, int& np) {
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t* queue = r.queue[wp];
    RowState st(r.state[wp]);
    const int so = r.shift[0], sm = r.shift[1], sl = r.shift[2];
    const float2 *outer = P + r.start[0], *middle = P + r.start[1], *last = P + r.start[2];
    bool more = true;
#pragma unroll 1
    do {
        if (st.looking == 0) {
            const int n = uniform(r.n_out);
            const L* out = so ? l0 : l2;
#pragma unroll 1
            while (st.waiting < 32 && st.due < n) {
                const int k = st.due + k_step * lane;
                const int ho = out[min(k, n - 1)];
                const float2 O = outer[ho];
                const RowRuns w = row_runs(r.end[0], sieve_row(O, r.inv[0]));
                const int len = k < n ? w.len : 0, steps = __reduce_max_sync(kFull, len);
                const float B = r.b;
#pragma unroll 1
                for (; st.t < steps && st.waiting < 32; ++st.t) {
                    const bool in = st.t < len;
                    const int hm = r.order[0][in ? w.at(st.t) : 0];
                    const float2 M = middle[hm];
                    const bool pass = in & pair_ok(M.x, M.y, O.x, O.y, B);
                    const unsigned mask = __ballot_sync(kFull, pass);
                    const int at = st.waiting + __popc(mask & lt);
                    if (pass && JPSI_IN(j.ctrl, at < kRowQueue)) queue[at] = (uint32_t)ho << so | (uint32_t)hm << sm;
                    st.waiting += __popc(mask);
                }
                const int both = uniform(st.waiting | st.t << 8);
                st.waiting = both & 255;
                st.t = both >> 8;
                if (st.t >= steps) {
                    st.due += 32 * k_step;
                    st.t = 0;
                }
            }
            if (st.waiting == 0) {
                more = false;
                break;
            }
            st.looking = min(st.waiting, 32);
            st.waiting -= st.looking;
            st.u = 0;
            __syncwarp();
        }
        const uint32_t en = queue[st.waiting + min(lane, st.looking - 1)];
        const float2 O = outer[en >> so & 511u], M = middle[en >> sm & 511u];
        const RowRuns w = row_runs(r.end[1], sieve_row(r.from_out ? O : M, r.inv[1]));
        const int len = lane < st.looking ? w.len : 0, steps = __reduce_max_sync(kFull, len);
        const float bo = r.b_out, bm = r.b_mid;
#pragma unroll 1
        for (; st.u < steps && np <= 32; ++st.u) {
            const bool in = st.u < len;
            const int hl = r.order[1][in ? w.at(st.u) : 0];
            const float2 Z = last[hl];
            const bool cand = in & pair_ok(Z.x, Z.y, O.x, O.y, bo) & pair_ok(Z.x, Z.y, M.x, M.y, bm);
            const unsigned mask = __ballot_sync(kFull, cand);
            const int at = np + __popc(mask & lt);
            if (cand && JPSI_IN(j.ctrl, at < 64)) pend[at] = station | en | (uint32_t)hl << sl;
            np += __popc(mask);
        }
        const int both = uniform(np | st.u << 8);
        np = both & 255;
        st.u = both >> 8;
        if (st.u >= steps) st.looking = 0;
    } while (np <= 32);
    __syncwarp();
    if (lane == 0) r.state[wp] = st.packed();
    return more;
}

// The triples whose pairs are all close enough, among the hits that the sieve
// left of layers 0 (l0[0, m0)) and 2 (l2[0, m2)) and of layer 1 (l1[0, m1), or all
// its m1 hits when l1 is null), 128 of them at a time in registers: each hit k_first +
// i k_step of l2 against layer 1, each pair found against l0.  They join the warp's
// pending triples (np), which are fitted 32 at a time, or at the end of the station
// when `all` is set: the fits of an event's non-trigger stations share their
// instructions.  A crowded station's are found from its row lists instead.
template <bool EMIT, bool FILTER, class W, class R, class L>
__device__ __forceinline__ void sieve_triples(const Job& j, W& w, uint32_t* pend, int lane, const Cuts& c, float B,
                                              int64_t e, int s, int s1, int s2, const L* l0, int m0, const L* l1,
                                              int m1, const L* l2, int m2, int k_first, int k_step, bool sink,
                                              int nT, bool all, bool crowded, R& rows, int& np) {
    const uint32_t lt = (1u << lane) - 1u;
    const int hi0 = l0[min(lane, max(m0 - 1, 0))];  // what is left of layer 0, its first 32
    const float2 Pi0 = w.P[m0 > 0 ? hi0 : 0];
    float2 Pj[4], Pk = make_float2(0.f, 0.f), Q = Pk;
    int j0 = -128, k = m2 + k_step, hk = 0, hj = 0, i0 = m0;  // next: layer 0 from i0 on for the pair (hj, hk)
    unsigned mine = 0;                               // this lane's rounds with further partners of hk
    bool more = m2 > k_first;
    for (;;) {
        if (__builtin_expect(crowded, 0)) {
            more = uniform(row_search(j, w.P, pend, rows, k_first, k_step, (uint32_t)s << 27, l0, l2, lane, np));
        } else {
#pragma unroll 1
            while (more && np <= 32) {
                if (i0 >= m0) {
                    const unsigned lanes = __ballot_sync(kFull, mine != 0);
                    if (lanes) {  // the next pair
                        const int from = __ffs(lanes) - 1;
                        hj = j0 + 32 * (__ffs(__shfl_sync(kFull, mine, from)) - 1) + from;
                        if (lane == from) mine &= mine - 1;
                        if (hj < m1) {  // (an infinite bound lets the places past the end through)
                            if (FILTER && l1) hj = l1[hj];
                            Q = w.P[s1 + hj];
                            i0 = 0;
                        }
                    } else {
                        k += k_step;
                        if (k >= m2) {  // the next 128 hits of layer 1
                            j0 += 128;
                            if (j0 >= m1) {
                                more = false;
                                continue;
                            }
                            k = k_first;
#pragma unroll
                            for (int r = 0; r < 4; ++r) {
                                const int p = j0 + 32 * r + lane;
                                const int h = min(p, m1 - 1);
                                Pj[r] = w.P[s1 + (FILTER && l1 ? (int)l1[h] : h)];
                                if (p >= m1) Pj[r].x = INFINITY;
                            }
                        }
                        hk = l2[k];
                        Pk = w.P[s2 + hk];
#pragma unroll
                        for (int r = 0; r < 4; ++r) mine |= pair_ok(Pj[r].x, Pj[r].y, Pk.x, Pk.y, B) ? 1u << r : 0u;
                    }
                    continue;
                }
                int hi = hi0;
                float2 Pi = Pi0;
                if (i0 > 0) {
                    hi = l0[min(i0 + lane, m0 - 1)];
                    Pi = w.P[hi];
                }
                const bool cand =
                    (i0 + lane < m0) & pair_ok(Pi.x, Pi.y, Q.x, Q.y, B) & pair_ok(Pi.x, Pi.y, Pk.x, Pk.y, B);
                const unsigned mask = __ballot_sync(kFull, cand);
                const int at = np + __popc(mask & lt);
                if (cand && JPSI_IN(j.ctrl, at < 64))
                    pend[at] = (uint32_t)s << 27 | (uint32_t)hi << 18 | (uint32_t)hj << 9 | (uint32_t)hk;
                np += __popc(mask);
                i0 += 32;
            }
        }
        np = uniform(np);
        np = light_fit<EMIT>(j, w, pend, lane, c, e, sink, nT, np, all && !more ? 0 : 32);
        if (!more) break;
    }
}

// Hits left of layer 2 beyond which a station is crowded: where the row lists cost
// less than trying each of those hits with all of layer 1.  One warp, limits 8, 12,
// 18 and 24: 40 000 events of 50 hits per layer with a 2 cm window 464, 471, 503 and
// 554 us, of 100 hits with 1 cm 441, 444, 466 and 507; the other way about, 60 hits
// with 1 cm (noalloc) 178, 172, 167 and 166, 100 hits with 0.7 cm 341, 325, 330 and
// 332.  A block shares those hits between four warps; limits 12, 24, 48 and 80: 150
// hits with 0.7 cm 223, 219, 221 and 223, with 1 cm 277, 280, 305 and 357; 250 hits with
// 0.7 cm 219, 217, 240 and 292.  Row lists made events of 250 hits per layer with a
// 1 cm window (3 000 events) 387 us, 599 on the block tile and 818 without them.
constexpr int kCrowdedWarp = 12, kCrowdedBlock = 24;

// Stages station s of event e and finds its triples (see above).  Returns 0, 1 for
// a hit with z <= 0 or 2 for one whose pruning bound is not finite.
template <bool EMIT>
__device__ __forceinline__ int light_station(const Job& j, WarpTile& w, int lane, const Cuts& c, int32_t o0, int n0,
                                             int n1, int n2, int64_t e, int s, bool sink, int nT, bool all, int& np) {
    const int most = max(max(n0, n1), n2);
    const Shift3 sh = kStream ? Shift3{uniform(w.sh[3 * s]), uniform(w.sh[3 * s + 1]), uniform(w.sh[3 * s + 2])}
                              : Shift3{0, 0, 0};
    float rmax, smax;
    bool ok, uneven = false;
    if (most <= 64)
        ok = sieve_stage<2>(j, w, lane, o0, n0, n1, n2, sh, rmax, smax);
    else if (most <= 128)
        ok = sieve_stage<4>(j, w, lane, o0, n0, n1, n2, sh, rmax, smax);
    else
        ok = sieve_stage<6>(j, w, lane, o0, n0, n1, n2, sh, rmax, smax);
    StationBounds sb = station_bounds(rmax, smax, j.K);
    if (__builtin_expect(!uniform(ok && sb.B < INFINITY), 0)) {
        const int st = uniform(sieve_classify(j, w.P, lane, o0, n0, n0 + n1, n0 + n1 + n2, sh, w.lay, rmax, smax));
        if (st) return st;
        sb = station_bounds(rmax, smax, j.K);
        uneven = uniform(uneven_bounds(pair_bounds(w.lay, j.K), sb.B));
    }
    int m0, m2;
    if (most <= 64)
        sieve_layers<2>(j, w, lane, n0, n1, n2, sb.inv, m0, m2);
    else if (most <= 128)
        sieve_layers<4>(j, w, lane, n0, n1, n2, sb.inv, m0, m2);
    else
        sieve_layers<6>(j, w, lane, n0, n1, n2, sb.inv, m0, m2);
    static_assert(SmallCfg::LAYER_CAP <= 6 * 32, "rounds of a layer");
    m2 = uniform(m2);
    m0 = uniform(m0);
    using Lists = RowLists<uint8_t, SmallCfg::LAYER_CAP, 1>;
    static_assert(sizeof(Lists) <= sizeof(w.map), "the lists take the maps' memory");
    Lists& rows = *reinterpret_cast<Lists*>(w.map);
    const bool crowded = uniform(m2 > (uneven ? 0 : kCrowdedWarp));
    if (__builtin_expect(crowded, 0))
        row_lists<32>(j, rows, w.P, lane, uneven ? pair_bounds(w.lay, j.K) : PairBounds{sb.B, sb.B, sb.B}, w.left[0],
                      m0, -1, n1, SmallCfg::LAYER_CAP, m2, n0, n0 + n1);
    if (m2 > 0 || (all && np > 0))
        sieve_triples<EMIT, false>(j, w, w.pend, lane, c, sb.B, e, s, n0, n0 + n1, w.left[0], m0,
                                   (const uint8_t*)nullptr, n1, w.left[1], m2, 0, 1, sink, nT, all, crowded, rows, np);
    return 0;
}

__device__ __forceinline__ void push_event(const Job& j, int64_t e, uint8_t cls) {
    j.ev_class[e] = cls;
    if (j.plain) return;  // the one-launch form's block kernel finds the event by its class
    if (cls == kClsMedium) {
        const int gi = atomicAdd(&j.ctrl->n_medium, 1);
        if (JPSI_IN(j.ctrl, gi < j.n_events)) j.mlist[gi] = (int32_t)e;
    } else if (cls == kClsHeavy) {
        const int gi = atomicAdd(&j.ctrl->n_heavy, 1);
        if (JPSI_IN(j.ctrl, gi < j.n_events)) j.hlist[gi] = (int32_t)e;
    } else {
        const int gi = atomicAdd(&j.ctrl->n_generic, 1);
        if (JPSI_IN(j.ctrl, gi < j.n_events)) j.glist[gi] = (int32_t)e;
    }
}

// Loads the event's offsets into the tile and checks its CSR span (non-
// decreasing, first >= 0 and == 0 for event 0, last <= n_hits and == n_hits for
// the last event) and its sizes.  Returns 0 (it fits the warp path), 1 (too
// large) or 2 (malformed), warp-uniform; every processed station of an event
// that fits has at most SmallCfg::HCAP hits.  The layer capacities may be lowered
// at run time (Job::cap_small, cap_medium: a tuning choice, results do not
// depend on it).  medium: it fits the medium tile.
__device__ __forceinline__ int light_offsets(const Job& j, WarpTile& w, int lane, int64_t e, bool& medium) {
    const int S3 = 3 * j.S;
    const int32_t* base = j.off + e * S3;
    const int rounds = S3 < 32 ? 1 : 2;
#pragma unroll 1
    for (int q = 0; q < rounds; ++q)
        if (lane + 32 * q <= S3) {
            w.off[lane + 32 * q] = __ldg(base + lane + 32 * q);
            if (kStream && lane + 32 * q < S3) w.sh[lane + 32 * q] = __ldg(j.shift + e * S3 + lane + 32 * q);
        }
    __syncwarp();
    int code = 0;
    bool med = true;
#pragma unroll 1
    for (int q = 0; q < rounds; ++q) {
        const int l = lane + 32 * q;
        if (l <= S3) {
            const int32_t a = w.off[l];
            if (l == 0 && (a < 0 || (e == 0 && a != 0))) code = 2;
            if (l == S3) {
                if ((int64_t)a > j.n_hits || (e == j.n_events - 1 && (int64_t)a != j.n_hits)) code = 2;
            } else {
                // compared, not subtracted: 2^31 - 1 and -2 differ by 2^31 - 1
                // in 32 bits.  (The sizes are right when no lane says 2.)
                const int s = l / 3;
                if (w.off[l + 1] < a) code = 2;
                const uint32_t d1 = (uint32_t)w.off[l + 1] - (uint32_t)a,
                               d3 = l == 3 * s ? (uint32_t)w.off[l + 3] - (uint32_t)a : 0u;
                if (j.mode == 1 || s == j.trig) {
                    if (d1 > (uint32_t)j.cap_small || d3 > (uint32_t)SmallCfg::HCAP) code = max(code, 1);
                    if (d1 > (uint32_t)j.cap_medium || d3 > (uint32_t)MediumCfg::HCAP) med = false;
                }
            }
        }
    }
    code = uniform(code);
    medium = __all_sync(kFull, med);
    return code;
}

__device__ void light_event_count(const Job& j, WarpTile& w, int lane, const Cuts& c, int64_t e) {
    const int S = j.S;
    bool medium;
    const int code = light_offsets(j, w, lane, e, medium);
    int moved = -1;  // the class of an event that leaves this path (kClsInvalid: malformed)
    if (code != 0) {
        moved = code == 2 ? kClsInvalid : medium && !j.plain ? kClsMedium : kClsHeavy;
    } else {
        const bool chain = j.mode == 1 && S > 1;
        const int nproc = j.mode == 1 ? S : 1;
        int32_t o0 = uniform(w.off[3 * j.trig]);  // (the trigger station comes first)
        // the first station's lines start towards L2 now; each station then
        // prefetches the next (prefetching all of them evicted some lines
        // before use: 17 % more DRAM reads, against 4 % for one ahead)
        if (kStream)
            prefetch_station(j, w.off, w.sh, j.trig, lane);
        else if (!j.host_hits)
            prefetch_hits_l2(j, o0, w.off[3 * j.trig + 3], lane);
        const bool sink = chain || j.distinct;  // the trigger triplets are kept: CHAIN slopes, candidates' hits
        int np = 0, nT = 0;
        if (lane < kMaxStations) {
            w.count[lane] = 0;
            w.partners[lane] = 0;
        }
#pragma unroll 1
        for (int si = 0; si < nproc; ++si) {
            const int s = station_of(si, j.trig);
            o0 = uniform(w.off[3 * s]);
            const int n0 = uniform(w.off[3 * s + 1]) - o0, n1 = uniform(w.off[3 * s + 2]) - o0 - n0,
                      n2 = uniform(w.off[3 * s + 3]) - o0 - n0 - n1;
            if (si + 1 < nproc) prefetch_station(j, w.off, w.sh, station_of(si + 1, j.trig), lane);
            const int st = light_station<false>(j, w, lane, c, o0, n0, n1, n2, e, s, sink, chain ? nT : 0,
                                                (sink && si == 0) || si + 1 == nproc, np);
            if (st != 0) {
                moved = st == 1 ? kClsInvalid : kClsGeneric;
                break;
            }
            if (si == 0) {
                nT = sink ? uniform(w.count[s]) : 0;
                if (nT > SmallCfg::TCAP) {
                    moved = kClsHeavy;
                    break;
                }
            }
            __syncwarp();  // the tile may be staged again
        }
        if (moved < 0) {
            static_assert(SmallCfg::TCAP <= 32, "one flag per lane");
            if (lane < S) j.unit_counts[e * S + lane] = w.count[lane];
            int tc = w.count[j.trig];
            if (chain) {  // the slopes with a partner in every other station
                const unsigned with = __reduce_and_sync(
                    kFull, lane < S && lane != j.trig ? w.partners[lane] : nT < 32 ? (1u << nT) - 1u : ~0u);
                tc = __popc(with);
                w.alive[lane] = with >> lane & 1u;
                __syncwarp();
            }
            if (j.distinct) {  // nT is warp-uniform
                const bool f = nT >= 2 && warp_disjoint_pair(w.Tijk, chain ? w.alive : nullptr, nT, lane);
                if (lane == 0) j.dpair[e] = f;
            }
            if (lane == 0) {
                j.track_counts[e] = tc;
                j.ev_class[e] = kClsLight;
            }
        }
    }
    if (moved >= 0 && lane == 0) {
        if (moved == kClsInvalid) {
            atomicOr(&j.ctrl->status, kStInvalid);
            j.ev_class[e] = kClsInvalid;
        } else {
            push_event(j, e, (uint8_t)moved);
        }
    }
    __syncwarp();  // the tile is free
}

__device__ void light_event_emit(const Job& j, WarpTile& w, int lane, const Cuts& c, int64_t e) {
    if (j.ev_class[e] != kClsLight) return;
    const int S = j.S;
    const int nproc = j.mode == 1 ? S : 1;
    bool any = false, medium;
    for (int si = 0; si < nproc; ++si) any |= j.unit_counts[e * S + station_of(si, j.trig)] != 0;
    if (!any) return;
    light_offsets(j, w, lane, e, medium);
    if (lane < kMaxStations) w.count[lane] = 0;
    int np = 0;
#pragma unroll 1
    for (int si = 0; si < nproc; ++si) {
        const int s = station_of(si, j.trig);
        const int cnt = j.unit_counts[e * S + s];
        if (cnt == 0) continue;
        const int32_t o0 = uniform(w.off[3 * s]);
        const int n0 = uniform(w.off[3 * s + 1]) - o0, n1 = uniform(w.off[3 * s + 2]) - o0 - n0,
                  n2 = uniform(w.off[3 * s + 3]) - o0 - n0 - n1;
        const int st = light_station<true>(j, w, lane, c, o0, n0, n1, n2, e, s, false, 0, true, np);
        if ((st != 0 || w.count[s] != cnt) && lane == 0) atomicOr(&j.ctrl->status, kStEmitMismatch);
        __syncwarp();
    }
}

template <bool EMIT>
__device__ __forceinline__ void light_event(const Job& j, WarpTile& w, int lane, const Cuts& c, int64_t e) {
    if (EMIT)
        light_event_emit(j, w, lane, c, e);
    else
        light_event_count(j, w, lane, c, e);
}

// The warp path: every event of the batch (statically one warp per event, or
// persistent warps grabbing `grab` events at a time).
//   Bound by instruction issue (0.75 of the slots, ALU pipe the busiest) and, in
// the loads of a station, by memory: 4 045 warp instructions per event of the
// 10^6-event workload, where sorting every hit into cells and walking windows of
// them took 10 200.  10^6 events: 10.41 -> 4.30 ms (3.37 TB/s of hits, 0.50 of
// the measured copy rate); the events of a 55 000-event log-normal timeslice that
// fit: 0.394 -> 0.190 ms; 80 000 events in PAPER mode: 0.212 -> 0.102 ms.
//   72 registers (28 warps per SM) were measured before the row lists: 4.73 ms,
// against 4.86 with 64 (32 warps, a few spills) and 80 (24 warps) and 5.40 with 56.
template <bool EMIT>
__global__ void __maxnreg__(72) k_light(const __grid_constant__ Job j) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    chain_wait();
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    WarpTile& w = reinterpret_cast<WarpTile*>(smem_raw)[wi];
    const Cuts c{j.cx, j.cy, j.K};
    // one call of light_event for both forms (the event code is inlined once)
    unsigned long long* ctr = &j.ctrl->work[EMIT ? 4 : 0];
    const int n_ev = (int)j.ev_count;  // events fit 31 bits (3 S + 1 offsets each)
    const int grab = j.persistent ? j.grab : 1;
    for (bool more = true; more; more = j.persistent) {
        int k0 = (int)(blockIdx.x * (blockDim.x >> 5)) + wi;
        if (j.persistent) {
            k0 = 0;  // (the counter stays below n_ev + the grid's warps * grab)
            if (lane == 0) k0 = (int)atomicAdd(ctr, (unsigned long long)grab);
        }
        k0 = uniform(k0);  // (the other lanes' 0 is no larger)
        if (k0 >= n_ev) break;
        const int k1 = min(k0 + grab, n_ev);
#pragma unroll 1
        for (int k = k0; k < k1; ++k) light_event<EMIT>(j, w, lane, c, j.ev_begin + k);
    }
    chain_next();
}

// ------------------------------------------------------ block-tile path

// Stages station s of the event whose offsets are in sm.off.  Returns 0, 1
// (z <= 0) or 2 (not prunable).
template <class B>
__device__ int stage_station_block(const Job& j, BlockSmem<B>& sm, int s) {
    int pbase = 0;
    for (int l = 0; l < 3; ++l) {
        const int32_t b = sm.off[3 * s + l], e = sm.off[3 * s + l + 1];
        int nl = 0;
        const int st = stage_layer_block(j, sm, l, b + (kStream ? sm.sh[3 * s + l] : 0), e - b, pbase, nl);
        if (st) return st;
        pbase += nl;
    }
    return 0;
}

template <class B>
__device__ __forceinline__ void load_event_offsets(const Job& j, BlockSmem<B>& sm, int64_t e) {
    const int S3 = 3 * j.S;
    for (int i = threadIdx.x; i <= S3; i += B::THREADS) {
        sm.off[i] = j.off[e * S3 + i];
        if (kStream && i < S3) sm.sh[i] = j.shift[e * S3 + i];
    }
    __syncthreads();
}

// Job::hT[gi].y of a block-tile event: >= 0, its stations run on separate
// blocks with that many trigger slopes in the pool from hT[gi].x on; or
constexpr int kHTOwned = -1;  // its first block does (did) all of it
constexpr int kHTMoved = -2;  // it went to the unpruned kernel

// Hands an event from the block-tile path to the unpruned kernel, once (the
// per-station blocks of one event may all find a reason).
__device__ __forceinline__ void heavy_to_generic(const Job& j, int gi, int64_t e) {
    if (atomicExch(&j.hT[gi].y, kHTMoved) != kHTMoved) push_event(j, e, kClsGeneric);
}

// One station of a block-tile event: staging, the triplet search of the
// station (Sec. 3.2 steps 1-2) and, in CHAIN mode, the trigger slopes in
// T[0, nT) that find no compatible triplet here lose their alive flag.
// Counting pass: writes the unit count (also returned in cnt); returns false
// when the event left the path (then nothing else may be done for it).
// Emit pass: writes rows.  Block-uniform arguments; all threads call it.
// Who hands an event on when a station cannot be pruned: gi >= 0 is the
// event's block-tile list entry (its state in Job::hT);
constexpr int kGiPlain = -1;  // the one-launch form: the same block goes on unpruned

// Pulls the hit lines of station s of the event in sm.off into L2 (block
// version of prefetch_hits_l2; addresses stay inside [o[0] & ~31, o[3])).
template <class B>
__device__ __forceinline__ void prefetch_station_block(const Job& j, const BlockSmem<B>& sm, int s) {
    if (j.host_hits) return;
    for (int l = 0; l < (kStream ? 3 : 1); ++l) {
        const int32_t g = kStream ? sm.sh[3 * s + l] : 0;
        const int32_t h0 = sm.off[3 * s + l] + g, h1 = sm.off[3 * s + (kStream ? l + 1 : 3)] + g;
        for (int32_t a = (h0 & ~31) + 32 * (int)threadIdx.x; a < h1; a += 32 * B::THREADS) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(j.x + a));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(j.y + a));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(j.z + a));
        }
    }
}

// s_next: the station this block stages next (-1: none), whose lines start
// towards L2 now; the station's own lines too, so that its second and third
// layers arrive while the first is staged.
template <bool EMIT, class B>
__device__ bool heavy_unit(const Job& j, BlockSmem<B>& sm, const Cuts& c, int gi, int64_t e, int s, TSink& ts,
                           const float2* T, uint8_t* alive, int nT, int& cnt, int s_next = -1,
                           const float2* Tt = nullptr) {
    using TV = TileView<B::NX, B::NY>;
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int64_t u = e * j.S + s;
    const int cnt_expected = EMIT ? j.unit_counts[u] : 0;
    prefetch_station_block(j, sm, s);
    if (s_next >= 0) prefetch_station_block(j, sm, s_next);
    const int st = stage_station_block(j, sm, s);
    if (st != 0) {
        if (tid == 0) {
            if (EMIT) {
                atomicOr(&j.ctrl->status, kStEmitMismatch);
            } else if (st == 1) {
                atomicOr(&j.ctrl->status, kStInvalid);
                j.ev_class[e] = kClsInvalid;
            } else if (gi == kGiPlain) {
                j.ev_class[e] = kClsGeneric;
            } else {
                heavy_to_generic(j, gi, e);
            }
        }
        return false;
    }
    if (tid == 0) {
        sm.s_rank = 0;
        sm.s_next = 0;
    }
    __syncthreads();
    int32_t* rows = EMIT ? j.triplets + 3 * j.trip_off[u] : nullptr;
    // the station's trigger-slope searches run on the warps beside its
    // enumeration rounds (both only read the staged tile)
    const bool empty = sm.meta[0].nlive == 0 || sm.meta[1].nlive == 0 || sm.meta[2].nlive == 0;
    const RoadItems rd{T, alive, EMIT || empty ? 0 : nT, Tt};
    enum_station<EMIT>(j, TV{sm.P, sm.idx, sm.bst, sm.meta}, sm.queue[wp],
                       Pending{sm.pend_pair[wp], sm.pend_k[wp], 0}, lane, c, ts, rows,
                       cnt_expected, u, &sm.s_rank, B::CLS, &sm.s_next, &rd);
    __syncthreads();
    cnt = sm.s_rank;
    if (EMIT) {
        if (tid == 0 && cnt != cnt_expected) atomicOr(&j.ctrl->status, kStEmitMismatch);
        return true;
    }
    if (tid == 0) j.unit_counts[u] = cnt;
    if (empty)  // no triplet at all in this station: no slope finds one
        for (int ti = tid; ti < nT; ti += B::THREADS) alive[ti] = 0;
    return true;
}

// Counting pass of one block-tile event (list index gi).  The trigger
// station comes first; in CHAIN mode its passing triplets' slopes go to the
// block's own list, and then, when the trigger-slope pool has room, to the
// pool: the other stations are then left to k_heavy_units (one block per
// station) and k_heavy_final.  Otherwise this block does them itself.  The
// event may move on to the unpruned kernel (too large, extreme coordinates
// or too many trigger triplets for the block's list).
__device__ void heavy_event(const Job& j, HeavySmem& sm, const Cuts& c, int gi, int64_t e) {
    const int tid = threadIdx.x, lane = tid & 31;
    const int S = j.S;
    const bool chain = j.mode == 1 && S > 1;
    const int nproc = j.mode == 1 ? S : 1;
    if (tid == 0) {
        sm.s_nT = 0;
        j.hT[gi] = make_int2(0, kHTOwned);
    }
    load_event_offsets(j, sm, e);
    bool fits = true;
    for (int si = 0; si < nproc; ++si) {
        const int32_t* o = sm.off + 3 * station_of(si, j.trig);
        if (o[1] - o[0] > kHLayerCap || o[2] - o[1] > kHLayerCap || o[3] - o[2] > kHLayerCap || o[3] - o[0] > kHHCap)
            fits = false;
    }
    if (!fits) {
        if (tid == 0) heavy_to_generic(j, gi, e);
        return;
    }
    float2* T = j.tlist + (int64_t)blockIdx.x * j.tlist_cap;
    uint8_t* alive = j.talive + (int64_t)blockIdx.x * j.tlist_cap;
    unsigned long long* ijk = j.distinct ? j.tlist_ijk + (int64_t)blockIdx.x * j.tlist_cap : nullptr;
    // free-streaming windows: the slopes' times in the same per-block storage
    float2* tt = kStream ? reinterpret_cast<float2*>(j.tlist_ijk + (int64_t)blockIdx.x * j.tlist_cap) : nullptr;
    int trig_count = 0, nT = 0;
    for (int si = 0; si < nproc; ++si) {
        const int s = station_of(si, j.trig);
        TSink ts{(chain || j.distinct) && si == 0, T, j.tlist_cap, &sm.s_nT};
        ts.ijk = ijk;
        ts.tt = tt;
        int cnt = 0;
        const int sn = si + 1 < nproc ? station_of(si + 1, j.trig) : -1;
        if (!heavy_unit<false>(j, sm, c, gi, e, s, ts, T, alive, si == 0 ? 0 : nT, cnt, sn, tt)) return;
        if (si > 0) {
            __syncthreads();
            continue;
        }
        trig_count = cnt;
        nT = sm.s_nT;
        if (nT > j.tlist_cap) {
            if (tid == 0) heavy_to_generic(j, gi, e);
            return;
        }
        if (!chain) {
            if (j.distinct) {  // PAPER: every passing trigger triplet is a candidate
                const bool f = nT >= 2 && block_disjoint_pair<kHThreads>(ijk, nullptr, nT, &sm.s_hx);
                if (tid == 0) j.dpair[e] = f;
            }
            break;
        }
        if (tid == 0) sm.s_pool = nT > 0 ? atomicAdd(&j.ctrl->tpool_n, (unsigned long long)nT) : 0ull;
        __syncthreads();
        const unsigned long long pb = sm.s_pool;
        if (pb + (unsigned long long)nT <= (unsigned long long)j.tpool_cap) {
            for (int i = tid; i < nT; i += kHThreads) {
                j.tpool[pb + i] = T[i];
                j.tpool_alive[pb + i] = 1;
                if (ijk) j.tpool_ijk[pb + i] = ijk[i];
                if (tt) reinterpret_cast<float2*>(j.tpool_ijk)[pb + i] = tt[i];
            }
            if (tid == 0) j.hT[gi] = make_int2((int)pb, nT);
            return;
        }
        for (int i = tid; i < nT; i += kHThreads) alive[i] = 1;
        __syncthreads();
    }
    int tc = trig_count;
    if (chain) {
        if (tid == 0) sm.s_cand = 0;
        __syncthreads();
        int a = 0;
        for (int ti = tid; ti < nT; ti += kHThreads) a += alive[ti];
        a = __reduce_add_sync(kFull, a);
        if (lane == 0 && a) atomicAdd(&sm.s_cand, a);
        __syncthreads();
        tc = sm.s_cand;
        if (j.distinct) {
            const bool f = nT >= 2 && block_disjoint_pair<kHThreads>(ijk, alive, nT, &sm.s_hx);
            if (tid == 0) j.dpair[e] = f;
        }
    }
    if (tid == 0) {
        if (j.mode == 0)
            for (int s = 0; s < S; ++s)
                if (s != j.trig) j.unit_counts[e * S + s] = 0;
        j.track_counts[e] = tc;
    }
}

// Medium path: 4-warp blocks take the events of the medium list, one at a time, and
// run every station of their event with the sieve of the warp path, shared by the
// warps: the trigger station first (in CHAIN mode its passing triplets'
// slopes, at most kTCap, stay in shared memory), then the others, whose passing
// triplets are held against those slopes.  An event with more trigger slopes goes on
// to the block tile; one with extreme coordinates to the unpruned kernel.
//   Bound by instruction issue and the barriers between the maps.  The events of
// a 55 000-event log-normal timeslice: 379 us with cell-sorted tiles, 260 with
// the sieve; of 100 000 free-streaming collisions: 1.23 -> 1.02 ms.  Four warps and
// eight blocks per SM (64 registers) against two warps and 13 blocks: the same
// on the timeslice, 4 % slower on the collisions, but an event takes little more than
// half as long: medium and block tiles of 1 000 collisions 161 -> 131 us, of 10 000
// log-normal events 363 -> 336 us.

__device__ __forceinline__ SieveBit medium_bit(float2 s, float inv) {
    const int cx = sieve_cell(s.x, inv), cy = sieve_cell(s.y, inv);
    return {((cy & (kMapRows - 1)) << 2) + ((cx >> 5) & 3), __funnelshift_l(0u, 1u, cx)};
}

// sieve_dilate for the block: a ring of 128 columns; each thread has RT consecutive
// rows.  With MEET, `other` is cleared behind it.
template <bool MEET>
__device__ __forceinline__ void medium_dilate(uint32_t* map, uint32_t* other) {
    constexpr int RT = kMapRows / MediumTile::THREADS;
    const int t = RT * threadIdx.x;
    __syncthreads();
    uint4* m4 = reinterpret_cast<uint4*>(map);
    uint4 q[RT + 2];
#pragma unroll
    for (int r = 0; r < RT + 2; ++r) q[r] = m4[(t + r + kMapRows - 1) & (kMapRows - 1)];
    uint32_t d[RT][4];
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        const uint4 a = q[r], b = q[r + 1], c = q[r + 2];
        const uint32_t v[4] = {a.x | b.x | c.x, a.y | b.y | c.y, a.z | b.z | c.z, a.w | b.w | c.w};
        uint4 o = make_uint4(~0u, ~0u, ~0u, ~0u);
        if (MEET) {
            uint4* o4 = reinterpret_cast<uint4*>(other);
            o = o4[t + r];
            o4[t + r] = make_uint4(0u, 0u, 0u, 0u);
        }
        const uint32_t ov[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
            d[r][i] = (v[i] | __funnelshift_l(v[(i + 3) & 3], v[i], 1) | __funnelshift_r(v[i], v[(i + 1) & 3], 1)) & ov[i];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RT; ++r) m4[t + r] = make_uint4(d[r][0], d[r][1], d[r][2], d[r][3]);
    __syncthreads();
}

// The hits of a layer (places [p0, p0 + n)) whose cells are set in `map`: their
// layer-local indices to `left` (any order), their cells to `mark` (if given).
__device__ __forceinline__ void medium_pass(const Job& j, MediumTile& w, float inv, int p0, int n, const uint32_t* map,
                                            uint32_t* mark, uint16_t* left, int* n_left) {
    constexpr int T = MediumTile::THREADS, R = MediumCfg::LAYER_CAP / T;
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t lt = (1u << lane) - 1u;
    unsigned bits = 0;
    int m = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (T * r >= n) break;  // block-uniform
        const SieveBit b = medium_bit(w.P[p0 + T * r + tid], inv);
        const bool in = (T * r + tid < n) & ((map[b.word] & b.bit) != 0);
        if (mark && in) atomicOr(&mark[b.word], b.bit);
        bits |= in ? 1u << r : 0u;
        m += __popc(__ballot_sync(kFull, in));
    }
    int at = 0;
    if (lane == 0 && m) at = atomicAdd(n_left, m);
    at = __shfl_sync(kFull, at, 0);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (T * r >= n) break;
        const unsigned mask = __ballot_sync(kFull, bits >> r & 1u);
        const int i = at + __popc(mask & lt);
        if ((bits >> r & 1u) && JPSI_IN(j.ctrl, i < MediumCfg::LAYER_CAP)) left[i] = (uint16_t)(T * r + tid);
        at += __popc(mask);
    }
}

// Stages station s of the event in w.off and finds its triples (see
// sieve_layers; a third map leaves fewer hits of layer 1 when layer 2 has more
// than kFilterMin).  Returns 0, 1 for a hit with z <= 0 or 2 for one whose pruning
// bound is not finite; block-uniform, all threads call it.
constexpr int kFilterMin = 8;
template <bool EMIT>
__device__ __forceinline__ int medium_station(const Job& j, MediumTile& w, const Cuts& c, int64_t e, int s, bool sink,
                                              int nT, bool all, int& np) {
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int32_t o0 = uniform(w.off[3 * s]);
    const int n0 = uniform(w.off[3 * s + 1]) - o0, n1 = uniform(w.off[3 * s + 2]) - o0 - n0,
              n2 = uniform(w.off[3 * s + 3]) - o0 - n0 - n1, n = n0 + n1 + n2;
    const int s1 = n0, s2 = n0 + n1;
    constexpr int T = MediumTile::THREADS;
    const Shift3 sh = shift3(w.sh, s);
    float smax = 0.0f, rmax = 0.0f, rmin = INFINITY;
    StationBounds sb;
    for (int p0 = 0; p0 < n; p0 += 4 * T) {
        float x[4], y[4], z[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (p0 + T * q < n) {  // block-uniform; threads past the end read the last hit again
                const int p = min(p0 + T * q + tid, n - 1);
                const int32_t h = o0 + p + sh.at(p, s1, s2);
                x[q] = __ldg(j.x + h);
                y[q] = __ldg(j.y + h);
                z[q] = __ldg(j.z + h);
            }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (p0 + T * q < n) {
                const float iz = rcp_approx(z[q]);
                const float2 v = make_float2(__fmul_rn(x[q], iz), __fmul_rn(y[q], iz));
                smax = max3_abs_nan(smax, v.x, v.y);
                rmax = max3_abs_nan(rmax, iz, 0.0f);
                rmin = fminf(rmin, iz);
                if (p0 + T * q + tid < n) w.P[p0 + T * q + tid] = v;
            }
    }
    auto reduce = [&]() {  // the block's maxima, minimum, and what they say of the hits
        const int si = __reduce_max_sync(kFull, __float_as_int(smax)), ri = __reduce_max_sync(kFull, __float_as_int(rmax)),
                  ni = __reduce_min_sync(kFull, __float_as_int(rmin));
        if (lane == 0) {
            w.red[wp][0] = si;
            w.red[wp][1] = ri;
            w.red[wp][2] = ni;
        }
        __syncthreads();
        const int wl = lane & (MediumTile::WARPS - 1);
        const int bs = __reduce_max_sync(kFull, w.red[wl][0]), br = __reduce_max_sync(kFull, w.red[wl][1]),
                  bn = __reduce_min_sync(kFull, w.red[wl][2]);
        smax = __int_as_float(bs);
        rmax = __int_as_float(br);
        sb = station_bounds(rmax, smax, j.K);
        return bs < 0x7f800000 && br < 0x7e800000 && bn > 0x00800000 && sb.B < INFINITY &&
               even_hits(br, bn, rmax, smax, j.K);
    };
    uint32_t *ma = w.map[0], *mb = w.map[1];
#pragma unroll
    for (int q = 0; q < 2 * kMapRows / T; ++q) reinterpret_cast<uint4*>(w.map)[T * q + tid] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < 3) w.n_left[tid] = 0;
    bool uneven = false;
    if (!uniform(reduce())) {  // odd coordinates or uneven hits: classify every hit exactly (see sieve_classify)
        bool zbad = false, wild = false;
        smax = rmax = 0.0f;
        if (tid < 3) w.lay[tid] = LayerMax{0.0f, 0.0f};
        __syncthreads();
#pragma unroll 1
        for (int l = 0; l < 3; ++l) {
            float r = 0.0f, sl = 0.0f;
            const int end = l == 0 ? s1 : l == 1 ? s2 : n;
#pragma unroll 1
            for (int p = (l == 0 ? 0 : l == 1 ? s1 : s2) + tid; p < end; p += T) {
                const int32_t g = o0 + p + (kStream ? sh.of(l) : 0);
                const HitPrep h = hit_prep(__ldg(j.x + g), __ldg(j.y + g), __ldg(j.z + g), j.K);
                zbad |= h.zbad;
                wild |= h.wild;
                const bool live = h.live & !h.wild;
                w.P[p] = live ? make_float2(h.sx, h.sy) : make_float2(INFINITY, INFINITY);
                if (live) {
                    sl = fmaxf(sl, fmaxf(fabsf(h.sx), fabsf(h.sy)));
                    r = fmaxf(r, h.r);
                }
            }
            smax = fmaxf(smax, sl);
            rmax = fmaxf(rmax, r);
            // (values >= 0 order like their bit patterns)
            const int ri = __reduce_max_sync(kFull, __float_as_int(r)), si = __reduce_max_sync(kFull, __float_as_int(sl));
            if (lane == 0) {
                atomicMax(reinterpret_cast<int*>(&w.lay[l].r), ri);
                atomicMax(reinterpret_cast<int*>(&w.lay[l].s), si);
            }
        }
        if (uniform(__syncthreads_or(zbad))) return 1;
        if (uniform(__syncthreads_or(wild))) return 2;
        reduce();
        uneven = uniform(uneven_bounds(pair_bounds(w.lay, j.K), sb.B));
    }
    for (int p0 = 0; p0 < n1; p0 += T) {
        const SieveBit b = medium_bit(w.P[s1 + p0 + tid], sb.inv);
        if (p0 + tid < n1) atomicOr(&ma[b.word], b.bit);
    }
    medium_dilate<false>(ma, nullptr);
    medium_pass(j, w, sb.inv, 0, n0, ma, mb, w.left[0], &w.n_left[0]);
    medium_dilate<true>(mb, ma);
    medium_pass(j, w, sb.inv, s2, n2, mb, ma, w.left[2], &w.n_left[2]);
    __syncthreads();
    const int m0 = uniform(w.n_left[0]), m2 = uniform(w.n_left[2]);
    int m1 = n1;
    const uint16_t* l1 = nullptr;
    if (m2 > kFilterMin) {
        medium_dilate<true>(ma, mb);
        medium_pass(j, w, sb.inv, s1, n1, ma, nullptr, w.left[1], &w.n_left[1]);
        __syncthreads();
        m1 = uniform(w.n_left[1]);
        l1 = w.left[1];
    }
    using Lists = RowLists<uint16_t, MediumCfg::LAYER_CAP, MediumTile::WARPS>;
    static_assert(sizeof(Lists) <= sizeof(w.map), "the lists take the maps' memory");
    Lists& rows = *reinterpret_cast<Lists*>(w.map);
    const bool crowded = m2 > (uneven ? 0 : kCrowdedBlock);
    if (crowded)
        row_lists<T>(j, rows, w.P, tid, uneven ? pair_bounds(w.lay, j.K) : PairBounds{sb.B, sb.B, sb.B}, w.left[0], m0,
                     l1 ? MediumCfg::LAYER_CAP : -1, m1, 2 * MediumCfg::LAYER_CAP, m2, s1, s2);
    sieve_triples<EMIT, true>(j, w, w.pend[wp], lane, c, sb.B, e, s, s1, s2, w.left[0], m0, l1, m1, w.left[2], m2, wp,
                              MediumTile::WARPS, sink, nT, all, crowded, rows, np);
    return 0;
}

template <bool EMIT>
__device__ void medium_event(const Job& j, MediumTile& w, const Cuts& c, int64_t e) {
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int S = j.S;
    const bool chain = j.mode == 1 && S > 1;
    const int nproc = j.mode == 1 ? S : 1;
    for (int i = tid; i <= 3 * S; i += MediumTile::THREADS) {
        w.off[i] = __ldg(j.off + e * 3 * S + i);
        if (kStream && i < 3 * S) w.sh[i] = __ldg(j.shift + e * 3 * S + i);
    }
    if (tid < kMaxStations) {
        w.count[tid] = 0;
        w.partners[tid] = 0;
    }
    __syncthreads();
    int np = 0, nT = 0;
    const bool sink = !EMIT && (chain || j.distinct);
#pragma unroll 1
    for (int si = 0; si < nproc; ++si) {
        const int s = station_of(si, j.trig);
        const int cnt = EMIT ? uniform(j.unit_counts[e * S + s]) : 0;
        if (EMIT && cnt == 0) continue;
        if (wp == 0) {  // the next station's lines start towards L2
            if (si == 0) prefetch_station(j, w.off, w.sh, s, lane);
            if (si + 1 < nproc) prefetch_station(j, w.off, w.sh, station_of(si + 1, j.trig), lane);
        }
        const int st = medium_station<EMIT>(j, w, c, e, s, sink, chain ? nT : 0,
                                            EMIT || (sink && si == 0) || si + 1 == nproc, np);
        if (EMIT) {
            __syncthreads();
            if ((st != 0 || w.count[s] != cnt) && tid == 0) atomicOr(&j.ctrl->status, kStEmitMismatch);
            continue;
        }
        if (st != 0) {
            if (tid == 0) {
                if (st == 1) {
                    atomicOr(&j.ctrl->status, kStInvalid);
                    j.ev_class[e] = kClsInvalid;
                } else {
                    push_event(j, e, kClsGeneric);
                }
            }
            return;
        }
        if (si == 0) {
            __syncthreads();
            nT = sink ? uniform(w.count[s]) : 0;
            if (nT > kTCap) {  // more trigger slopes than this path keeps
                if (tid == 0) push_event(j, e, kClsHeavy);
                return;
            }
        }
        __syncthreads();  // the tile may be staged again
    }
    if (EMIT) return;
    static_assert(kTCap <= MediumTile::THREADS, "one flag per thread");
    if (tid < S) j.unit_counts[e * S + tid] = w.count[tid];
    int tc = w.count[j.trig];
    if (chain) {  // the slopes with a partner in every other station
        bool with = tid < nT;
        for (int s = 0; s < S; ++s) with = with && (s == j.trig || (w.partners[s] >> tid & 1ull));
        if (tid < MediumTile::TCAP) w.alive[tid] = with;
        tc = __syncthreads_count(with);
    }
    if (j.distinct) {
        const bool f =
            nT >= 2 && block_disjoint_pair<MediumTile::THREADS>(w.Tijk, chain ? w.alive : nullptr, nT, &w.s_flag);
        if (tid == 0) j.dpair[e] = f;
    }
    if (tid == 0) j.track_counts[e] = tc;
}

template <bool EMIT>
__global__ void __launch_bounds__(MediumTile::THREADS, MediumTile::BLOCKS) k_medium(const __grid_constant__ Job j) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    chain_wait();
    MediumTile& w = *reinterpret_cast<MediumTile*>(smem_raw);
    const Cuts c{j.cx, j.cy, j.K};
    const int n_med = *(volatile int32_t*)&j.ctrl->n_medium, m0 = *(volatile int32_t*)&j.ctrl->m_begin;
    unsigned long long* ctr = &j.ctrl->work[EMIT ? 5 : 1];
    for (;;) {
        if (threadIdx.x == 0) w.s_gi = m0 + (int)atomicAdd(ctr, 1ull);
        __syncthreads();
        const int gi = uniform(w.s_gi);
        __syncthreads();
        if (gi >= n_med) break;
        const int64_t e = uniform(j.mlist[gi]);
        if (!EMIT || uniform(j.ev_class[e]) == kClsMedium) medium_event<EMIT>(j, w, c, e);
        __syncthreads();
    }
    chain_next();
}

// Orders the block-tile list by decreasing event size (hits, in kSortBins
// classes), so the persistent blocks take the largest events first and the
// smaller ones fill in behind them.  One block: a counting sort over the classes
// (three barriers, where a bitonic sort of the same keys took 51 us for the 1 700
// block-tile events of a 55 000-event log-normal timeslice, this takes 9);
// lists longer than kSortCap keep their order (they have enough events to
// balance).
constexpr int kSortCap = 8192, kSortBins = 256;
__global__ void __launch_bounds__(1024) k_sort_heavy(const __grid_constant__ Job j) {
    __shared__ int32_t ev[kSortCap];
    __shared__ uint8_t cls[kSortCap];
    __shared__ int start[kSortBins];
    __shared__ int s_max;
    chain_next();
    chain_wait();
    const int h0 = *(volatile int32_t*)&j.ctrl->h_begin;
    const int n = *(volatile int32_t*)&j.ctrl->n_heavy - h0;
    int32_t* list = j.hlist + h0;
    if (n < 2 || n > kSortCap) return;
    const int64_t S3 = 3 * j.S;
    constexpr int R = kSortCap / 1024;
    int hits[R];
    int most = 0;
    if (threadIdx.x < kSortBins) start[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_max = 1;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = threadIdx.x + 1024 * r;
        hits[r] = 0;
        if (i < n) {
            const int32_t e = list[i];
            ev[i] = e;
            hits[r] = max(j.off[(e + 1) * S3] - j.off[e * S3], 0);
            most = max(most, hits[r]);
        }
    }
    most = __reduce_max_sync(kFull, most);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_max, most);
    __syncthreads();
    const float scale = (float)kSortBins / (float)s_max;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = threadIdx.x + 1024 * r;
        if (i < n) {
            const int b = kSortBins - 1 - min((int)((float)hits[r] * scale), kSortBins - 1);  // class 0: the largest
            cls[i] = (uint8_t)b;
            atomicAdd(&start[b], 1);
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {  // exclusive scan of the class sizes, eight consecutive ones per lane
        constexpr int Q = kSortBins / 32;
        int c[Q], sum = 0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            c[q] = start[Q * threadIdx.x + q];
            sum += c[q];
        }
        int run = warp_incl_scan(sum, threadIdx.x) - sum;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            start[Q * threadIdx.x + q] = run;
            run += c[q];
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += 1024) {
        const int at = atomicAdd(&start[cls[i]], 1);
        if (JPSI_IN(j.ctrl, at < n)) list[at] = ev[i];
    }
}

// Counting pass: persistent blocks take block-tile events from the list.
__global__ void __launch_bounds__(kHThreads, 3) k_heavy(const __grid_constant__ Job j) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    chain_wait();
    HeavySmem& sm = *reinterpret_cast<HeavySmem*>(smem_raw);
    const Cuts c{j.cx, j.cy, j.K};
    const int n_heavy = *(volatile int32_t*)&j.ctrl->n_heavy, h0 = *(volatile int32_t*)&j.ctrl->h_begin;
    for (;;) {
        if (threadIdx.x == 0) sm.s_gi = h0 + (int)atomicAdd(&j.ctrl->work[2], 1ull);
        __syncthreads();
        const int gi = sm.s_gi;
        __syncthreads();
        if (gi >= n_heavy) break;
        heavy_event(j, sm, c, gi, j.hlist[gi]);
        __syncthreads();
    }
    chain_next();
}

// One block per (event, station) unit of the block-tile path.  Counting pass
// (CHAIN): the non-trigger stations of events whose trigger slopes went to
// the pool.  Emit pass: every processed station with triplets.
template <bool EMIT>
__global__ void __launch_bounds__(kHThreads, 3) k_heavy_units(const __grid_constant__ Job j) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    chain_wait();
    HeavySmem& sm = *reinterpret_cast<HeavySmem*>(smem_raw);
    const int S = j.S;
    if (!EMIT && (j.mode != 1 || S < 2)) return;
    const int per = EMIT ? (j.mode == 1 ? S : 1) : S - 1;  // units per event
    const Cuts c{j.cx, j.cy, j.K};
    const int h0 = *(volatile int32_t*)&j.ctrl->h_begin;
    const long long n_items = (long long)(*(volatile int32_t*)&j.ctrl->n_heavy - h0) * per;
    for (;;) {
        // thread 0 takes an item and decides (the state it reads may change
        // under other blocks; the block must act on one reading)
        if (threadIdx.x == 0) {
            long long k = (long long)atomicAdd(&j.ctrl->work[EMIT ? 6 : 8], 1ull);
            int hx = 0, hy = 0;
            if (k < n_items) {
                const int gi = h0 + (int)(k / per);
                const int64_t e = j.hlist[gi];
                const int s = station_of((int)(k % per) + (EMIT ? 0 : 1), j.trig);
                bool skip = j.ev_class[e] != kClsHeavy;
                if (EMIT) {
                    skip |= j.unit_counts[e * S + s] == 0;
                } else {
                    const int2 h = j.hT[gi];
                    hx = h.x;
                    hy = h.y;
                    skip |= hy < 0;  // finished by its first block, or moved on
                }
                if (skip) k = -1;
            }
            sm.s_item = k;
            sm.s_hx = hx;
            sm.s_hy = hy;
        }
        __syncthreads();
        const long long k = sm.s_item;
        const int hx = sm.s_hx, hy = sm.s_hy;
        __syncthreads();
        if (k >= n_items) break;
        if (k < 0) continue;
        const int gi = h0 + (int)(k / per);
        const int64_t e = j.hlist[gi];
        const int s = station_of((int)(k % per) + (EMIT ? 0 : 1), j.trig);
        load_event_offsets(j, sm, e);
        TSink ts{false, nullptr, 0, nullptr};
        int cnt = 0;
        heavy_unit<EMIT>(j, sm, c, gi, e, s, ts, j.tpool + hx, j.tpool_alive + hx, hy, cnt, -1,
                         kStream ? reinterpret_cast<const float2*>(j.tpool_ijk) + hx : nullptr);
        __syncthreads();
    }
    chain_next();
}

// CHAIN track counts of the events whose stations ran on separate blocks:
// the trigger slopes still alive after every station (one warp per event).
__global__ void k_heavy_final(const __grid_constant__ Job j) {
    chain_next();
    chain_wait();
    if (j.mode != 1 || j.S < 2) return;
    const int n_heavy = *(volatile int32_t*)&j.ctrl->n_heavy, h0 = *(volatile int32_t*)&j.ctrl->h_begin;
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    for (int gi = h0 + ((blockIdx.x * blockDim.x + threadIdx.x) >> 5); gi < n_heavy; gi += nw) {
        const int2 h = j.hT[gi];
        const int64_t e = j.hlist[gi];
        if (h.y < 0 || j.ev_class[e] != kClsHeavy) continue;
        int a = 0;
        for (int t = lane; t < h.y; t += 32) a += j.tpool_alive[h.x + t];
        a = __reduce_add_sync(kFull, a);
        if (lane == 0) j.track_counts[e] = a;
        if (j.distinct) {
            const bool f = a >= 2 && warp_disjoint_pair(j.tpool_ijk + h.x, j.tpool_alive + h.x, h.y, lane);
            if (lane == 0) j.dpair[e] = f;
        }
    }
}

// --------------------------------------------------- unpruned block path

struct GHit {
    float x, y, z;
    HitPrep p;
};

__device__ __forceinline__ GHit ghit(const Job& j, int64_t h) {
    GHit g;
    g.x = __ldg(j.x + h);
    g.y = __ldg(j.y + h);
    g.z = __ldg(j.z + h);
    g.p = hit_prep(g.x, g.y, g.z, j.K);
    return g;
}

// Brute-force P2 search over every hit of every other station.
__device__ bool road_global(const Job& j, const int32_t* soff, const int32_t* sh, const Cuts& c, float mx, float my,
                            float2 Tt) {
    for (int s = 0; s < j.S; ++s) {
        if (s == j.trig) continue;
        const int32_t* o = soff + 3 * s;
        const Shift3 g = shift3(sh, s);
        bool found = false;
        for (int32_t h0 = o[0] + g.a; h0 < o[1] + g.a && !found; ++h0) {
            const float x0 = __ldg(j.x + h0), y0 = __ldg(j.y + h0), z0 = __ldg(j.z + h0);
            if (!tube_pass(x0, y0, z0, mx, my, c)) continue;
            for (int32_t h1 = o[1] + g.b; h1 < o[2] + g.b && !found; ++h1) {
                const float x1 = __ldg(j.x + h1), y1 = __ldg(j.y + h1), z1 = __ldg(j.z + h1);
                if (!tube_pass(x1, y1, z1, mx, my, c)) continue;
                for (int32_t h2 = o[2] + g.c; h2 < o[3] + g.c && !found; ++h2) {
                    const float xs[3] = {x0, x1, __ldg(j.x + h2)};
                    const float ys[3] = {y0, y1, __ldg(j.y + h2)};
                    const float zs[3] = {z0, z1, __ldg(j.z + h2)};
                    if (!tube_pass(xs[2], ys[2], zs[2], mx, my, c)) continue;
                    float fx, fy;
                    found = fit_pass(xs, ys, zs, c, fx, fy) && chain_pass(xs, ys, zs, mx, my, c);
                    if (kStream && found) {
                        float pmin, pmax;
                        coincident3(__ldg(j.t + h0), __ldg(j.t + h1), __ldg(j.t + h2), j.dt, pmin, pmax);
                        found = partner_coincident(pmin, pmax, Tt, j.dt);
                    }
                }
            }
        }
        if (!found) return false;
    }
    return true;
}

// Shared scratch of the unpruned search of one event (from the caller).
struct GenShared {
    int32_t* soff;  // [3 * kMaxStations + 1] the event's offsets
    int32_t* sh;    // [kShifts] and shifts (free-streaming windows)
    int* s_count;
    int* s_cand;
    int* s_bad;
    unsigned long long* s_pool;
};

constexpr int kGenThreads = 256;  // block size of the unpruned search (both callers)

// distinct_hits on the unpruned path: a second pass over the trigger
// station writes the packed hits of the event's candidates (passing
// triplets; in CHAIN mode those with a compatible triplet in every other
// station) to out[0, cap), ranked by the block-shared counter.
__device__ void generic_candidates(const Job& j, const int32_t* soff, const Cuts& c, unsigned long long* out, int cap,
                                   int* s_rank) {
    const int32_t* o = soff + 3 * j.trig;
    const bool chain = j.mode == 1 && j.S > 1;
    const int64_t n0 = o[1] - o[0], n1 = o[2] - o[1], n2 = o[3] - o[2];
    const int64_t npairs = n0 * n1;
    for (int64_t p = threadIdx.x; p < npairs; p += blockDim.x) {
        const int64_t i = p / n1, jx = p - i * n1;
        const GHit hi = ghit(j, o[0] + i), hj = ghit(j, o[1] + jx);
        if (!hi.p.live || !hj.p.live) continue;
        if (!hi.p.wild && !hj.p.wild && !pair_ok(hi.p.sx, hi.p.sy, hj.p.sx, hj.p.sy, __fadd_rn(hi.p.b, hj.p.b)))
            continue;
        for (int64_t k = 0; k < n2; ++k) {
            const GHit hk = ghit(j, o[2] + k);
            if (!hk.p.live) continue;
            if (!hk.p.wild) {
                if (!hi.p.wild && !pair_ok(hi.p.sx, hi.p.sy, hk.p.sx, hk.p.sy, __fadd_rn(hi.p.b, hk.p.b))) continue;
                if (!hj.p.wild && !pair_ok(hj.p.sx, hj.p.sy, hk.p.sx, hk.p.sy, __fadd_rn(hj.p.b, hk.p.b))) continue;
            }
            const float xs[3] = {hi.x, hj.x, hk.x}, ys[3] = {hi.y, hj.y, hk.y}, zs[3] = {hi.z, hj.z, hk.z};
            float mx, my;
            if (!fit_pass(xs, ys, zs, c, mx, my)) continue;
            if (chain && !road_global(j, soff, nullptr, c, mx, my, make_float2(0.f, 0.f))) continue;  // (no streams here)
            const int r = atomicAdd(s_rank, 1);
            if (r < cap) out[r] = pack_ijk((int)i, (int)jx, (int)k);
        }
    }
}

// The unpruned search of one event by one block: any size, any coordinates
// (pruning only where the per-hit bound is finite).  Counting pass: unit
// counts, track count and recorded entries; emit pass: rows.  All threads of
// the block call it.
template <bool EMIT>
__device__ void generic_event(const Job& j, int64_t e, const GenShared& g) {
    const Cuts c{j.cx, j.cy, j.K};
    const int S = j.S, S3 = 3 * S;
    const bool chain = j.mode == 1 && S > 1;
    const int nproc = j.mode == 1 ? S : 1;
    int32_t* soff = g.soff;
    __syncthreads();  // earlier users of the shared scratch are done
    for (int i = threadIdx.x; i <= S3; i += blockDim.x) {
        soff[i] = j.off[e * S3 + i];
        if (kStream && i < S3) g.sh[i] = j.shift[e * S3 + i];
    }
    if (threadIdx.x == 0) *g.s_cand = 0;
    __syncthreads();
    int trig_count = 0;
    bool bad_event = false;
    for (int si = 0; si < nproc && !bad_event; ++si) {
        const int s = station_of(si, j.trig);
        const int64_t u = e * S + s;
        const int32_t* o = soff + 3 * s;
        const Shift3 b = shift3(g.sh, s);
        if (EMIT && j.unit_counts[u] == 0) continue;
        if (threadIdx.x == 0) {
            *g.s_count = 0;
            *g.s_bad = 0;
        }
        __syncthreads();
        if (!EMIT) {
            for (int32_t p = o[0] + threadIdx.x; p < o[3]; p += blockDim.x)
                if (__ldg(j.z + p + b.at(p, o[1], o[2])) <= 0.0f) *g.s_bad = 1;
            __syncthreads();
            if (*g.s_bad) {
                if (threadIdx.x == 0) {
                    atomicOr(&j.ctrl->status, kStInvalid);
                    j.ev_class[e] = kClsInvalid;
                }
                bad_event = true;
                break;
            }
        }
        const int64_t n0 = o[1] - o[0], n1 = o[2] - o[1], n2 = o[3] - o[2];
        const int64_t npairs = n0 * n1;
        int32_t* rows = EMIT ? j.triplets + 3 * j.trip_off[u] : nullptr;
        const int ulimit = EMIT ? j.unit_counts[u] : 0;
        int local = 0;
        const bool collect = !EMIT && chain && s == j.trig;
        for (int64_t p = threadIdx.x; p < npairs; p += blockDim.x) {
            const int64_t i = p / n1, jx = p - i * n1;
            const GHit hi = ghit(j, o[0] + b.a + i), hj = ghit(j, o[1] + b.b + jx);
            if (!hi.p.live || !hj.p.live) continue;
            if (!hi.p.wild && !hj.p.wild && !pair_ok(hi.p.sx, hi.p.sy, hj.p.sx, hj.p.sy, __fadd_rn(hi.p.b, hj.p.b)))
                continue;
            for (int64_t k = 0; k < n2; ++k) {
                const GHit hk = ghit(j, o[2] + b.c + k);
                if (!hk.p.live) continue;
                if (!hk.p.wild) {
                    if (!hi.p.wild && !pair_ok(hi.p.sx, hi.p.sy, hk.p.sx, hk.p.sy, __fadd_rn(hi.p.b, hk.p.b)))
                        continue;
                    if (!hj.p.wild && !pair_ok(hj.p.sx, hj.p.sy, hk.p.sx, hk.p.sy, __fadd_rn(hj.p.b, hk.p.b)))
                        continue;
                }
                const float xs[3] = {hi.x, hj.x, hk.x}, ys[3] = {hi.y, hj.y, hk.y}, zs[3] = {hi.z, hj.z, hk.z};
                float mx, my;
                if (!fit_pass(xs, ys, zs, c, mx, my)) continue;
                float2 Tt = make_float2(0.f, 0.f);
                if constexpr (kStream) {  // coincident and owned by this window
                    const bool co = coincident3(__ldg(j.t + o[0] + b.a + i), __ldg(j.t + o[1] + b.b + jx), __ldg(j.t + o[2] + b.c + k), j.dt,
                                                Tt.x, Tt.y);
                    if (!(co && Tt.x >= __ldg(j.wb + e) && Tt.x < __ldg(j.wb + e + 1))) continue;
                }
                ++local;
                if (!EMIT && j.tscr) {
                    const int rk = atomicAdd(g.s_count, 1);
                    if (i >= kPackLimit || jx >= kPackLimit || k >= kPackLimit) {
                        atomicOr(&j.ctrl->status, kStNoScratch);
                    } else {
                        const unsigned long long at = atomicAdd(&j.ctrl->scratch_n, 1ull);
                        if (at < (unsigned long long)j.tscr_cap) {
                            TripEntry te;
                            te.unit = (int32_t)u;
                            te.rank = rk;
                            te.ijk = (unsigned long long)i | ((unsigned long long)jx << 20) |
                                     ((unsigned long long)k << 40) | ((unsigned long long)kClsGeneric << kTagShift);
                            j.tscr[at] = te;
                        }
                    }
                }
                if (EMIT) {
                    const int pos = atomicAdd(g.s_count, 1);
                    if (pos < ulimit &&  // never past the unit's rows
                        JPSI_IN(j.ctrl, (rows - j.triplets) / 3 + pos < j.trip_cap)) {
                        int32_t* r = rows + 3 * (int64_t)pos;
                        r[0] = (int32_t)i;
                        r[1] = (int32_t)jx;
                        r[2] = (int32_t)k;
                    }
                }
                if (collect && road_global(j, soff, g.sh, c, mx, my, Tt)) atomicAdd(g.s_cand, 1);
            }
        }
        if (!EMIT && !j.tscr && local) atomicAdd(g.s_count, local);
        __syncthreads();
        if (threadIdx.x == 0) {
            if (EMIT) {
                if (*g.s_count != j.unit_counts[u]) atomicOr(&j.ctrl->status, kStEmitMismatch);
            } else {
                j.unit_counts[u] = *g.s_count;
            }
        }
        if (s == j.trig) trig_count = *g.s_count;
        __syncthreads();
    }
    if (!EMIT && !bad_event && threadIdx.x == 0) {
        if (j.mode == 0)
            for (int s = 0; s < S; ++s)
                if (s != j.trig) j.unit_counts[e * S + s] = 0;
        j.track_counts[e] = chain ? *g.s_cand : trig_count;
    }
    if (!EMIT && !bad_event && j.distinct) {  // block-uniform
        const int nc = chain ? *g.s_cand : trig_count;
        bool f = false;
        if (nc >= 2) {
            __syncthreads();
            if (threadIdx.x == 0) {
                *g.s_pool = atomicAdd(&j.ctrl->tpool_n, (unsigned long long)nc);
                *g.s_count = 0;
            }
            __syncthreads();
            const unsigned long long pb = *g.s_pool;
            if (pb + (unsigned long long)nc <= (unsigned long long)j.tpool_cap) {
                generic_candidates(j, soff, c, j.tpool_ijk + pb, nc, g.s_count);
                __syncthreads();
                f = block_disjoint_pair<kGenThreads>(j.tpool_ijk + pb, nullptr, nc, g.s_bad);
            } else if (threadIdx.x == 0) {
                atomicOr(&j.ctrl->status, kStNoPool);
            }
        }
        if (threadIdx.x == 0) j.dpair[e] = f;
    }
    __syncthreads();
}

// Persistent blocks take the events of the unpruned list.
template <bool EMIT>
__global__ void __launch_bounds__(kGenThreads) k_generic(const __grid_constant__ Job j) {
    __shared__ int32_t soff[3 * kMaxStations + 1];
    __shared__ int32_t sh[kShifts];
    __shared__ int s_gi, s_count, s_cand, s_bad;
    __shared__ unsigned long long s_pool;
    chain_wait();
    const int n_gen = *(volatile int32_t*)&j.ctrl->n_generic, g0 = *(volatile int32_t*)&j.ctrl->g_begin;
    for (;;) {
        if (threadIdx.x == 0) s_gi = g0 + (int)atomicAdd(&j.ctrl->work[EMIT ? 7 : 3], 1ull);
        __syncthreads();
        const int gi = s_gi;
        if (gi >= n_gen) break;
        const int64_t e = j.glist[gi];
        if (!EMIT || j.ev_class[e] == kClsGeneric)
            generic_event<EMIT>(j, e, GenShared{soff, sh, &s_count, &s_cand, &s_bad, &s_pool});
        __syncthreads();
    }
    chain_next();
}

// ------------------------------------------------- one-launch form, blocks

// The one-launch form (jpsi_run_plain) has no event lists, queues, sort,
// pool hand-off or graphs: a static grid of one warp per event (k_light with
// Job::plain), then a static grid of one block per event (below).  A block
// whose event the warp finished returns at once; the others run the whole
// event here: every station on the block tile, or the unpruned search when
// the event does not fit the tile or has extreme coordinates.
constexpr int kPlainTCap = 128;  // trigger slopes kept in shared memory (more: the pool)

struct PlainSmem {
    HeavySmem h;
    float2 T[kPlainTCap];
    uint8_t alive[kPlainTCap];
};

// One block-tile event of the one-launch form.  Returns true when the event
// must go on to the unpruned search (its class is then kClsGeneric).
template <bool EMIT>
__device__ bool plain_block_event(const Job& j, PlainSmem& ps, int64_t e) {
    HeavySmem& sm = ps.h;
    const int tid = threadIdx.x, lane = tid & 31;
    const int S = j.S;
    const bool chain = j.mode == 1 && S > 1;
    const int nproc = j.mode == 1 ? S : 1;
    const Cuts c{j.cx, j.cy, j.K};
    load_event_offsets(j, sm, e);
    if (EMIT) {
        for (int si = 0; si < nproc; ++si) {
            const int s = station_of(si, j.trig);
            if (j.unit_counts[e * S + s] == 0) continue;
            TSink ts{false, nullptr, 0, nullptr};
            int cnt = 0;
            heavy_unit<true>(j, sm, c, kGiPlain, e, s, ts, nullptr, nullptr, 0, cnt,
                             si + 1 < nproc ? station_of(si + 1, j.trig) : -1);
            __syncthreads();
        }
        return false;
    }
    bool fits = true;
    for (int si = 0; si < nproc; ++si) {
        const int32_t* o = sm.off + 3 * station_of(si, j.trig);
        if (o[1] - o[0] > kHLayerCap || o[2] - o[1] > kHLayerCap || o[3] - o[2] > kHLayerCap || o[3] - o[0] > kHHCap)
            fits = false;
    }
    if (!fits) {
        if (tid == 0) j.ev_class[e] = kClsGeneric;
        return true;
    }
    float2* T = ps.T;
    uint8_t* alive = ps.alive;
    unsigned long long* ijk = nullptr;  // distinct_hits: the candidates' packed hits (in the pool)
    float2* tt = nullptr;               // free-streaming windows: the slopes' times (in the pool)
    int trig_count = 0, nT = 0;
    for (int si = 0; si < nproc; ++si) {
        const int s = station_of(si, j.trig);
        if (tid == 0) sm.s_nT = 0;
        __syncthreads();
        TSink ts{(chain || j.distinct) && si == 0, T, kPlainTCap, &sm.s_nT};
        int cnt = 0;
        const int sn = si + 1 < nproc ? station_of(si + 1, j.trig) : -1;
        if (!heavy_unit<false>(j, sm, c, kGiPlain, e, s, ts, T, alive, si == 0 ? 0 : nT, cnt, sn, tt)) {
            __syncthreads();
            return j.ev_class[e] == kClsGeneric;
        }
        __syncthreads();
        if (si > 0) continue;
        trig_count = cnt;
        if (!chain && !j.distinct) break;
        nT = sm.s_nT;
        if (nT > kPlainTCap || (j.distinct && nT >= 2) || (kStream && chain && nT > 0)) {
            // more slopes than the block keeps, or (distinct_hits) the
            // candidates' hits or (free-streaming windows) the slopes' times
            // wanted: room in the batch's pool, and the trigger station once
            // more (same count, nothing recorded)
            if (tid == 0) sm.s_pool = atomicAdd(&j.ctrl->tpool_n, (unsigned long long)nT);
            __syncthreads();
            const unsigned long long pb = sm.s_pool;
            if (pb + (unsigned long long)nT > (unsigned long long)j.tpool_cap) {
                if (tid == 0) j.ev_class[e] = kClsGeneric;
                return true;
            }
            T = j.tpool + pb;
            alive = j.tpool_alive + pb;
            if (j.distinct) ijk = j.tpool_ijk + pb;
            if constexpr (kStream) tt = reinterpret_cast<float2*>(j.tpool_ijk) + pb;
            if (tid == 0) sm.s_nT = 0;
            __syncthreads();
            TSink ts2{true, T, nT, &sm.s_nT};
            ts2.norec = true;
            ts2.ijk = ijk;
            ts2.tt = tt;
            if (!heavy_unit<false>(j, sm, c, kGiPlain, e, s, ts2, nullptr, nullptr, 0, cnt)) {
                __syncthreads();
                return j.ev_class[e] == kClsGeneric;
            }
            __syncthreads();
        }
        if (!chain) {  // PAPER with distinct_hits: every passing trigger triplet is a candidate
            const bool f = nT >= 2 && block_disjoint_pair<kHThreads>(ijk, nullptr, nT, &sm.s_hx);
            if (tid == 0) j.dpair[e] = f;
            break;
        }
        for (int i = tid; i < nT; i += kHThreads) alive[i] = 1;
        __syncthreads();
    }
    int tc = trig_count;
    if (chain) {
        if (tid == 0) sm.s_cand = 0;
        __syncthreads();
        int a = 0;
        for (int ti = tid; ti < nT; ti += kHThreads) a += alive[ti];
        a = __reduce_add_sync(kFull, a);
        if (lane == 0 && a) atomicAdd(&sm.s_cand, a);
        __syncthreads();
        tc = sm.s_cand;
        if (j.distinct) {
            const bool f = nT >= 2 && block_disjoint_pair<kHThreads>(ijk, alive, nT, &sm.s_hx);
            if (tid == 0) j.dpair[e] = f;
        }
    }
    if (tid == 0) {
        if (j.mode == 0)
            for (int s = 0; s < S; ++s)
                if (s != j.trig) j.unit_counts[e * S + s] = 0;
        j.track_counts[e] = tc;
    }
    return false;
}

template <bool EMIT>
__global__ void __launch_bounds__(kHThreads, 3) k_plain_block(const __grid_constant__ Job j) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    chain_wait();
    PlainSmem& ps = *reinterpret_cast<PlainSmem*>(smem_raw);
    const int64_t e = j.ev_begin + blockIdx.x;
    if (e >= j.ev_begin + j.ev_count) return;
    const uint8_t cls = j.ev_class[e];
    bool generic = cls == kClsGeneric;
    if (cls == kClsHeavy) generic = plain_block_event<EMIT>(j, ps, e);
    if (generic) generic_event<EMIT>(j, e, GenShared{ps.h.off, ps.h.sh, &ps.h.s_rank, &ps.h.s_cand, &ps.h.s_next, &ps.h.s_pool});
}

// -------------------------------------------------------- accept bits

__global__ void k_accept(const __grid_constant__ Job j) {
    chain_next();
    chain_wait();
    if (!j.accept_bits) return;
    const int64_t nwords = (j.n_events + 31) / 32;
    const int lane = threadIdx.x & 31;
    const int64_t wstride = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); w < nwords; w += wstride) {
        const int64_t e = w * 32 + lane;
        // distinct_hits with min_candidates 2: two candidates sharing no hit
        const bool v = e < j.n_events && (j.distinct && j.minc == 2 ? j.dpair[e] != 0 : j.track_counts[e] >= j.minc);
        const unsigned bits = __ballot_sync(kFull, v);
        if (lane == 0) j.accept_bits[w] = bits;
    }
}

// --------------------------------------------------------------- scan

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t* sh, int64_t& total) {
    // sh: kScanThreads/32 + 1 entries
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int64_t incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int64_t o = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) sh[w] = incl;
    __syncthreads();
    if (w == 0) {
        const int nw = blockDim.x >> 5;
        int64_t s = lane < nw ? sh[lane] : 0;
        int64_t si = s;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int64_t o = __shfl_up_sync(kFull, si, d);
            if (lane >= d) si += o;
        }
        if (lane < nw) sh[lane] = si - s;
        if (lane == 31) sh[32] = si;
    }
    __syncthreads();
    const int64_t r = sh[w] + incl - v;
    total = sh[32];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const __grid_constant__ Job j) {
    __shared__ int64_t sh[33];
    chain_next();
    chain_wait();
    const int64_t n = j.n_events * j.S;
    const int64_t ntiles = (n + kScanTile - 1) / kScanTile;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        int64_t v = 0;
        const int64_t b = tile * kScanTile + (int64_t)threadIdx.x * kScanItems;
#pragma unroll
        for (int q = 0; q < kScanItems; ++q)
            if (b + q < n) v += j.unit_counts[b + q];
        int64_t total;
        block_excl_scan(v, sh, total);
        if (threadIdx.x == 0) j.block_sums[tile] = total;
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_top(const __grid_constant__ Job j) {
    __shared__ int64_t sh[33];
    chain_next();
    chain_wait();
    const int64_t n = j.n_events * j.S;
    const int64_t ntiles = (n + kScanTile - 1) / kScanTile;
    int64_t carry = 0;
    for (int64_t b = 0; b < ntiles; b += kScanThreads) {
        const int64_t i = b + threadIdx.x;
        const int64_t v = i < ntiles ? j.block_sums[i] : 0;
        int64_t total;
        const int64_t ex = block_excl_scan(v, sh, total);
        if (i < ntiles) j.block_sums[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) {
        j.trip_off[n] = carry;
        j.ctrl->trip_total = carry;
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_down(const __grid_constant__ Job j) {
    __shared__ int64_t sh[33];
    chain_next();
    chain_wait();
    const int64_t n = j.n_events * j.S;
    const int64_t ntiles = (n + kScanTile - 1) / kScanTile;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t b = tile * kScanTile + (int64_t)threadIdx.x * kScanItems;
        int32_t v[kScanItems];
        int64_t sum = 0;
#pragma unroll
        for (int q = 0; q < kScanItems; ++q) {
            v[q] = b + q < n ? j.unit_counts[b + q] : 0;
            sum += v[q];
        }
        int64_t total;
        int64_t run = block_excl_scan(sum, sh, total) + j.block_sums[tile];
#pragma unroll
        for (int q = 0; q < kScanItems; ++q)
            if (b + q < n) {
                j.trip_off[b + q] = run;
                run += v[q];
            }
    }
}

// ------------------------------------------------------ triplet scatter

// Moves each recorded triplet to its row trip_off[unit] + rank.  Entries
// written by a path that did not keep the event (it moved on to the next
// path part-way) are dropped; the final path recorded the event again.
__global__ void k_scatter(const __grid_constant__ Job j) {
    chain_next();
    chain_wait();
    // enqueued behind the count: only a record and a buffer that hold every triplet
    const unsigned long long n = j.ctrl->scratch_n;
    if (!j.triplets || n > (unsigned long long)j.tscr_cap || j.ctrl->trip_total > j.trip_cap ||
        (*(volatile int32_t*)&j.ctrl->status & (kStInvalid | kStNoScratch | kStNoPool)))
        return;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long q = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride) {
        const TripEntry te = j.tscr[q];
        const int64_t e = te.unit / j.S;
        const unsigned tag = (unsigned)((te.ijk >> kTagShift) & 7u);
        if (j.ev_class[e] != tag) continue;
        const int64_t row = j.trip_off[te.unit] + te.rank;
        if (!JPSI_IN(j.ctrl, row >= 0 && row < j.trip_cap)) continue;
        int32_t* r = j.triplets + 3 * row;
        r[0] = (int32_t)(te.ijk & 0xfffffu);
        r[1] = (int32_t)((te.ijk >> 20) & 0xfffffu);
        r[2] = (int32_t)((te.ijk >> 40) & 0xfffffu);
    }
}

// ------------------------------------------------- per-layer z geometry

// Per-hit z from a detector geometry table (every hit of layer l of station s
// at z_layer[s*3 + l]) for events [ev0, ev1): warps take events in turn and fill
// one layer after the other.  Bound by the stores (a search of each hit's layer,
// six dependent reads of shared memory, took 52 us for 11.9 M hits, this 16).  Writes stay inside [0, n_hits)
// whatever the offsets hold (malformed offsets fail the selection afterwards).
__global__ void __launch_bounds__(256) k_expand_z(const int32_t* __restrict__ off,
                                                  const float* __restrict__ z_layer, float* __restrict__ z,
                                                  int64_t ev0, int64_t ev1, int S, int64_t n_hits) {
    const int S3 = 3 * S, lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t e = ev0 + (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); e < ev1; e += nwarps) {
        const int32_t* o = off + e * S3;
        const int64_t end = min((int64_t)__ldg(o + S3), n_hits);
        int64_t done = 0;
        for (int l0 = 0; l0 < S3; l0 += 31) {  // 31 layers: 32 offsets, one per lane
            const int m = min(31, S3 - l0);
            const int32_t mine = __ldg(o + l0 + min(lane, m));
            const float zmine = __ldg(z_layer + l0 + min(lane, m - 1));
            for (int l = 0; l < m; ++l) {
                const int64_t h0 = max((int64_t)__shfl_sync(kFull, mine, l), done);  // (never a hit twice)
                const int64_t h1 = min((int64_t)__shfl_sync(kFull, mine, l + 1), end);
                const float v = __shfl_sync(kFull, zmine, l);
#pragma unroll 4
                for (int64_t h = h0 + lane; h < h1; h += 32) z[h] = v;
                done = max(done, h1);
            }
        }
    }
}

// ------------------------------------------------------------ launchers

size_t light_smem_bytes(int wpb) { return (size_t)wpb * sizeof(WarpTile); }
static size_t medium_smem_bytes() { return sizeof(MediumTile); }
size_t heavy_smem_bytes() { return sizeof(HeavySmem); }
static size_t plain_smem_bytes() { return sizeof(PlainSmem); }

// Kernel attributes are per device: set once for each device a context or a
// call runs on (serving threads may get here at the same time).
static std::mutex g_attr_mu;
static uint64_t g_attr_done = 0;  // bit d: device d done (devices >= 64: every call)

static cudaError_t ensure_attrs() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_attr_mu);
    const uint64_t bit = dev < 64 ? (uint64_t)1 << dev : 0;
    if (g_attr_done & bit) return cudaSuccess;
    const int maxw = 8;
    e = cudaFuncSetAttribute(k_light<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)light_smem_bytes(maxw));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_light<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)light_smem_bytes(maxw));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_medium<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)medium_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_medium<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)medium_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_heavy, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)heavy_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_heavy_units<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)heavy_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_heavy_units<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)heavy_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_plain_block<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)plain_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_plain_block<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)plain_smem_bytes());
    if (e == cudaSuccess) g_attr_done |= bit;
    return e;
}

int light_max_blocks_per_sm(int wpb) {
    if (ensure_attrs() != cudaSuccess) return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_light<false>, wpb * 32, light_smem_bytes(wpb)) !=
        cudaSuccess)
        return 0;
    return nb;
}

int heavy_max_blocks_per_sm() {
    if (ensure_attrs() != cudaSuccess) return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_heavy, kHThreads, heavy_smem_bytes()) !=
        cudaSuccess)
        return 0;
    return nb;
}

int medium_max_blocks_per_sm() {
    if (ensure_attrs() != cudaSuccess) return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_medium<false>, MediumTile::THREADS, medium_smem_bytes()) !=
        cudaSuccess)
        return 0;
    return nb;
}

int generic_max_blocks_per_sm(int threads) {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_generic<false>, threads, 0) != cudaSuccess) return 0;
    return nb;
}

// Blocks of a captured kernel that can have work for this job, at most `full`:
// small batches do not pay for the setup of grids that fill the chip (an empty
// k_medium with its 2128 blocks takes 8 us, a one-tile scan over 304 blocks 6).
unsigned useful_blocks(const void* f, const Job& j, unsigned full) {
    const int64_t ne = std::max<int64_t>(j.ev_count, 1), words = (j.n_events + 31) / 32;
    int64_t n = full;
    if (f == (const void*)k_light<false> || f == (const void*)k_light<true>)
        n = (ne + j.grab - 1) / j.grab;  // (a block's further warps find no event)
    else if (f == (const void*)k_medium<false> || f == (const void*)k_heavy || f == (const void*)k_generic<false>)
        n = ne;
    else if (f == (const void*)k_heavy_units<false>)
        n = ne * std::max(j.S - 1, 1);
    else if (f == (const void*)k_heavy_final)
        n = (ne + 7) / 8;
    else if (f == (const void*)k_accept)
        n = (words + 7) / 8;
    else if (f == (const void*)k_scan_reduce || f == (const void*)k_scan_down)
        n = (j.n_events * j.S + kScanTile - 1) / kScanTile;
    return (unsigned)std::min<int64_t>(full, std::max<int64_t>(n, 1));
}

const void* light_count_kernel_ptr() { return (const void*)k_light<false>; }

// Launches a kernel of a run behind the one before it on the stream (see
// chain_wait): its blocks are set up while the one before drains.
template <class A>
static void chain_launch(void (*k)(A), unsigned grid, unsigned block, size_t smem, cudaStream_t st, const A& a) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    (void)cudaLaunchKernelEx(&cfg, k, a);  // errors: cudaGetLastError of the launchers
}

// Kernels take the job by value (a __grid_constant__ parameter), so every
// field read is a constant-bank operand rather than a load.
cudaError_t launch_light_count(const Job& job, int64_t n_events, const LaunchCfg& lc, bool persistent,
                               cudaStream_t st) {
    cudaError_t e = ensure_attrs();
    if (e != cudaSuccess) return e;
    const int wpb = lc.light_wpb;
    const size_t smem = light_smem_bytes(wpb);
    Job j = job;
    j.persistent = persistent ? 1 : 0;
    const int64_t nb = persistent ? lc.light_blocks : std::max<int64_t>((n_events + wpb - 1) / wpb, 1);
    k_light<false><<<(unsigned)nb, wpb * 32, smem, st>>>(j);
    return cudaGetLastError();
}

cudaError_t launch_count_lists(const Job& j, const LaunchCfg& lc, cudaStream_t st) {
    chain_launch(k_medium<false>, lc.medium_blocks, MediumTile::THREADS, medium_smem_bytes(), st, j);
    chain_launch(k_sort_heavy, 1, 1024, 0, st, j);
    chain_launch(k_heavy, lc.heavy_blocks, kHThreads, heavy_smem_bytes(), st, j);
    chain_launch(k_heavy_units<false>, lc.heavy_blocks, kHThreads, heavy_smem_bytes(), st, j);
    chain_launch(k_heavy_final, lc.scan_blocks, 256, 0, st, j);
    chain_launch(k_generic<false>, lc.generic_blocks, kGenThreads, 0, st, j);
    return cudaGetLastError();
}

cudaError_t launch_count_tail(const Job& j, const LaunchCfg& lc, cudaStream_t st) {
    chain_launch(k_accept, lc.scan_blocks, 256, 0, st, j);
    chain_launch(k_scan_reduce, lc.scan_blocks, kScanThreads, 0, st, j);
    chain_launch(k_scan_top, 1, kScanThreads, 0, st, j);
    chain_launch(k_scan_down, lc.scan_blocks, kScanThreads, 0, st, j);
    return cudaGetLastError();
}

cudaError_t launch_count_rest(const Job& j, const LaunchCfg& lc, cudaStream_t st) {
    const cudaError_t e = launch_count_lists(j, lc, st);
    return e != cudaSuccess ? e : launch_count_tail(j, lc, st);
}

cudaError_t launch_expand_z(const int32_t* off, const float* z_layer, float* z, int64_t ev0, int64_t ev1, int S,
                            int64_t n_hits, int n_sm, cudaStream_t st) {
    if (ev1 <= ev0) return cudaSuccess;
    const int64_t grid = std::min<int64_t>((ev1 - ev0 + 7) / 8, (int64_t)n_sm * 8);
    k_expand_z<<<(unsigned)grid, 256, 0, st>>>(off, z_layer, z, ev0, ev1, S, n_hits);
    return cudaGetLastError();
}

// One-launch form: the static warp grid, then the static block grid and the
// tail (accept bits, scan); its emit phase is the same two grids.
static cudaError_t launch_plain_grids(const Job& job, bool emit, bool warps, bool blocks, const LaunchCfg& lc,
                                      cudaStream_t st) {
    cudaError_t e = ensure_attrs();
    if (e != cudaSuccess) return e;
    Job j = job;
    j.persistent = 0;
    j.plain = 1;
    const int wpb = lc.light_wpb;
    const int64_t n = j.ev_count;
    if (warps) {
        const int64_t nb = std::max<int64_t>((n + wpb - 1) / wpb, 1);
        if (emit)
            k_light<true><<<(unsigned)nb, wpb * 32, light_smem_bytes(wpb), st>>>(j);
        else
            k_light<false><<<(unsigned)nb, wpb * 32, light_smem_bytes(wpb), st>>>(j);
    }
    if (blocks) {
        const unsigned nb = (unsigned)std::max<int64_t>(n, 1);
        if (emit)
            k_plain_block<true><<<nb, kHThreads, plain_smem_bytes(), st>>>(j);
        else
            k_plain_block<false><<<nb, kHThreads, plain_smem_bytes(), st>>>(j);
    }
    return cudaGetLastError();
}

cudaError_t launch_plain_light(const Job& j, const LaunchCfg& lc, cudaStream_t st) {
    return launch_plain_grids(j, false, true, false, lc, st);
}

cudaError_t launch_plain_rest(const Job& j, const LaunchCfg& lc, cudaStream_t st) {
    const cudaError_t e = launch_plain_grids(j, false, false, true, lc, st);
    return e != cudaSuccess ? e : launch_count_tail(j, lc, st);
}

cudaError_t launch_plain_emit(const Job& j, const LaunchCfg& lc, cudaStream_t st) {
    return launch_plain_grids(j, true, true, true, lc, st);
}

cudaError_t launch_scatter(const Job& j, const LaunchCfg& lc, cudaStream_t st) {
    chain_launch(k_scatter, lc.scan_blocks, 256, 0, st, j);
    return cudaGetLastError();
}

cudaError_t launch_emit_phase(const Job& job, int64_t n_events, const LaunchCfg& lc, bool persistent,
                              cudaStream_t st) {
    cudaError_t e = ensure_attrs();
    if (e != cudaSuccess) return e;
    const int wpb = lc.light_wpb;
    const size_t smem = light_smem_bytes(wpb);
    Job j = job;
    j.persistent = persistent ? 1 : 0;
    const int64_t nb = persistent ? lc.light_blocks : std::max<int64_t>((n_events + wpb - 1) / wpb, 1);
    k_light<true><<<(unsigned)nb, wpb * 32, smem, st>>>(j);
    k_medium<true><<<lc.medium_blocks, MediumTile::THREADS, medium_smem_bytes(), st>>>(j);
    k_heavy_units<true><<<lc.heavy_blocks, kHThreads, heavy_smem_bytes(), st>>>(j);
    k_generic<true><<<lc.generic_blocks, kGenThreads, 0, st>>>(j);
    return cudaGetLastError();
}

#if JPSI_STREAM
// ------------------------------------------- free-streaming event building
//
// A timeslice's hits are grouped by (station, layer), each group sorted by
// time.  Window k = [b_k, b_k+1) becomes event k of a window batch: group g
// of event k holds the group-g hits whose times lie in the window's range
// (the trigger station: [b_k, fl32(b_k+1 + dt)], which holds every triplet
// owned by the window; the other stations of CHAIN mode from a margin below
// b_k - dt to the same end, which holds every partner that can be coincident
// with such a triplet).  The batch is only offsets and shifts: the selection
// kernels of this build read the hits where they lie in the timeslice (a copy
// of the ranges took 0.96 ms of a 10^5-collision timeslice, 3.53 ms, and 16
// bytes per hit of the ranges) and apply the time tests themselves; the rows
// they write index the window batch and are moved back to timeslice group
// indices at the end.

// Last group q < S3 with so[q] <= h (so: the 3S+1 offsets, non-decreasing).
__device__ __forceinline__ int group_of(const int32_t* so, int S3, int64_t h) {
    int q = 0;
#pragma unroll
    for (int step = 32; step > 0; step >>= 1)
        if (q + step < S3 && so[q + step] <= h) q += step;
    return q;
}

// First index in [lo, hi) whose time is >= v (> v with STRICT); stays in
// [lo, hi] whatever the times hold.
template <bool STRICT>
__device__ __forceinline__ int64_t t_search(const float* __restrict__ t, int64_t lo, int64_t hi, float v) {
    while (lo < hi) {
        const int64_t m = lo + ((hi - lo) >> 1);
        const float tm = __ldg(t + m);
        if (STRICT ? tm <= v : tm < v)
            lo = m + 1;
        else
            hi = m;
    }
    return lo;
}

// The timeslice's own checks: times sorted within each group and not NaN,
// z > 0 for every hit of a station the mode reads, window bounds finite and
// strictly increasing.  Sets kStInvalid.
//   Bound by the reads of t and z.  A block takes one run of the hits, 1024 at a
// time, with four loads of each array in flight per thread; nearly always they
// are of one group, which moves on with the run (a search per hit made this an
// instruction-bound kernel: 120 M hits 590 -> 235 us).
__global__ void __launch_bounds__(256) k_win_check(const __grid_constant__ WinJob w) {
    __shared__ int32_t so[3 * kMaxStations + 1];
    const int S3 = 3 * w.S;
    for (int i = threadIdx.x; i <= S3; i += blockDim.x) so[i] = w.off[i];
    __syncthreads();
    bool bad = false;
    constexpr int Q = 4;
    const int64_t run = ((w.n_hits + gridDim.x - 1) / gridDim.x + 256 * Q - 1) / (256 * Q) * (256 * Q);
    const int64_t c0 = blockIdx.x * run, c1 = min(c0 + run, w.n_hits);
    int gb = c0 < c1 ? group_of(so, S3, c0) : 0;
    for (int64_t c = c0; c < c1; c += 256 * Q) {
        const int64_t last = min(c + 256 * Q, c1) - 1, h0 = c + threadIdx.x;
        while (gb < S3 - 1 && so[gb + 1] <= c) ++gb;
        const bool one = so[gb + 1] > last;  // (so[S3] = n_hits)
        const int ge = one ? gb : S3 - 1;
        const bool zread = w.z && (w.chain || (gb <= 3 * w.trig + 2 && ge >= 3 * w.trig));
        float t[Q], before[Q], z[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t h = min(h0 + 256 * q, last);
            t[q] = __ldg(w.t + h);
            before[q] = h > 0 ? __ldg(w.t + h - 1) : -INFINITY;
            z[q] = zread ? __ldg(w.z + h) : 1.0f;
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t h = min(h0 + 256 * q, last);
            const int g = one ? gb : group_of(so, S3, h);
            if (isnan(t[q]) || (h > so[g] && !(t[q] >= before[q]))) bad = true;
            if ((w.chain || g / 3 == w.trig) && z[q] <= 0.f) bad = true;
        }
    }
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w.K > 0 && k <= w.K; k += stride) {
        const float b = __ldg(w.wb + k);  // (no windows: bounds may be null)
        if (!isfinite(b) || (k > 0 && !(b > __ldg(w.wb + k - 1)))) bad = true;
    }
    if (!w.z && blockIdx.x == 0 && threadIdx.x < S3) {
        const int g = threadIdx.x;
        if (so[g + 1] > so[g] && (w.chain || g / 3 == w.trig) && __ldg(w.z_layer + g) <= 0.f) bad = true;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&w.ctrl->status, kStInvalid);
}

// Each (window, group) range: first hit and size.
__global__ void __launch_bounds__(256) k_win_ranges(const __grid_constant__ WinJob w) {
    __shared__ int32_t so[3 * kMaxStations + 1];
    const int S3 = 3 * w.S;
    for (int i = threadIdx.x; i <= S3; i += blockDim.x) so[i] = w.off[i];
    __syncthreads();
    const int64_t n = w.K * S3, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride) {
        const int64_t k = q / S3;
        const int g = (int)(q - k * S3), s = g / 3;
        int64_t lo = so[g], hi = so[g];
        if (s == w.trig || w.chain) {
            const float b0 = __ldg(w.wb + k), end = __fadd_rn(__ldg(w.wb + k + 1), w.dt);
            float from = b0;
            if (s != w.trig) {
                // a partner's hits are no earlier than (latest trigger-triplet
                // time) - dt, less one rounding of the sum: a margin of 1e-6
                // relative covers it, the exact tests decide
                double lod = (double)b0 - (double)w.dt;
                lod -= 1e-6 * (fabs((double)b0) + (double)w.dt) + 1e-30;
                from = nextafterf(__double2float_rn(lod), -INFINITY);
            }
            lo = t_search<false>(w.t, so[g], so[g + 1], from);
            // the end lies a window on: steps of doubling length find a short
            // interval that holds it (1.2 M ranges of 10 M hits each: 183 -> 99 us)
            int64_t a = lo, step = 64, to = so[g + 1];
            while (a + step < to && __ldg(w.t + a + step) <= end) {
                a += step;
                step *= 2;
            }
            hi = t_search<true>(w.t, a, min(a + step, to), end);
        }
        w.wlo[q] = (int32_t)lo;
        w.wcnt[q] = (int32_t)(hi - lo);
    }
}

// The window batch: its offsets (from the scan), and how far its hits lie from
// there in the timeslice.  The selection reads them where they are.
__global__ void __launch_bounds__(256) k_win_place(const __grid_constant__ WinJob w) {
    const int64_t n = w.K * 3 * w.S, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q <= n; q += stride) {
        const int64_t at = w.woff[q];
        w.off_out[q] = (int32_t)at;
        if (q < n) w.wcnt[q] = (int32_t)(w.wlo[q] - at);  // (the sizes are in the scan)
    }
}

// The window batch of few windows of a large timeslice without per-hit z: its
// offsets, and its hits copied there, one warp per (window, group) range.
__global__ void __launch_bounds__(256) k_win_gather(const __grid_constant__ WinJob w) {
    const int S3 = 3 * w.S, lane = threadIdx.x & 31;
    const int64_t n = w.K * S3, nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < n; q += nwarps) {
        const int64_t at = w.woff[q], lo = w.wlo[q], cnt = w.woff[q + 1] - at;
        const float v = __ldg(w.z_layer + (int)(q % S3));
        if (lane == 0) {
            w.off_out[q] = (int32_t)at;
            w.wcnt[q] = 0;
        }
        for (int64_t i = lane; i < cnt; i += 32) {
            w.xo[at + i] = __ldg(w.x + lo + i);
            w.yo[at + i] = __ldg(w.y + lo + i);
            w.to[at + i] = __ldg(w.t + lo + i);
            w.zo[at + i] = v;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) w.off_out[n] = (int32_t)w.woff[n];
}

// Per-hit z of the timeslice from the per-group table.
__global__ void __launch_bounds__(256) k_win_fill_z(const __grid_constant__ WinJob w, float* __restrict__ z) {
    __shared__ int32_t so[3 * kMaxStations + 1];
    const int S3 = 3 * w.S;
    for (int i = threadIdx.x; i <= S3; i += blockDim.x) so[i] = w.off[i];
    __syncthreads();
    for (int g = 0; g < S3; ++g) {
        const float v = __ldg(w.z_layer + g);
        for (int64_t h = so[g] + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; h < so[g + 1];
             h += (int64_t)gridDim.x * blockDim.x)
            z[h] = v;
    }
}

// Triplet rows of unit (k, s): window-batch layer indices plus the start of
// the window's range in the timeslice group, less the group's start.
__global__ void __launch_bounds__(256) k_win_rows(const __grid_constant__ WinJob w, const int64_t* trip_off,
                                                  int32_t* tr) {
    const int64_t nu = w.K * w.S;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < nu; u += nwarps) {
        const int64_t a = trip_off[u], b = trip_off[u + 1];
        if (a == b) continue;
        const int64_t k = u / w.S;
        const int s = (int)(u - k * w.S);
        const int64_t q = k * 3 * w.S + 3 * s;
        const int32_t d0 = w.wlo[q] - __ldg(w.off + 3 * s), d1 = w.wlo[q + 1] - __ldg(w.off + 3 * s + 1),
                      d2 = w.wlo[q + 2] - __ldg(w.off + 3 * s + 2);
        for (int64_t r = a + lane; r < b; r += 32) {
            tr[3 * r] += d0;
            tr[3 * r + 1] += d1;
            tr[3 * r + 2] += d2;
        }
    }
}

static unsigned win_grid(int64_t threads, int n_sm) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((threads + 255) / 256, (int64_t)n_sm * 8));
}

cudaError_t launch_window_ranges(const WinJob& w, cudaStream_t st) {
    const int64_t n = w.K * 3 * w.S;
    k_win_check<<<win_grid(std::max(w.n_hits, w.K + 1), w.n_sm), 256, 0, st>>>(w);
    k_win_ranges<<<win_grid(n, w.n_sm), 256, 0, st>>>(w);
    // the sizes' scan, with the scan kernels of the selection reading a job
    // whose "units" are the (window, group) ranges
    Job j{};
    j.n_events = w.K;
    j.S = 3 * w.S;
    j.unit_counts = w.wcnt;
    j.block_sums = w.block_sums;
    j.trip_off = w.woff;
    j.ctrl = w.ctrl;
    chain_launch(k_scan_reduce, w.n_sm * 2, kScanThreads, 0, st, j);
    chain_launch(k_scan_top, 1, kScanThreads, 0, st, j);
    chain_launch(k_scan_down, w.n_sm * 2, kScanThreads, 0, st, j);
    return cudaGetLastError();
}

cudaError_t launch_window_place(const WinJob& w, cudaStream_t st) {
    k_win_place<<<win_grid(w.K * 3 * w.S + 1, w.n_sm), 256, 0, st>>>(w);
    return cudaGetLastError();
}

cudaError_t launch_window_gather(const WinJob& w, cudaStream_t st) {
    k_win_gather<<<win_grid(w.K * 3 * w.S * 32, w.n_sm), 256, 0, st>>>(w);
    return cudaGetLastError();
}

cudaError_t launch_window_z(const WinJob& w, float* z, cudaStream_t st) {
    k_win_fill_z<<<win_grid(w.n_hits / (3 * w.S) + 1, w.n_sm), 256, 0, st>>>(w, z);
    return cudaGetLastError();
}

cudaError_t launch_window_rows(const WinJob& w, const int64_t* trip_off, int32_t* triplets, cudaStream_t st) {
    k_win_rows<<<win_grid(w.K * w.S * 32, w.n_sm), 256, 0, st>>>(w, trip_off, triplets);
    return cudaGetLastError();
}
#endif  // JPSI_STREAM

}  // namespace basek / streamk
}  // namespace jpsi

#if !JPSI_STREAM
// ======================================================================
// Allocation-free counting entry point (jpsi_select_noalloc, include/jpsi.h).
//
// For callers that may not allocate device memory at run time.  Its only
// scratch is the file-scope array below: the control block, one class byte
// per event and the three per-event lists of the warp kernel, for at most
// kNoAllocMaxEvents events (the job itself is a kernel parameter).  Every GPU that loads the
// library holds the array until the process exits.  Host code must not use
// the array's name as a device address: each device's address comes from
// cudaGetSymbolAddress, taken once per device with that device current.
// ======================================================================
namespace jpsi {

constexpr int64_t kNoAllocMaxEvents = (int64_t)1 << 18;  // 262,144 events per call
constexpr size_t kNoAllocCtrlOff = 0;
constexpr size_t kNoAllocClassOff = 512;
constexpr size_t kNoAllocListOff = kNoAllocClassOff + (size_t)kNoAllocMaxEvents;
constexpr size_t kNoAllocBytes = kNoAllocListOff + 3 * sizeof(int32_t) * (size_t)kNoAllocMaxEvents;
static_assert(sizeof(Ctrl) <= kNoAllocClassOff - kNoAllocCtrlOff, "control block slot");

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

constexpr int kNoAllocMaxDevices = 64;
static std::mutex g_noalloc_mu;
static unsigned char* g_noalloc_dev[kNoAllocMaxDevices];  // device address of the array, per device

// Device address of the scratch array on `dev` (the current device).
static cudaError_t noalloc_scratch(int dev, unsigned char** out) {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_dev[dev]) {
        void* ptr = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_dev[dev] = static_cast<unsigned char*>(ptr);
    }
    *out = g_noalloc_dev[dev];
    return cudaSuccess;
}

}  // namespace jpsi

extern "C" jpsi_status jpsi_select_noalloc(const jpsi_params* p, const jpsi_batch* b, int32_t* track_counts,
                                           int32_t* unit_counts, void* cuda_stream) {
    using namespace jpsi;
    using namespace jpsi::basek;
    if (!p || !b) return JPSI_EINVAL;
    if (p->n_stations < 1 || p->n_stations > kMaxStations || p->trigger_station < 0 ||
        p->trigger_station >= p->n_stations || (p->mode != JPSI_MODE_PAPER && p->mode != JPSI_MODE_CHAIN) ||
        p->ndf < 1 || p->min_candidates < 0 || !(p->t_xz >= 0.0f) || !(p->t_yz >= 0.0f) ||
        std::isinf(p->t_xz) || std::isinf(p->t_yz) || p->distinct_hits != 0)
        return JPSI_EINVAL;  // (distinct_hits changes accept bits only, which this entry point does not return)
    if (b->n_events < 0 || b->n_events > kNoAllocMaxEvents) return JPSI_EINVAL;  // beyond the static scratch
    if (b->n_hits < 0 || b->n_hits >= ((int64_t)1 << 31) || (b->n_events == 0 && b->n_hits != 0)) return JPSI_EINVAL;
    if (b->n_events == 0) return JPSI_OK;
    if (!b->offsets || (b->n_hits > 0 && (!b->x || !b->y || !b->z)) || !track_counts || !unit_counts)
        return JPSI_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) return JPSI_ECUDA;
    unsigned char* base = nullptr;
    if (noalloc_scratch(dev, &base) != cudaSuccess) return JPSI_ECUDA;
    Ctrl* dctrl = reinterpret_cast<Ctrl*>(base + kNoAllocCtrlOff);
    Job j{};
    j.x = b->x;
    j.y = b->y;
    j.z = b->z;
    j.off = b->offsets;
    j.n_events = b->n_events;
    j.n_hits = j.n_src = b->n_hits;
    j.ev_begin = 0;
    j.ev_count = b->n_events;
    j.S = p->n_stations;
    j.trig = p->trigger_station;
    j.mode = p->mode;
    j.minc = p->min_candidates;
    j.cx = (float)p->ndf * p->t_xz;
    j.cy = (float)p->ndf * p->t_yz;
    {  // pruning slope factor sqrt(max C)(1 + 1e-4) + 1e-20, rounded up (as for contexts)
        const double kk = std::sqrt((double)std::max(j.cx, j.cy)) * (1.0 + 1e-4) + 1e-20;
        float f = (float)kk;
        if ((double)f < kk) f = std::nextafter(f, INFINITY);
        j.K = f;
    }
    j.cap_small = SmallCfg::LAYER_CAP;
    j.cap_medium = MediumCfg::LAYER_CAP;
    j.persistent = 1;
    j.unit_counts = unit_counts;
    j.track_counts = track_counts;
    j.ev_class = base + kNoAllocClassOff;
    int32_t* lists = reinterpret_cast<int32_t*>(base + kNoAllocListOff);
    j.mlist = lists;
    j.hlist = lists + kNoAllocMaxEvents;
    j.glist = lists + 2 * kNoAllocMaxEvents;
    j.ctrl = dctrl;  // tlist, accept bits, offsets, triplets and entries stay null: the warp kernel alone runs
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    int n_sm = 0;
    if (cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return JPSI_ECUDA;
    const int wpb = 4;
    const int per_sm = light_max_blocks_per_sm(wpb);
    if (per_sm < 1) return JPSI_ECUDA;
    j.grab = b->n_events > (int64_t)4 * wpb * n_sm * per_sm ? 2 : 1;  // (as for contexts)
    if (cudaMemsetAsync(dctrl, 0, sizeof(Ctrl), st) != cudaSuccess) return JPSI_ECUDA;  // counters start at zero
    k_light<false><<<n_sm * per_sm, 32 * wpb, light_smem_bytes(wpb), st>>>(j);
    if (cudaGetLastError() != cudaSuccess) return JPSI_ECUDA;
    Ctrl ctl{};
    if (cudaMemcpyAsync(&ctl, dctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, st) != cudaSuccess) return JPSI_ECUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return JPSI_ECUDA;
    if (ctl.status & kStBounds) return JPSI_ECUDA;  // (checked build only)
    if (ctl.status & kStInvalid) return JPSI_EINVAL;
    // an event beyond the warp tile (or with extreme coordinates) needs the
    // other kernels and their scratch: not available here
    if (ctl.n_medium + ctl.n_heavy + ctl.n_generic > 0) return JPSI_EINVAL;
    return JPSI_OK;
}
#endif  // !JPSI_STREAM
