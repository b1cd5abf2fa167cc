// Several time steps of one tile in a single launch (FP32 / FP16 storage): a
// block copies its tile with a margin from the source buffer into shared
// memory, updates it in place k times while the part of the margin that is
// still correct shrinks by one cell a step, and writes its output cells to the
// other buffer. One pass over memory then serves k steps, at the price of
// updating the margins of neighbouring tiles twice.
//
// The region is RX x RY cells (compile-time, so that every shared-memory
// access is a base register plus an immediate). A launch of k steps outputs
// RX - 2 margin columns (the margin is k rounded up to the 4 cells of a 16-byte
// copy) and RY - 2k rows of it. The populations have one slot per cell and
// direction, in alternating layouts:
//   odd steps   pull direction i of cell x from slot (x - e_i, i) and store it
//               in the slots they read, (x + e_i, opp(i));
//   even steps  therefore find their pulled populations in their own slots
//               (x, opp(i)), and store to (x, i);
//   step k      stores to global memory.
// No slot is read or written by two cells in one step, so a step needs no
// second copy and one barrier. Solid cells are not updated, which leaves the
// slots a halfway wall link i (source x - e_i solid) would be pulled from to
// the cell x itself: when it stores a direction opp(i) that runs into the wall,
// it also puts what the wall returns (its own population with the wall's
// terms) where its next step will look for direction i. Every step then loads
// alike, and only cells at a wall store more. The outermost cells of the
// region read slots that hold nothing valid; what they compute reaches one
// cell further in each step and never an output cell.
//
// A thread updates two cells of a column at once, (x, r) and (x, r + 1), as one
// float2 pair: consecutive lanes then touch consecutive words of a row and no
// x shift needs a shuffle. Rows are split by parity into two halves of each
// plane, so that pair u of a step lies at word u of its half whatever RX is:
// flattened indexing leaves no lane idle at a row's end and no bank conflict.
// FP16 storage keeps its values in shared memory as the FP32 images of the
// rounded ones, so a step gives the bits it gives through global memory.
//
// Regions arrive through a tensor map, one bulk copy per row parity: per-thread
// 16-byte copies and one bulk copy per row kept the load/store unit or the copy
// engine busy for as long as the steps took (82 and 74 us a step at 4096 x 2048
// cells, the tensor map 66). FP16 halves land where the FP32 planes will be and
// are expanded in place through registers (per-thread loads and conversions
// instead: 27.2 us a step at 2048 x 1024, expanded copies 21.6, 20.2 with
// regions of 40 x 32). The blocks of an SM are small enough
// that three or four are resident: one copies while others compute. Tried
// without gain: pulling the first step from global memory directly (86 us), 2
// blocks of 72 x 26 cells (64), 288 to 448 threads (66: each thread sets up a
// step's constants for fewer pairs), one block per SM of 72 x 52 (92).
//
// Bound: the shared-memory pipe and the FP32 pipe together. A pair's step is 28
// loads, 28 stores (1.07 cycles each per warp and SM) and 101 packed operations
// (0.56 to 0.81 cycles); alone they run at 0.75 cells per cycle and SM, in
// place at 0.66. Small lattices are bound by the latency of a step (about 1300
// cycles) and of a launch. Measured, us per step, one step per launch -> this:
// FP32 4096 x 2048 138 -> 60, 1024^2 22 -> 11, 600^2 7.0 -> 5.1, 128^2 5.5 ->
// 1.4, 64^2 5.9 -> 1.2; with the D2Q9 temperature model 177 -> 88 at 4096 x
// 2048; FP16 2048 x 1024 24.5 -> 20.2, 1024^2 14.1 -> 12.0, 600^2 9.1 -> 5.7,
// 128^2 5.8 -> 1.5.
#pragma once

#include <cuda.h>

#include "nomrt_kernels.cuh"
#include "step_tma.cuh"

namespace nomrt {

constexpr int kTileWalls = 15;  // walls whose constants a block keeps in shared memory
constexpr int kTileWallWords = kWallFloats;

template <int TQ, int RX, int RY>
struct TileLayout {
    static_assert(RY % 2 == 0 && RX % 4 == 0, "rows are updated in pairs and copied in 16-byte pieces");
    static constexpr int NQ = 9 + TQ;
    static constexpr int PS = RX * RY / 2;  // cells of one row parity: words per plane of a half
    // words from one half's planes to the other's: each half is a dense box of the source's tensor map, on a
    // 128-byte boundary. The region's corner cells run one word over their plane's ends, into slots of the
    // neighbouring plane that no valid cell reads (the word before plane q's first is plane q - 1's last cell,
    // the word after its last plane q + 1's first cell; the planes reached so are e = 0, +-e_y ones or a
    // first row's)
    static constexpr int HS = (NQ * PS + 31) / 32 * 32;
    static constexpr int kHead = 32;        // words before the planes: the copies' barrier
    // FP16: the box a half arrives in (bytes), wide enough to start on a multiple of 8 cells
    static constexpr int kHalfCols = RX + 8;
    static constexpr int kHalfBox = NQ * (RY / 2) * kHalfCols * 2;
    static constexpr int kHalfStride = (kHalfBox + 127) / 128 * 128;
    static_assert(2 * kHalfStride <= 8 * HS, "the copied halves lie where the planes will");
    // the maps (bytes): one half after the other, with guard bytes around each
    static constexpr int kGuard = 4;
    static constexpr int MS = PS + kGuard;
    static constexpr int kMapBytes = 2 * MS + kGuard;
    static constexpr size_t bytes() {
        return 4 * (size_t)(kHead + 2 * HS + (kTileWalls + 1) * kTileWallWords) + 2 * kMapBytes;
    }
    // word / map byte of cell (x + dx, row) relative to pair index u: half `par`, pair rows dj further on
    static constexpr int at(int par, int dj, int dx) { return par * HS + dj * RX + dx; }
    static constexpr int map(int par, int dj, int dx) { return kGuard + par * MS + dj * RX + dx; }
};

__device__ constexpr int kTileEx[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
__device__ constexpr int kTileEy[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
__device__ constexpr int kTileOpp[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};

// The values two cells' populations have after one trip through the storage.
template <typename S>
__device__ __forceinline__ float2 stored(float2 v) {
    if constexpr (sizeof(S) == 2) return __half22float2(__float22half2_rn(v));
    else return v;
}

// A coordinate of the region on a periodic axis.
__device__ __forceinline__ int tile_wrap(int v, int n) {
    if (v >= 0 && v < n) return v;
    v %= n;
    return v < 0 ? v + n : v;
}

// The lattice's walls, known to the host: how many, and whether any has a Ladd term.
struct TileWalls {
    int n, moving;
};

// Wall constants (WallDev::f) in shared memory. Entry 0 (no wall) returns a population unchanged.
struct TileWall {
    const float *tab;  // kTileWallWords per wall
    bool moving;       // some wall has a Ladd term
    __device__ __forceinline__ float cf(int w, int i) const { return tab[w * kTileWallWords + i]; }
    __device__ __forceinline__ float tsgn(int w) const { return tab[w * kTileWallWords + 9]; }
    template <int TQ>
    __device__ __forceinline__ float tb(int w, int i) const {
        return tab[w * kTileWallWords + (TQ == 9 ? 11 + i : 10)];
    }
};

// Whether link i is set in a link-map byte of a fluid cell.
__device__ __forceinline__ bool tile_link(unsigned m, int i) { return (m >> (i - 1)) & 1u; }

// The link map and the wall ids of the region's solid cells into `maps` (4 cells
// per copy; cells off the lattice count as solid). Returns whether any cell of
// this thread has a link or is solid.
template <int TQ, int RX, int RY, int T>
__device__ __forceinline__ bool tile_maps(const Geom &g, uint8_t *maps, int gx0, int gy0) {
    using Lay = TileLayout<TQ, RX, RY>;
    constexpr int N = RX / 4 * RY, ROUNDS = (N + T - 1) / T;
    uint32_t m[ROUNDS], any = 0;
    int at[ROUNDS];  // first cell of the four, -1: not four cells of one row of the lattice
#pragma unroll
    for (int k = 0; k < ROUNDS; ++k) {
        const int c = (int)threadIdx.x + k * T;
        const int row = c / (RX / 4), x = (c - row * (RX / 4)) * 4;
        const int gx = gx0 + x;
        int gy = gy0 + row;
        if (g.py) gy = tile_wrap(gy, g.ny);
        const bool in = c < N && gy >= 0 && gy < g.ny && gx >= 0 && gx + 4 <= (g.px ? g.nx : g.pitch);
        at[k] = in ? gy * g.pitch + gx : -1;
        m[k] = in && NOMRT_OK(g, g.mask + at[k], 4, 60) ? __ldg(reinterpret_cast<const uint32_t *>(g.mask + at[k]))
                                                        : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int k = 0; k < ROUNDS; ++k) {
        const int c = (int)threadIdx.x + k * T;
        if (c >= N) break;
        const int row = c / (RX / 4), x = (c - row * (RX / 4)) * 4;
        uint32_t w = 0;
        if (at[k] >= 0) {
            if (m[k] != 0u && NOMRT_OK(g, g.flags + at[k], 4, 60))
                w = __ldg(reinterpret_cast<const uint32_t *>(g.flags + at[k]));
        } else if (g.px) {
            int gy = gy0 + row;
            if (g.py) gy = tile_wrap(gy, g.ny);
            if (gy >= 0 && gy < g.ny) {
                m[k] = 0;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int o = gy * g.pitch + tile_wrap(gx0 + x + e, g.nx);
                    if (NOMRT_OK(g, g.mask + o, 1, 60)) m[k] |= (uint32_t)__ldg(g.mask + o) << (8 * e);
                    if (NOMRT_OK(g, g.flags + o, 1, 60)) w |= (uint32_t)__ldg(g.flags + o) << (8 * e);
                }
            }
        }
        any |= m[k];
        const int to = Lay::map(row & 1, row >> 1, x);
        *reinterpret_cast<uint32_t *>(maps + to) = m[k];
        *reinterpret_cast<uint32_t *>(maps + Lay::kMapBytes + to) = w;
    }
    return any != 0;
}

// One half of the region (every second row, from lattice row gy) through the
// source buffer's tensor map: x, row pair, row parity, plane. Rows and columns
// off the lattice arrive as zeros or as the padding's values.
__device__ __forceinline__ void tile_copy_half(void *to, const CUtensorMap *map, int gx, int gy, uint64_t *bar) {
    const int par = gy & 1;
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
        "[%2];" ::"r"(smem_u32(to)),
        "l"(map), "r"(smem_u32(bar)), "r"(gx), "r"((gy - par) / 2), "r"(par), "r"(0)
        : "memory");
}

// FP16: the two halves as copied to the start of `pop`, whose first cell lies
// `shift` cells (0 or 4) before the region's, to their FP32 images in place:
// every thread holds its cells in registers while all are read.
template <int TQ, int RX, int RY, int T>
__device__ __forceinline__ void tile_expand(float *pop, int shift) {
    using Lay = TileLayout<TQ, RX, RY>;
    constexpr int ROW = Lay::kHalfCols / 4, U = Lay::NQ * (RY / 2) * ROW, ROUNDS = (2 * U + T - 1) / T;
    uint2 v[ROUNDS];
#pragma unroll
    for (int k = 0; k < ROUNDS; ++k) {
        const int n = (int)threadIdx.x + k * T, par = n >= U;
        if (n < 2 * U)
            v[k] = *reinterpret_cast<const uint2 *>(reinterpret_cast<const char *>(pop) + par * Lay::kHalfStride +
                                                    (n - par * U) * 8);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ROUNDS; ++k) {
        const int n = (int)threadIdx.x + k * T, par = n >= U;
        const int row = (n - par * U) / ROW, x = (n - par * U - row * ROW) * 4 - shift;
        if (n >= 2 * U || x < 0 || x >= RX) continue;
        __half2 h[2];
        memcpy(h, &v[k], 8);
        const float2 a = __half22float2(h[0]), b = __half22float2(h[1]);
        *reinterpret_cast<float4 *>(pop + par * Lay::HS + row * RX + x) = make_float4(a.x, a.y, b.x, b.y);
    }
}

// The region's cells [x0, x1) x all rows, cell by cell (periodic axes wrapped).
template <typename S, int TQ, int RX, int RY, int T, typename PA>
__device__ __forceinline__ void tile_load_cells(const PA &pl, const Geom &g, float *pop, int gx0, int gy0, int x0,
                                                int x1) {
    using Lay = TileLayout<TQ, RX, RY>;
    const int cols = x1 - x0;
    if (cols <= 0) return;
    for (int n = (int)threadIdx.x; n < cols * RY; n += T) {
        const int row = n / cols, x = x0 + n - row * cols;
        int gx = gx0 + x, gy = gy0 + row;
        if (g.px) gx = tile_wrap(gx, g.nx);
        if (g.py) gy = tile_wrap(gy, g.ny);
        if (gx < 0 || gx >= g.nx || gy < 0 || gy >= g.ny) continue;
        const unsigned o = (unsigned)(gy * g.pitch + gx);
        float *to = pop + Lay::at(row & 1, row >> 1, x);
        float v[Lay::NQ];
#pragma unroll
        for (int q = 0; q < Lay::NQ; ++q) {
            const S *p = pl.src_at(q) + o;
            v[q] = NOMRT_OK(g, p, sizeof(S), 62) ? Ld<S, true>::one(p) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < Lay::NQ; ++q) to[q * Lay::PS] = v[q];
    }
}

// What a cell at a wall stores besides its own directions: for each link i of
// its byte m, the population that runs into the wall, v(d) with d = opp(i), as
// the wall returns it, in the slot the cell's next step pulls direction i from.
// AHEAD: that step is an odd one, and looks in (x - e_i, i); else in (x, d).
// p: the cell's pair; at(d, dx): the word of row d, column dx around the cell.
template <int TQ, int PS, bool AHEAD, typename V, typename AT, typename MAP>
__device__ __forceinline__ void tile_links(float *p, const uint8_t *flag, const TileWall &W, unsigned m, V v, AT at,
                                           MAP map) {
    // the temperature links' wall terms first: independent look-ups
    float ts[TQ], tb[TQ];
#pragma unroll
    for (int i = 1; i < TQ; ++i) {
        const int d = kTileOpp[i];
        const int w = flag[map(kTileEy[d], kTileEx[d])];
        ts[i] = W.tsgn(w);
        tb[i] = W.tb<TQ>(w, i);
    }
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        const int d = kTileOpp[i];
        const int to = (AHEAD ? i : d) * PS + (AHEAD ? at(kTileEy[d], kTileEx[d]) : at(0, 0));
        float fv = v(d);
        if (W.moving) fv += W.cf(flag[map(kTileEy[d], kTileEx[d])], i);
        if (tile_link(m, i)) p[to] = fv;
        if (i < TQ) {
            const float tv = ts[i] * v(9 + d) + tb[i];
            if (tile_link(m, i)) p[9 * PS + to] = tv;
        }
    }
}

// Step `level` (1-based) of a block's region; PULL: an odd step, OUT: the last
// one; WALLED: some cell of the region is solid or at a wall. (gx0, gy0): the
// lattice cell of the region's first cell; [x0, x1): its output columns (OUT).
template <bool PULL, bool OUT, bool WALLED, typename S, int TQ, bool BGK, int RX, int RY, int T, typename PA>
__device__ __forceinline__ void tile_pass(const PA &pl, const Geom &g, const RatesC<float> &r, float *pop,
                                          const uint8_t *maps, const TileWall &W, int level, int gx0, int gy0, int x0,
                                          int x1) {
    using Lay = TileLayout<TQ, RX, RY>;
    constexpr int PS = Lay::PS;
    // the pairs cover region rows level .. RY - level - 1, from an odd row in odd steps
    constexpr int ROW = PULL ? 1 : 0;
    const int base = (level >> 1) * RX;
    const int cols = OUT ? x1 - x0 : RX;
    const int units = (RY / 2 - level) * cols;
    // word of the row d (-1, 0, 1) of cell c (0: first row, 1: second) at x + dx, relative to u
    auto at = [](int c, int d, int dx) constexpr {
        const int row = ROW + c + d + 2;  // even: the half is its parity, the pair row half of it less one
        return Lay::at(row & 1, (row >> 1) - 1, dx);
    };
    auto map = [](int c, int d, int dx) constexpr {
        const int row = ROW + c + d + 2;
        return Lay::map(row & 1, (row >> 1) - 1, dx);
    };
    for (int n = (int)threadIdx.x; n < units; n += T) {
        // the last step's lanes lie along the output columns alone, so that a warp's stores fill whole lines
        const int j = OUT ? n / cols : 0, x = OUT ? x0 + n - j * cols : 0;
        const int u = OUT ? base + j * RX + x : base + n;
        float *const p = pop + u;
        float2 f[9], t[TQ];
        unsigned ma = 0, mb = 0;
        if constexpr (WALLED) {
            ma = maps[map(0, 0, 0) + u];
            mb = maps[map(1, 0, 0) + u];
        }
#pragma unroll
        for (int i = 0; i < 9 + TQ; ++i) {
            const int d = i < 9 ? i : i - 9;
            const int o = PULL ? i : kTileOpp[d] + (i < 9 ? 0 : 9);
            const float2 v = PULL ? make_float2(p[o * PS + at(0, -kTileEy[d], -kTileEx[d])],
                                                p[o * PS + at(1, -kTileEy[d], -kTileEx[d])])
                                  : make_float2(p[o * PS + at(0, 0, 0)], p[o * PS + at(1, 0, 0)]);
            if (i < 9) f[d] = v;
            else t[d] = v;
        }
        if constexpr (BGK) collide_bgk_x<float2, RatesC<float>, TQ>(r, f, t);
        else collide_x<float2, TQ>(r, f, t);
        const bool fa = ma != (unsigned)kSolid, fb = mb != (unsigned)kSolid;
        if constexpr (OUT) {
            const int gy = gy0 + level + 2 * j;
            const unsigned off = (unsigned)(gy * g.pitch + gx0 + x);
            if (gy < g.ny && fa) {
#pragma unroll
                for (int i = 0; i < 9 + TQ; ++i) {
                    S *q = pl.dst_at(i) + off;
                    if (NOMRT_OK(g, q, sizeof(S), 63)) Store<S>::st(q, i < 9 ? f[i].x : t[i - 9].x);
                }
            }
            if (gy + 1 < g.ny && fb) {
                const unsigned offb = off + (unsigned)g.pitch;
#pragma unroll
                for (int i = 0; i < 9 + TQ; ++i) {
                    S *q = pl.dst_at(i) + offb;
                    if (NOMRT_OK(g, q, sizeof(S), 63)) Store<S>::st(q, i < 9 ? f[i].y : t[i - 9].y);
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = stored<S>(f[i]);
#pragma unroll
            for (int i = 0; i < TQ; ++i) t[i] = stored<S>(t[i]);
#pragma unroll
            for (int i = 0; i < 9 + TQ; ++i) {
                const int d = i < 9 ? i : i - 9;
                const int o = PULL ? kTileOpp[d] + (i < 9 ? 0 : 9) : i;
                const int toa = PULL ? at(0, kTileEy[d], kTileEx[d]) : at(0, 0, 0);
                const int tob = PULL ? at(1, kTileEy[d], kTileEx[d]) : at(1, 0, 0);
                const float2 v = i < 9 ? f[d] : t[d];
                if (fa) p[o * PS + toa] = v.x;
                if (fb) p[o * PS + tob] = v.y;
            }
            if (WALLED && (((ma != 0u) & fa) | ((mb != 0u) & fb))) {
                const uint8_t *const flag = maps + Lay::kMapBytes + u;
                tile_links<TQ, PS, !PULL>(p, flag, W, fa ? ma : 0u, [&](int q) { return q < 9 ? f[q].x : t[q - 9].x; },
                                          [&](int d, int dx) constexpr { return at(0, d, dx); },
                                          [&](int d, int dx) constexpr { return map(0, d, dx); });
                tile_links<TQ, PS, !PULL>(p, flag, W, fb ? mb : 0u, [&](int q) { return q < 9 ? f[q].y : t[q - 9].y; },
                                          [&](int d, int dx) constexpr { return at(1, d, dx); },
                                          [&](int d, int dx) constexpr { return map(1, d, dx); });
            }
        }
    }
}

// All k steps of a region whose populations (and wall links) are in place.
template <bool WALLED, typename S, int TQ, bool BGK, int RX, int RY, int T, typename PA>
__device__ __forceinline__ void tile_passes(const PA &pl, const Geom &g, const RatesC<float> &r, float *pop,
                                            const uint8_t *maps, const TileWall &W, int k, int gx0, int gy0, int x0,
                                            int x1) {
    for (int l = 1;;) {
        if (l == k) {
            tile_pass<true, true, WALLED, S, TQ, BGK, RX, RY, T>(pl, g, r, pop, maps, W, l, gx0, gy0, x0, x1);
            break;
        }
        tile_pass<true, false, WALLED, S, TQ, BGK, RX, RY, T>(pl, g, r, pop, maps, W, l, gx0, gy0, x0, x1);
        __syncthreads();
        if (++l == k) {
            tile_pass<false, true, WALLED, S, TQ, BGK, RX, RY, T>(pl, g, r, pop, maps, W, l, gx0, gy0, x0, x1);
            break;
        }
        tile_pass<false, false, WALLED, S, TQ, BGK, RX, RY, T>(pl, g, r, pop, maps, W, l, gx0, gy0, x0, x1);
        __syncthreads();
        ++l;
    }
}

// Before the first step: the wall links of the whole region, from the
// populations as loaded.
template <int TQ, int RX, int RY, int T>
__device__ __forceinline__ void tile_first_links(float *pop, const uint8_t *maps, const TileWall &W) {
    using Lay = TileLayout<TQ, RX, RY>;
    // pairs of rows (2j + 1, 2j + 2): the rows of the first step's cells
    auto at = [](int c, int d, int dx) constexpr {
        const int row = 1 + c + d + 2;
        return Lay::at(row & 1, (row >> 1) - 1, dx);
    };
    auto map = [](int c, int d, int dx) constexpr {
        const int row = 1 + c + d + 2;
        return Lay::map(row & 1, (row >> 1) - 1, dx);
    };
    for (int u = (int)threadIdx.x; u < (RY / 2 - 1) * RX; u += T) {
        float *const p = pop + u;
        unsigned ma = maps[map(0, 0, 0) + u], mb = maps[map(1, 0, 0) + u];
        if (ma == (unsigned)kSolid) ma = 0;
        if (mb == (unsigned)kSolid) mb = 0;
        if ((ma | mb) == 0u) continue;
        const uint8_t *const flag = maps + Lay::kMapBytes + u;
        tile_links<TQ, Lay::PS, true>(p, flag, W, ma, [&](int q) { return p[q * Lay::PS + at(0, 0, 0)]; },
                                      [&](int d, int dx) constexpr { return at(0, d, dx); },
                                      [&](int d, int dx) constexpr { return map(0, d, dx); });
        tile_links<TQ, Lay::PS, true>(p, flag, W, mb, [&](int q) { return p[q * Lay::PS + at(1, 0, 0)]; },
                                      [&](int d, int dx) constexpr { return at(1, d, dx); },
                                      [&](int d, int dx) constexpr { return map(1, d, dx); });
    }
}

// Columns a launch of k steps reads on the left of its output: k rounded up to a 16-byte copy.
__host__ __device__ constexpr int tile_margin(int k) { return (k + 3) & ~3; }
// Output columns and rows of one tile.
template <int RX>
__host__ __device__ constexpr int tile_cols(int k) { return (RX - tile_margin(k) - k) & ~3; }
template <int RY>
__host__ __device__ constexpr int tile_rows(int k) { return RY - 2 * k; }

// How a launch runs (bits). Early: read what does not change between steps
// before waiting for the previous launch (a grid whose blocks can become
// resident before it ends). Late: report the region's copy as not arrived in time
// (a test of the report): a single FP32 lattice takes the wait of every thread but
// the first as run out; FP16 and batches, which a condition at the wait cost 1-2 %,
// begin with the flag set.
constexpr int kTileEarly = 1, kTileLate = 2;

// Where a late copy is reported: a status word and another (a batch's beside its
// member's), or NULL; and whether this lattice's copies are the late ones. Read
// only where they are needed.
struct TileReport {
    int *status, *also;
    int late;
};

// k steps of the tile whose first output cell is (ox, oy), ox a multiple of 4.
// map: the source buffer's tensor map.
template <typename S, int TQ, bool BGK, int RX, int RY, int T, typename PA>
__device__ __forceinline__ void tile_steps(const PA &pl, const Geom &g, const RatesC<float> &r, TileWalls walls,
                                           const CUtensorMap *map, int k, int ox, int oy, int mode,
                                           const TileReport &rep) {
    using Lay = TileLayout<TQ, RX, RY>;
    extern __shared__ __align__(128) float tile_smem[];
    uint64_t *const bar = reinterpret_cast<uint64_t *>(tile_smem);
    volatile int *const gave_up = reinterpret_cast<int *>(bar + 1);
    float *const pop = tile_smem + Lay::kHead;
    float *const wall_tab = pop + 2 * Lay::HS;
    uint8_t *const maps = reinterpret_cast<uint8_t *>(wall_tab + (kTileWalls + 1) * kTileWallWords);
    const int gx0 = ox - tile_margin(k), gy0 = oy - k;
    const TileWall W{wall_tab, walls.moving != 0};
    // every region but one that wraps along y is copied through the tensor map (a copy starts on 16 bytes)
    const bool boxed = !(g.py && (gy0 < 0 || gy0 + RY > g.ny));
    constexpr bool HALF = sizeof(S) == 2, PRESET = HALF || !std::is_same<PA, Planes<S>>::value;
    static_assert(!HALF || RX % 8 == 0, "a box row is whole 16-byte pieces");
    const int bx0 = HALF ? gx0 & ~7 : gx0;
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_fence_init();
        *gave_up = PRESET && boxed && (mode & kTileLate) != 0 && rep.late != 0;
    }
    const bool early = (mode & kTileEarly) != 0;
    bool any = false;
    auto wall_constants = [&]() {
        for (int n = (int)threadIdx.x; n < (walls.n + 1) * kTileWallWords; n += T) {
            const int w = n / kTileWallWords, e = n - w * kTileWallWords;
            const WallDev *d = g.walls + w;
            if (NOMRT_OK(g, d, sizeof(WallDev), 64)) wall_tab[n] = d->f[e];
        }
        // the wall-id map's guard bytes: the region's corner cells look there
        if (threadIdx.x < 3 * Lay::kGuard)
            maps[Lay::kMapBytes + (threadIdx.x / Lay::kGuard) * Lay::MS + threadIdx.x % Lay::kGuard] = 0;
    };
    if (early) {
        any = tile_maps<TQ, RX, RY, T>(g, maps, gx0, gy0);
        wall_constants();
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (boxed) {
        if (threadIdx.x == 0) {
            constexpr int BX = HALF ? Lay::kHalfCols : RX;
            // bounds-checking build: the box's first and last cells on the lattice
            const int xa = max(bx0, 0), xb = min(bx0 + BX, g.pitch) - 1;
            const int ya = max(gy0, 0), yb = min(gy0 + RY, g.ny) - 1;
            const bool ok = NOMRT_OK(g, pl.src_at(0) + (size_t)ya * g.pitch + xa, sizeof(S), 61) &&
                            NOMRT_OK(g, pl.src_at(Lay::NQ - 1) + (size_t)yb * g.pitch + xb, sizeof(S), 61);
            mbar_arrive_expect_tx(bar, ok ? (uint32_t)(Lay::NQ * RY * BX * sizeof(S)) : 0u);
            if (ok) {
                tile_copy_half(pop, map, bx0, gy0, bar);
                tile_copy_half(reinterpret_cast<char *>(pop) + (HALF ? Lay::kHalfStride : 4 * Lay::HS), map, bx0,
                               gy0 + 1, bar);
            }
        }
    } else {
        tile_load_cells<S, TQ, RX, RY, T>(pl, g, pop, gx0, gy0, 0, RX);
    }
    if (!early) any = tile_maps<TQ, RX, RY, T>(g, maps, gx0, gy0);
    const bool walled = __syncthreads_or(any);  // also: the barrier is initialised
    if (boxed && ((!PRESET && (mode & kTileLate) && rep.late && threadIdx.x != 0) || !mbar_wait_bounded(bar, 0))) *gave_up = 1;
    if (HALF && boxed) {
        tile_expand<TQ, RX, RY, T>(pop, gx0 - bx0);
        __syncthreads();
    }
    // a periodic x: the columns beyond the seam
    const int c1 = (g.nx & ~3) - gx0;
    if (boxed && g.px && (gx0 < 0 || c1 < RX)) {
        tile_load_cells<S, TQ, RX, RY, T>(pl, g, pop, gx0, gy0, 0, min(RX, max(0, -gx0)));
        tile_load_cells<S, TQ, RX, RY, T>(pl, g, pop, gx0, gy0, max(0, min(RX, c1)), RX);
        __syncthreads();
    }
    if (walled) {
        if (!early) {
            wall_constants();
            __syncthreads();
        }
        tile_first_links<TQ, RX, RY, T>(pop, maps, W);
        __syncthreads();
    }
    const int x0 = ox - gx0, x1 = min(x0 + tile_cols<RX>(k), g.nx - gx0);
    if (walled) tile_passes<true, S, TQ, BGK, RX, RY, T>(pl, g, r, pop, maps, W, k, gx0, gy0, x0, x1);
    else tile_passes<false, S, TQ, BGK, RX, RY, T>(pl, g, r, pop, maps, W, k, gx0, gy0, x0, x1);
    // a copy that did not arrive in time (what was stored above is then invalid): reported by every thread that
    // sees the flag, the one that gave up among them, after one more bounded wait so that the copy cannot land
    // in a later block's shared memory
    if (*gave_up) {
        mbar_wait_bounded(bar, 0);
        atomicExch(rep.status, kStatusTimeout);
        if (rep.also) atomicExch(rep.also, kStatusTimeout);
    }
}

template <typename S, int TQ, bool BGK, int RX, int RY, int T, int MINB>
__global__ void __launch_bounds__(T, MINB)
    k_tile(const Planes<S> pl, const Geom g, const RatesC<float> r, const __grid_constant__ CUtensorMap map,
           TileWalls walls, int k, int row0, int mode, int *status) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    tile_steps<S, TQ, BGK, RX, RY, T>(pl, g, r, walls, &map, k, (int)blockIdx.x * tile_cols<RX>(k),
                                      row0 + (int)blockIdx.y * tile_rows<RY>(k), mode,
                                      TileReport{status, nullptr, 1});
}

}  // namespace nomrt
