// Launchers of the several-steps-per-launch kernels (tile.cuh): the tile shapes,
// the choice of shape and steps per launch for a lattice, tensor maps.
#pragma once

#include <algorithm>
#include <atomic>
#include <cmath>

#include "tile.cuh"

namespace nomrt {

struct TileShape {
    int rx, ry, threads, per_sm;  // region, block, resident blocks asked of ptxas
    size_t smem;
};

// Output columns and rows of a tile of a shape in a launch of k steps.
inline int shape_cols(const TileShape &s, int k) { return (s.rx - tile_margin(k) - k) & ~3; }
inline int shape_rows(const TileShape &s, int k) { return s.ry - 2 * k; }

// The rows and columns a lattice's tiles cover: a non-periodic axis ends in a
// frame of cells that are not updated.
struct TileCover {
    int row0, rows, cols;
};
inline TileCover tile_cover(const KParams &p) {
    return TileCover{p.py ? 0 : 1, p.py ? p.ny : p.ny - 2, p.px ? p.nx : p.nx - 1};
}

// Estimated cycles of one launch of k steps, all its tiles. Up to two waves of
// resident blocks: a launch's own cost, and per wave the steps, each at least
// its latency (one pass of a thread over its pairs, a barrier) or what the SM's
// blocks take of its pipes when they start together. Many waves: the blocks are
// out of step with one another and with the copies, so the slower of the pipes
// and the way to HBM (or L2, for a lattice that fits it) sets the pace. The
// constants are a least-squares fit to 551 timed launches of 16 shapes with 2
// to 8 steps on lattices of 64^2 to 4096 x 2048 cells and on batches of 24 to
// 64 cavities (rms error 13 %); the shape and steps it picks run within 2 % of
// the fastest of them but for 180^2 cells (19 %). Fitted in FP32, before the next
// block's prefetch went and before FP16's regions came through the tensor map:
// FP16's conversions are not in it.
inline double tile_cycles(const TileShape &s, int k, long long tiles, int nq, double cell_bytes, bool fits_l2,
                          int sms) {
    constexpr double kLaunch = 11600, kRound = 1.18;
    constexpr double kTogether[4] = {153, 141, 142, 125};  // cycles per 32 pairs with 1..4 blocks on the SM
    constexpr double kBlock = 3640, kWarpStep = 8.1, kHbm = 21.2;  // many waves; bytes per cycle and SM
    // a pair's cost goes with its populations (fitted with 14)
    const double scale = nq / 14.0, kLatency = 920 * scale, kPairWarp = 80.3 * scale;
    double pair_warps = 0;
    const int cols = shape_cols(s, k), rows = shape_rows(s, k);
    auto pairs = [&](int l) { return (s.ry / 2 - l) * (l < k ? s.rx : cols); };
    for (int l = 1; l <= k; ++l) pair_warps += (pairs(l) + 31) / 32;
    auto wave = [&](int n) {
        double t = 0;
        for (int l = 1; l <= k; ++l) {
            const int rounds = (pairs(l) + s.threads - 1) / s.threads;
            t += std::max(kLatency * (1 + kRound * (rounds - 1)),
                          n * ((pairs(l) + 31) / 32) * scale * kTogether[std::min(n, 4) - 1]);
        }
        return t;
    };
    const long long slots = (long long)sms * s.per_sm;
    const long long full = tiles / slots, rest = tiles % slots;
    if (full <= 1)
        return kLaunch + (double)full * wave(s.per_sm) + (rest ? wave((int)((rest + sms - 1) / sms)) : 0.0);
    const double steps = kBlock + s.per_sm * (pair_warps * kPairWarp + k * (s.threads / 32) * kWarpStep);
    const double bytes = s.per_sm * cols * rows * cell_bytes / (fits_l2 ? 3 * kHbm : kHbm);
    return kLaunch + std::pow(std::pow(steps, 7.5) + std::pow(bytes, 7.5), 1 / 7.5) * ((double)tiles / (double)slots) +
           0.5 * wave(s.per_sm);
}

// Estimated cycles of a single step of the lattices in one launch, as graphs
// replay it: the populations of the rows with cells, read and written, and
// those of wall rows, written, at HBM's rate (FP16 in whole blocks of 512 cells,
// whose conversions take as long in a block that is not full); at least a
// block's own cost per row of 512 cells; and a launch's latency.
inline double single_cycles(const KParams *const *lats, int n, int nq, int elem, int sms) {
    constexpr double kHbm = 21.2, kRowBlock = 315;  // bytes and cycles per SM
    const double launch = elem == 4 ? 5200 : 6200, least = elem == 4 ? 11400 : 9900;
    double bytes = 0, blocks = 0;
    for (int m = 0; m < n; ++m) {
        const KParams &p = *lats[m];
        const int rows = tile_cover(p).rows, segments = (p.pitch + 511) / 512;
        if (rows <= 0) continue;
        bytes += 2.0 * nq * elem * (elem == 4 ? p.nx : 512.0 * segments) * (rows + 0.5 * (p.ny - rows));
        blocks += (double)p.ny * segments;
    }
    return std::max(least, launch + std::max(bytes / (kHbm * sms), blocks * kRowBlock / sms));
}

// The share of a single step's estimate that a step of the tiles may take. A
// tile does the work of all its rows whatever the lattice has, so wide lattices
// of few rows are faster stepped singly; the line lies where 150 timed pairs
// cross (145 on the faster side, the worst at 1.25 times the other), and no
// lattice of 0.15 to 7 times as many columns as rows comes near it. FP16 tiles
// take their estimate's 1.2 to 1.7 times in one or two rows of tiles. Measured,
// us a step, tiles / single steps (and the estimates' ratio): FP32 262144 columns
// x 14 rows 46 / 67 (0.50), x 6 39 / 33 (0.99), x 4 38 / 22 (1.34), 1048576 x 4 146 / 91
// (1.38), 4194304 x 2 570 / 211 (2.30), 20000 x 4 4.1 / 6.1 (0.70), nine temperature
// populations 60000 x 10 16.6 / 16.3 (0.73), x 8 15.0 / 12.0 (0.81); FP16 65536 x 32
// 24.5 / 26.1 (0.87), 60000 x 20 19.4 / 12.7 (0.95), x 4 11.7 / 5.9 (1.58), 262144 x 4 45 /
// 14 (2.35), but nine populations 485 x 870 7.9 / 9.5 (0.98).
inline double tile_share(const KParams *const *lats, int n, int elem) {
    if (elem == 4) return 0.76;
    for (int m = 0; m < n; ++m)
        if (tile_cover(*lats[m]).rows > 32) return 1.0;
    return 0.89;
}

constexpr int kTileMaxSteps = 8;
constexpr double kL2Bytes = 100e6;  // what of the 129 MB L2 two buffers can count on

// Cells up to which a run of `steps` steps of one FP16 lattice takes the tiles. A
// block keeps FP32 images, so it computes as long as an FP32 lattice's and rounds
// every population besides, while single steps are bound by HBM at half the
// bytes. Measured, us per step, single -> several steps per launch: 1024^2 14.1
// -> 12.0, 2048 x 1024 24.5 -> 20.2, 2500^2 59.8 -> 57.5, 4096 x 2048 72.6 ->
// 74.3; with nine temperature populations 1777^2 49.3 -> 43.5, 4096 x 1024 53.9
// -> 55.1. Runs of two steps: 1402^2 26.3 -> 23.4, 2050^2 46.0 -> 44.5, 2450^2 59.9
// -> 60.8; with nine 802^2 13.9 -> 13.7, 1026^2 19.2 -> 19.9. A batch's single
// steps are further from that bound (64 lattices of 300^2: 105 -> 71) and have no
// such limit.
inline double tile_most_f16(int nq, int steps) {
    if (nq <= 14) return steps == 2 ? 5.0e6 : 6.5e6;
    return steps == 2 ? 0.9e6 : 4.0e6;
}

// The shape and steps per launch with the least estimated time per step, or shape
// -1 where single steps are estimated faster. Lattices with node-based walls or more walls than a block keeps step once per
// launch. FP16: several regions of 32 rows per SM only where they make more than
// two waves; below, the estimate misjudges them (600^2: 6.1 us a step against
// 5.7; 256^2 with nine temperature populations 3.3 against 3.0; but 1111 x 333
// 7.8 against 8.2).
inline TilePlan choose_tile(const KParams *const *lats, int n, bool batch, int nq, int elem, const TileShape *shapes,
                            int n_shapes, int sms) {
    TilePlan best;
    double least = 0, cells = 0;
    if (n < 1 || sms <= 0) return best;
    for (int m = 0; m < n; ++m) {
        const KParams &p = *lats[m];
        const TileCover c = tile_cover(p);
        if (p.n_nee > 0 || p.n_walls > kTileWalls || (!batch && (c.rows <= 0 || c.cols <= 0))) return best;
        cells += (double)p.nx * p.ny;
    }
    if (elem == 2 && !batch && cells > tile_most_f16(nq, kTileMaxSteps)) return best;
    const double cell_bytes = 2.0 * nq * elem;
    const bool fits_l2 = cell_bytes * cells < kL2Bytes;
    // tiles of a launch of k steps (-1: more than a launch can have)
    auto count = [&](const TileShape &s, int k) -> long long {
        const int tx = shape_cols(s, k), ty = shape_rows(s, k);
        long long tiles = 0;
        for (int m = 0; m < n; ++m) {
            const TileCover c = tile_cover(*lats[m]);
            if (c.rows <= 0 || c.cols <= 0) continue;
            const long long gx = (c.cols + tx - 1) / tx, gy = (c.rows + ty - 1) / ty;
            if (!batch && gy > 65535) return -1;  // a lattice alone: the launch grid's y limit
            tiles += gx * gy;
        }
        return tiles > 0x3FFFFFFF ? -1 : tiles;
    };
    for (int i = 0; i < n_shapes; ++i)
        for (int k = 2; k <= kTileMaxSteps; ++k) {
            if (shape_cols(shapes[i], k) < 4 || shape_rows(shapes[i], k) < 2) break;
            const long long tiles = count(shapes[i], k);
            if (tiles < 0) continue;
            if (elem == 2 && shapes[i].ry >= 32 && shapes[i].per_sm > 1 && tiles <= 2LL * sms * shapes[i].per_sm)
                continue;
            const double t = tile_cycles(shapes[i], k, tiles, nq, cell_bytes, fits_l2, sms) / k;
            if (best.shape < 0 || t < least) {
                best.shape = i;
                best.steps = k;
                least = t;
            }
        }
    if (best.shape < 0) return best;
    const double single = single_cycles(lats, n, nq, elem, sms);
    if (least > tile_share(lats, n, elem) * single) return TilePlan{};
    if (elem == 2 && !batch && cells > tile_most_f16(nq, 2)) best.least = 3;
    // launches of one step (two steps that have to end on the buffer they began on): by the same estimates, or
    // up to one wave of tiles, FP16 two, where single steps launched one by one take longer than replayed (24
    // lattices of 32 to 128: 7.7 us a step against 10.2; 8 of 200 to 400, 1.8 waves, FP32 14.8 / 14.4, FP16 14.9
    // / 15.9; 64 of 128 to 1024 FP16 393 / 352; one of 4 x 262144 172 / 250)
    const TileShape &s = shapes[best.shape];
    const long long tiles = count(s, 1);
    best.one = tiles >= 0 && (tiles <= (elem == 2 ? 2LL : 1LL) * sms * s.per_sm ||
                              tile_cycles(s, 1, tiles, nq, cell_bytes, fits_l2, sms) <= 0.76 * single);
    return best;
}

// The tensor map of buffer `buf` for boxes of `cols` x RY cells: x, row pair, row
// parity, plane (for an odd ny the last row pair's second row lies past the
// plane, in the lattice's block; the kernel treats it as off the lattice).
inline cudaError_t make_tile_map(const KParams &p, int buf, int elem, int nq, int cols, int ry, CUtensorMap *map) {
    using Encode = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static std::atomic<void *> entry{nullptr};
    void *fn = entry.load(std::memory_order_acquire);
    if (!fn) {
        cudaDriverEntryPointQueryResult found;
        const cudaError_t e =
            cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found);
        if (e != cudaSuccess) return e;
        if (found != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        entry.store(fn, std::memory_order_release);
    }
    const cuuint64_t row = (cuuint64_t)p.pitch * elem;
    const cuuint64_t dims[4] = {(cuuint64_t)p.pitch, (cuuint64_t)(p.ny + 1) / 2, 2, (cuuint64_t)nq};
    const cuuint64_t strides[3] = {2 * row, row, (cuuint64_t)p.plane * elem};
    const cuuint32_t box[4] = {(cuuint32_t)cols, (cuuint32_t)ry / 2, 1, (cuuint32_t)nq};
    const cuuint32_t one[4] = {1, 1, 1, 1};
    const CUtensorMapDataType type = elem == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    const CUresult r = reinterpret_cast<Encode>(fn)(map, type, 4, p.pop[buf], dims, strides, box, one,
                                                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// SMs of the current device, read once per device (0 if it cannot be read).
inline int tile_sms(int dev) {
    static std::atomic<int> sms[kMaxDevices];
    if (dev < 0 || dev >= kMaxDevices) return 0;
    int n = sms[dev].load(std::memory_order_relaxed);
    if (n == 0 && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess)
        sms[dev].store(n, std::memory_order_relaxed);
    return n;
}

// Dynamic shared memory of a launch of `tiles` blocks: the shape's, or, where
// the grid fits the GPU at n blocks per SM, as much as lets no more than n
// reside, so that the blocks spread over all SMs (as programmatic dependents
// they would otherwise double up on the SMs the previous launch leaves first:
// 64^2 cells, 8 steps per launch, 1.48 against 1.21 us a step).
inline size_t tile_smem_bytes(const TileShape &s, long long tiles, int sms) {
    constexpr size_t kSm = 227 * 1024, kPerBlock = 1024;  // shared memory per SM, and what the system takes per block
    if (sms <= 0) return s.smem;
    const long long n = (tiles + sms - 1) / sms;
    if (n > s.per_sm) return s.smem;
    return std::max(s.smem, (kSm / (size_t)n - kPerBlock - 256) & ~(size_t)1023);
}

template <typename S>
using TileKernel = void (*)(const Planes<S>, const Geom, const RatesC<float>, const CUtensorMap, TileWalls, int, int, int,
                            int *);

// The current device, the kernel's shared-memory limit raised on it once.
template <typename K>
cudaError_t tile_ready(K kern, std::atomic<bool> *ready, int *dev) {
    cudaError_t e = cudaGetDevice(dev);
    if (e != cudaSuccess) return e;
    if (*dev < 0 || *dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (!ready[*dev].load(std::memory_order_acquire)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (e != cudaSuccess) return e;
        ready[*dev].store(true, std::memory_order_release);
    }
    return cudaSuccess;
}

// One launch of k steps.
template <typename S>
cudaError_t launch_tile(TileKernel<S> kern, const TileShape &s, std::atomic<bool> *ready, const KParams &p,
                        const CUtensorMap &map, int src, int k, cudaStream_t st) {
    int dev = 0;
    const cudaError_t e = tile_ready(kern, ready, &dev);
    if (e != cudaSuccess) return e;
    const int sms = tile_sms(dev);
    const TileCover c = tile_cover(p);
    const int tx = shape_cols(s, k), ty = shape_rows(s, k);
    if (tx < 4 || ty < 2) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((c.cols + tx - 1) / tx, (c.rows + ty - 1) / ty);
    cfg.blockDim = dim3(s.threads);
    const long long tiles = (long long)cfg.gridDim.x * cfg.gridDim.y;
    cfg.dynamicSmemBytes = tile_smem_bytes(s, tiles, sms);
    cfg.stream = st;
    // a programmatic dependent of the previous launch (the kernel waits for that grid's
    // completion before it reads a population)
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, make_planes<S>(p, src), make_geom(p), make_rates<float>(p), map,
                              TileWalls{p.n_walls, p.moving}, k, c.row0,
                              (tiles <= (long long)sms * s.per_sm ? kTileEarly : 0) | (p.late ? kTileLate : 0), p.status);
}

// The shapes of one storage, temperature lattice and collision: region columns
// and rows, threads, resident blocks per SM.
template <int RX, int RY, int T, int MINB>
struct ShapeOf {};

template <typename S, int TQ, bool BGK, typename... SHAPES>
struct TileSet;

template <typename S, int TQ, bool BGK, int... RX, int... RY, int... T, int... MINB>
struct TileSet<S, TQ, BGK, ShapeOf<RX, RY, T, MINB>...> {
    static constexpr int N = sizeof...(RX);
    static const TileShape *shapes() {
        static const TileShape s[N] = {TileShape{RX, RY, T, MINB, TileLayout<TQ, RX, RY>::bytes()}...};
        return s;
    }
    static TilePlan plan(const KParams &p, int sms) {
        const KParams *const one = &p;
        return choose_tile(&one, 1, false, 9 + TQ, (int)sizeof(S), shapes(), N, sms);
    }
    static cudaError_t maps(const KParams &p, int shape, CUtensorMap map[2]) {
        if (shape < 0 || shape >= N) return cudaErrorInvalidValue;
        for (int b = 0; b < 2; ++b) {
            const cudaError_t e = make_tile_map(p, b, (int)sizeof(S), 9 + TQ, shapes()[shape].rx + (sizeof(S) == 2 ? 8 : 0),
                                                shapes()[shape].ry, map + b);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    static cudaError_t launch(const KParams &p, int shape, const CUtensorMap &map, int src, int k, cudaStream_t st) {
        static const TileKernel<S> kernels[N] = {k_tile<S, TQ, BGK, RX, RY, T, MINB>...};
        static std::atomic<bool> ready[N][kMaxDevices];
        if (shape < 0 || shape >= N) return cudaErrorInvalidValue;
        return launch_tile<S>(kernels[shape], shapes()[shape], ready[shape], p, map, src, k, st);
    }
    static const TileLaunchers *get() {
        static const TileLaunchers L = {&plan, &maps, &launch};
        return &L;
    }
};

}  // namespace nomrt
