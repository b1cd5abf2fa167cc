// Several steps per launch of every member of a launch group (tile.cuh): one
// block per tile of any member. The members' descriptors, their tensor maps
// included, travel in the launch's parameter block, so that a block's member
// (found by a binary search over the members' first tiles) and the rates shared
// by the group are block-uniform operands.
// Bound as k_tile is. Measured, us per step, one step per launch -> this: 64
// cavities of sides 128 to 1024 434 -> 204 (FP16 350 -> 258; with the members'
// own kernels side by side 448 and 298), 24 of 32 to 128 7.2 -> 4.3 (FP16 13.6 ->
// 5.1), 64 cavities of 300^2 119 -> 57 (FP16 105 -> 71).
#pragma once

#include "tile_launch.cuh"

namespace nomrt {

constexpr int kGroupLats = 64;  // members per launch (the parameter block holds their descriptors)

// The values of the MRT collision (collide_x) that follow from one lattice's nu,
// alpha, g beta, T0 and body force; the rest of RatesC<float> that it reads is
// shared by a launch group.
struct MemberRates {
    float s_nu4, om_nu4, h_nu2, nh_nu, om_a, z_a, hx, hFy0, hg_beta, T_ref;
};

inline MemberRates member_rates(const RatesC<float> &r) {
    return MemberRates{r.s_nu4, r.om_nu4, r.h_nu2, r.nh_nu, r.om_a, r.z_a, r.hx, r.hFy0, r.hg_beta, r.T_ref};
}

__host__ __device__ __forceinline__ void apply_member(RatesC<float> &r, const MemberRates &v) {
    r.s_nu4 = v.s_nu4;
    r.ns_nu4 = -v.s_nu4;
    r.om_nu4 = v.om_nu4;
    r.h_nu2 = v.h_nu2;
    r.nh_nu = v.nh_nu;
    r.om_a = v.om_a;
    r.z_a = v.z_a;
    r.hx = v.hx;
    r.hFy0 = v.hFy0;
    r.hg_beta = v.hg_beta;
    r.T_ref = v.T_ref;
}

// One member in a launch's parameter block.
struct TileMember {
    CUtensorMap map;    // of the source buffer
    Geom g;
    const void *src;    // plane 0 of the source and of the destination buffer
    void *dst;
    unsigned long long plane;  // elements per plane
    MemberRates v;
    TileWalls walls;
    TileReport report;  // the member's status word and the batch's
    int row0;           // first row of the member's tiles
    int tiles_x;        // tiles per row of tiles
};

struct TileGroup {
    RatesC<float> rc;   // rates shared by the group
    int nlats;
    int k;              // steps of this launch
    int mode;           // kTileEarly, kTileLate
    int first[kGroupLats + 1];  // first tile of each member; first[nlats]: tiles of the launch
    TileMember lat[kGroupLats];
};
static_assert(sizeof(TileGroup) <= 32764, "a launch group's descriptors must fit the kernel parameter space");

template <typename S>
struct BasePlanes {
    const S *src;
    S *dst;
    size_t plane;
    __device__ __forceinline__ const S *src_at(int q) const { return src + q * plane; }
    __device__ __forceinline__ S *dst_at(int q) const { return dst + q * plane; }
};

template <typename S, int RX, int RY, int T, int MINB>
__global__ void __launch_bounds__(T, MINB) k_tile_batch(const __grid_constant__ TileGroup P) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int b = (int)blockIdx.x;
    int lo = 0, hi = P.nlats - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (P.first[mid] <= b) lo = mid;
        else hi = mid - 1;
    }
    const TileMember &L = P.lat[lo];
    const int local = b - P.first[lo];
    const int by = local / L.tiles_x, bx = local - by * L.tiles_x;
    const BasePlanes<S> pl{static_cast<const S *>(L.src), static_cast<S *>(L.dst), (size_t)L.plane};
    const Geom g = L.g;
    RatesC<float> r = P.rc;  // shared rates: parameter-bank operands
    apply_member(r, L.v);
    tile_steps<S, 5, false, RX, RY, T>(pl, g, r, L.walls, &L.map, P.k, bx * tile_cols<RX>(P.k),
                                       L.row0 + by * tile_rows<RY>(P.k), P.mode, L.report);
}

// The several-steps-per-launch kernels of a batch (MRT, D2Q5).
struct TileBatchLaunchers {
    // the plan for members on a GPU of `sms` SMs; shape -1: some member cannot, or single steps are faster
    TilePlan (*plan)(const KParams *const *members, int n, int sms);
    cudaError_t (*maps)(const KParams &, int shape, CUtensorMap map[2]);
    // k steps of a group whose members' buffers and maps are set; fills in the tiles
    cudaError_t (*launch)(TileGroup &, int shape, int k, cudaStream_t st);
};

const TileBatchLaunchers *tile_batch_launchers(int storage);

template <typename S, typename... SHAPES>
struct TileBatchSet;

template <typename S, int... RX, int... RY, int... T, int... MINB>
struct TileBatchSet<S, ShapeOf<RX, RY, T, MINB>...> {
    static constexpr int N = sizeof...(RX);
    using One = TileSet<S, 5, false, ShapeOf<RX, RY, T, MINB>...>;
    static TilePlan plan(const KParams *const *members, int n, int sms) {
        return choose_tile(members, n, true, 14, (int)sizeof(S), One::shapes(), N, sms);
    }
    static cudaError_t maps(const KParams &p, int shape, CUtensorMap map[2]) { return One::maps(p, shape, map); }
    static cudaError_t launch(TileGroup &G, int shape, int k, cudaStream_t st) {
        using Kernel = void (*)(const TileGroup);
        static const Kernel kernels[N] = {k_tile_batch<S, RX, RY, T, MINB>...};
        static std::atomic<bool> ready[N][kMaxDevices];
        if (shape < 0 || shape >= N) return cudaErrorInvalidValue;
        const TileShape &s = One::shapes()[shape];
        int dev = 0;
        cudaError_t e = tile_ready(kernels[shape], ready[shape], &dev);
        if (e != cudaSuccess) return e;
        const int sms = tile_sms(dev);
        const int tx = shape_cols(s, k), ty = shape_rows(s, k);
        if (tx < 4 || ty < 2) return cudaErrorInvalidValue;
        long long at = 0;
        for (int m = 0; m < G.nlats; ++m) {
            const Geom &g = G.lat[m].g;
            const int rows = g.py ? g.ny : g.ny - 2, cols = g.px ? g.nx : g.nx - 1;
            G.lat[m].tiles_x = std::max(1, (cols + tx - 1) / tx);
            G.first[m] = (int)at;
            at += (long long)G.lat[m].tiles_x * std::max(0, (rows + ty - 1) / ty);
            if (at > 0x7FFFFFFF) return cudaErrorInvalidValue;
        }
        G.first[G.nlats] = (int)at;
        if (at == 0) return cudaSuccess;
        G.k = k;
        G.mode = at <= (long long)sms * s.per_sm ? kTileEarly : 0;
        for (int m = 0; m < G.nlats; ++m)
            if (G.lat[m].report.late) G.mode |= kTileLate;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)at);
        cfg.blockDim = dim3(s.threads);
        cfg.dynamicSmemBytes = tile_smem_bytes(s, at, sms);
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kernels[shape], G);
    }
    static const TileBatchLaunchers *get() {
        static const TileBatchLaunchers L = {&plan, &maps, &launch};
        return &L;
    }
};

}  // namespace nomrt
