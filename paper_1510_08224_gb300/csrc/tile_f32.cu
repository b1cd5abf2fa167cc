// Several steps per launch (tile.cuh): FP32 storage, MRT collisions, D2Q5 temperature.
#include "tile_launch.cuh"

namespace nomrt {

const TileLaunchers *tile_f32() {
    return TileSet<float, 5, false, ShapeOf<24, 20, 224, 4>, ShapeOf<32, 20, 288, 4>, ShapeOf<32, 24, 384, 2>,
                   ShapeOf<40, 24, 256, 4>, ShapeOf<40, 24, 128, 4>, ShapeOf<40, 32, 192, 3>,
                   ShapeOf<48, 32, 768, 1>>::get();
}

const TileLaunchers *tile_f32_bgk();
const TileLaunchers *tile_f32_q9();
const TileLaunchers *tile_f32_q9_bgk();
const TileLaunchers *tile_f16();
const TileLaunchers *tile_f16_bgk();
const TileLaunchers *tile_f16_q9();
const TileLaunchers *tile_f16_q9_bgk();

const TileLaunchers *tile_launchers(int storage, int tq, int bgk) {
    if (storage == 1)
        return tq == 9 ? (bgk ? tile_f32_q9_bgk() : tile_f32_q9()) : (bgk ? tile_f32_bgk() : tile_f32());
    if (storage == 2)
        return tq == 9 ? (bgk ? tile_f16_q9_bgk() : tile_f16_q9()) : (bgk ? tile_f16_bgk() : tile_f16());
    return nullptr;
}

}  // namespace nomrt
