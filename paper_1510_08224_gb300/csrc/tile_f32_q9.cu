// Several steps per launch (tile.cuh): FP32 storage, D2Q9 temperature.
#include "tile_launch.cuh"

namespace nomrt {

// 40 x 24 cells with 160 threads were picked by the estimate and lost to 256 threads
// (2048 x 1024: 26.0 against 23.9 us a step; 1024^2: 16.1 against 14.7).
const TileLaunchers *tile_f32_q9() {
    return TileSet<float, 9, false, ShapeOf<24, 20, 224, 3>, ShapeOf<24, 24, 288, 2>, ShapeOf<32, 24, 384, 2>,
                   ShapeOf<40, 24, 256, 3>>::get();
}

const TileLaunchers *tile_f32_q9_bgk() {
    return TileSet<float, 9, true, ShapeOf<24, 20, 224, 3>, ShapeOf<24, 24, 288, 2>, ShapeOf<32, 24, 384, 2>,
                   ShapeOf<40, 24, 256, 3>>::get();
}

}  // namespace nomrt
