// Several steps per launch (tile.cuh): FP16 storage, D2Q9 temperature.
#include "tile_launch.cuh"

namespace nomrt {

const TileLaunchers *tile_f16_q9() {
    return TileSet<__half, 9, false, ShapeOf<24, 20, 224, 3>, ShapeOf<24, 24, 288, 2>, ShapeOf<32, 24, 384, 2>,
                   ShapeOf<40, 24, 256, 3>, ShapeOf<40, 32, 320, 2>>::get();
}

const TileLaunchers *tile_f16_q9_bgk() {
    return TileSet<__half, 9, true, ShapeOf<24, 20, 224, 3>, ShapeOf<24, 24, 288, 2>, ShapeOf<32, 24, 384, 2>,
                   ShapeOf<40, 24, 256, 3>, ShapeOf<40, 32, 320, 2>>::get();
}

}  // namespace nomrt
