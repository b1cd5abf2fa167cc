// Several steps per launch (tile.cuh): FP16 storage, MRT collisions, D2Q5 temperature.
#include "tile_launch.cuh"

namespace nomrt {

const TileLaunchers *tile_f16() {
    return TileSet<__half, 5, false, ShapeOf<24, 20, 224, 4>, ShapeOf<32, 20, 288, 4>, ShapeOf<32, 24, 384, 2>,
                   ShapeOf<40, 24, 256, 3>, ShapeOf<40, 24, 128, 4>, ShapeOf<40, 32, 256, 3>,
                   ShapeOf<48, 32, 768, 1>>::get();
}

}  // namespace nomrt
