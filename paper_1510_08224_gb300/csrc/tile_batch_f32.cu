// Several steps per launch of a batch's members (tile_batch.cuh): FP32 storage.
#include "tile_batch.cuh"

namespace nomrt {

const TileBatchLaunchers *tile_batch_f16();

const TileBatchLaunchers *tile_batch_launchers(int storage) {
    if (storage == 2) return tile_batch_f16();
    return TileBatchSet<float, ShapeOf<24, 20, 224, 4>, ShapeOf<32, 20, 288, 4>, ShapeOf<32, 24, 384, 2>,
                        ShapeOf<40, 24, 256, 4>, ShapeOf<40, 24, 128, 4>, ShapeOf<40, 32, 192, 3>>::get();
}

}  // namespace nomrt
