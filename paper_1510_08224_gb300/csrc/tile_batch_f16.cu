// Several steps per launch of a batch's members (tile_batch.cuh): FP16 storage.
#include "tile_batch.cuh"

namespace nomrt {

const TileBatchLaunchers *tile_batch_f16() {
    return TileBatchSet<__half, ShapeOf<24, 20, 224, 4>, ShapeOf<32, 20, 288, 4>, ShapeOf<32, 24, 384, 2>,
                        ShapeOf<40, 24, 256, 4>, ShapeOf<40, 24, 128, 4>, ShapeOf<40, 32, 256, 3>>::get();
}

}  // namespace nomrt
