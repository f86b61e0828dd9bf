// pa_sweep_l14.cu — the launch shapes of the +-1 sweep at L = 14, 16.
#include "pa_sweep_tile.cuh"

namespace pa {

static const ShapeEntry kShapes14[] = {
    PA_SHAPE(14, 8, 784, 1),
    PA_SHAPE(14, 8, 224, 1),
    PA_SHAPE(14, 4, 392, 1),
};
ShapeList sweep_shapes_14() { return {kShapes14, (int)(sizeof(kShapes14) / sizeof(kShapes14[0]))}; }

static const ShapeEntry kShapes16[] = {
    PA_SHAPE(16, 4, 512, 1),
    PA_SHAPE(16, 4, 256, 1),
};
ShapeList sweep_shapes_16() { return {kShapes16, (int)(sizeof(kShapes16) / sizeof(kShapes16[0]))}; }

}  // namespace pa
