// pa_sweep_l2.cu — the launch shapes of the +-1 sweep at L = 2, 4.
#include "pa_sweep_tile.cuh"

namespace pa {

static const ShapeEntry kShapes2[] = {
    PA_SHAPE(2, 32, 128, 1),
    PA_SHAPE(2, 32, 64, 2),
};
ShapeList sweep_shapes_2() { return {kShapes2, (int)(sizeof(kShapes2) / sizeof(kShapes2[0]))}; }

static const ShapeEntry kShapes4[] = {
    PA_SHAPE(4, 32, 256, 2),
    PA_SHAPE(4, 32, 128, 4),
    PA_SHAPE(4, 32, 512, 1),
    PA_SHAPE(4, 8, 128, 4),
};
ShapeList sweep_shapes_4() { return {kShapes4, (int)(sizeof(kShapes4) / sizeof(kShapes4[0]))}; }

}  // namespace pa
