// pa_sweep_l8.cu — the launch shapes of the +-1 sweep at L = 8.
#include "pa_sweep_tile.cuh"

namespace pa {

static const ShapeEntry kShapes8[] = {
    PA_SHAPE(8, 32, 256, 2),
    PA_SHAPE(8, 32, 512, 1),
    PA_SHAPE(8, 16, 256, 2),
    PA_SHAPE(8, 8, 256, 2),
};
ShapeList sweep_shapes_8() { return {kShapes8, (int)(sizeof(kShapes8) / sizeof(kShapes8[0]))}; }

}  // namespace pa
