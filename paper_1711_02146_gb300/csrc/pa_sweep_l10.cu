// pa_sweep_l10.cu — the launch shapes of the +-1 sweep at L = 10.
#include "pa_sweep_tile.cuh"

namespace pa {

static const ShapeEntry kShapes10[] = {
    PA_SHAPE(10, 32, 640, 1),
    PA_SHAPE(10, 16, 320, 2),
    PA_SHAPE(10, 8, 160, 3),
};
ShapeList sweep_shapes_10() { return {kShapes10, (int)(sizeof(kShapes10) / sizeof(kShapes10[0]))}; }

}  // namespace pa
