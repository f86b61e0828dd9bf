// pa_sweep_l6.cu — the launch shapes of the +-1 sweep at L = 6.
#include "pa_sweep_tile.cuh"

namespace pa {

static const ShapeEntry kShapes6[] = {
    PA_SHAPE(6, 32, 384, 2),
    PA_SHAPE(6, 32, 192, 4),
    PA_SHAPE(6, 32, 576, 1),
    PA_SHAPE(6, 8, 288, 2),
};
ShapeList sweep_shapes_6() { return {kShapes6, (int)(sizeof(kShapes6) / sizeof(kShapes6[0]))}; }

}  // namespace pa
