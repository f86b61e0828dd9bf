// pa_sweep_l12.cu — the launch shapes of the +-1 sweep at L = 12.
#include "pa_sweep_tile.cuh"

namespace pa {

static const ShapeEntry kShapes12[] = {
    PA_SHAPE(12, 16, 576, 1),
    PA_SHAPE(12, 16, 768, 1),
    PA_SHAPE(12, 8, 384, 2),
};
ShapeList sweep_shapes_12() { return {kShapes12, (int)(sizeof(kShapes12) / sizeof(kShapes12[0]))}; }

}  // namespace pa
