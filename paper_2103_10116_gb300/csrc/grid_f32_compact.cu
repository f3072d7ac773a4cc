// grid_f32_compact.cu -- the one-launch solves over the device (grid_solve.cuh), b and x in float, products on float values,
// at most 64 registers per thread.
#include "grid_solve.cuh"

namespace spx {
template int grid_launch<float, float, false, true>(spx_ctx *, const GridArgs &, int, int, int, int);
template int grid_launch<float, float, true, true>(spx_ctx *, const GridArgs &, int, int, int, int);
}
