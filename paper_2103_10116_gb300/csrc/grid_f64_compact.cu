// grid_f64_compact.cu -- the one-launch solves over the device (grid_solve.cuh), b and x in double, products on double values,
// at most 64 registers per thread.
#include "grid_solve.cuh"

namespace spx {
template int grid_launch<double, double, false, true>(spx_ctx *, const GridArgs &, int, int, int, int);
template int grid_launch<double, double, true, true>(spx_ctx *, const GridArgs &, int, int, int, int);
}
