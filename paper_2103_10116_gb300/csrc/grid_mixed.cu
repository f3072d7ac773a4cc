// grid_mixed.cu -- the one-launch solves over the device (grid_solve.cuh), b and x in double, products on float values.
#include "grid_solve.cuh"

namespace spx {
template int grid_launch<double, float, false, false>(spx_ctx *, const GridArgs &, int, int, int, int);
template int grid_launch<double, float, true, false>(spx_ctx *, const GridArgs &, int, int, int, int);
}
