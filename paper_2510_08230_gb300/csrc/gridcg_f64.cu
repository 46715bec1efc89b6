// gridcg_f64.cu - persistent grid-wide CG instantiated for double values.
#include "gridcg.cuh"

namespace gk {
template gk_status solve_grid_cg<double, double>(gk_matrix, const double*, double*, int, double, int32_t,
                                             cudaStream_t, SolveOut*, bool);
}
