// gridgm_f64.cu - persistent grid-wide GMRES instantiated for double values.
#include "gridgm.cuh"

namespace gk {
template gk_status solve_grid_gmres<double, double>(gk_matrix, const double*, double*, int, double, int32_t,
                                                int, cudaStream_t, SolveOut*, bool);
}
