// gridgm_f32.cu - persistent grid-wide GMRES instantiated for float values.
#include "gridgm.cuh"

namespace gk {
template gk_status solve_grid_gmres<float, float>(gk_matrix, const float*, float*, int, double, int32_t,
                                                int, cudaStream_t, SolveOut*, bool);
}
