// gridgm_f16.cu - persistent grid-wide GMRES instantiated for __half values.
#include "gridgm.cuh"

namespace gk {
template gk_status solve_grid_gmres<__half, float>(gk_matrix, const float*, float*, int, double, int32_t,
                                                int, cudaStream_t, SolveOut*, bool);
}
