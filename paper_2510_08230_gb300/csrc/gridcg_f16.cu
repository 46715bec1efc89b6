// gridcg_f16.cu - persistent grid-wide CG instantiated for __half values.
#include "gridcg.cuh"

namespace gk {
template gk_status solve_grid_cg<__half, float>(gk_matrix, const float*, float*, int, double, int32_t,
                                             cudaStream_t, SolveOut*, bool);
}
