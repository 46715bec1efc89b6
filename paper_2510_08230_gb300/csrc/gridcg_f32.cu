// gridcg_f32.cu - persistent grid-wide CG instantiated for float values.
#include "gridcg.cuh"

namespace gk {
template gk_status solve_grid_cg<float, float>(gk_matrix, const float*, float*, int, double, int32_t,
                                             cudaStream_t, SolveOut*, bool);
}
