// gridcg_bf16.cu - persistent grid-wide CG instantiated for __nv_bfloat16 values.
#include "gridcg.cuh"

namespace gk {
template gk_status solve_grid_cg<__nv_bfloat16, float>(gk_matrix, const float*, float*, int, double, int32_t,
                                             cudaStream_t, SolveOut*, bool);
}
