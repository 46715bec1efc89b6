// gridgm_bf16.cu - persistent grid-wide GMRES instantiated for __nv_bfloat16 values.
#include "gridgm.cuh"

namespace gk {
template gk_status solve_grid_gmres<__nv_bfloat16, float>(gk_matrix, const float*, float*, int, double, int32_t,
                                                int, cudaStream_t, SolveOut*, bool);
}
