// fish_p2_hse.cu -- the two-column L_d kernels with the hydrostatic correction (see fish_p2.cu).
#include "fish_col_impl.cuh"

namespace fish {
template cudaError_t col_fluid_launch<P2, true, 0, LIM_VANLEER, true, false>(const ColFluidArgs<float> &, cudaStream_t);
template cudaError_t col_fluid_launch<P2, true, 1, LIM_VANLEER, true, false>(const ColFluidArgs<float> &, cudaStream_t);
template cudaError_t col_fluid_launch<P2, true, 0, LIM_MINMOD, true, false>(const ColFluidArgs<float> &, cudaStream_t);
template cudaError_t col_fluid_launch<P2, true, 1, LIM_MINMOD, true, false>(const ColFluidArgs<float> &, cudaStream_t);
}
