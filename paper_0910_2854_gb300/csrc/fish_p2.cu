// fish_p2.cu -- the two-column sweep kernels: FP32 pencils advanced in pairs
// with the packed FP32x2 instructions of sm_100+ (compiled with the FP32
// flags of fish_f32.cu).  This unit holds the dispatcher and the Van Leer
// kernels; fish_p2_mm.cu and fish_p2_hy.cu the minmod and hybrid ones,
// fish_p2_hse.cu those with the hydrostatic correction, so they compile in
// parallel.
#include "fish_col_impl.cuh"

namespace fish {
#define FISH_P2_OTHER(LIMV)                                                                                     \
    extern template cudaError_t col_fluid_launch<P2, false, 0, LIMV, true, false>(const ColFluidArgs<float> &,  \
                                                                                 cudaStream_t);                \
    extern template cudaError_t col_fluid_launch<P2, false, 1, LIMV, true, false>(const ColFluidArgs<float> &,  \
                                                                                 cudaStream_t);                \
    extern template cudaError_t col_fluid_launch<P2, false, 2, LIMV, true, false>(const ColFluidArgs<float> &,  \
                                                                                 cudaStream_t);
FISH_P2_OTHER(LIM_MINMOD)
FISH_P2_OTHER(LIM_HYBRID)
#undef FISH_P2_OTHER
#define FISH_P2_HSE(GRAV, LIMV)                                                                                 \
    extern template cudaError_t col_fluid_launch<P2, true, GRAV, LIMV, true, false>(const ColFluidArgs<float> &, \
                                                                                   cudaStream_t);
FISH_P2_HSE(0, LIM_VANLEER)
FISH_P2_HSE(1, LIM_VANLEER)
FISH_P2_HSE(0, LIM_MINMOD)
FISH_P2_HSE(1, LIM_MINMOD)
#undef FISH_P2_HSE
template cudaError_t col_fluid<P2>(const ColFluidArgs<float> &, bool, bool, cudaStream_t);
#ifdef FISH_CT_PAIRS
template cudaError_t col_ct<P2>(const ColCTArgs<float> &, bool, cudaStream_t);
#endif
}
