// fish_tile_f64.cu -- FP64 instantiation of the thread-per-cell sweep kernels
// of small boxes (fish_tile.cuh), compiled without FMA contraction like
// fish_f64.cu.
#include "fish_tile_impl.cuh"

namespace fish {
template cudaError_t tile_fluid<double>(const ColFluidArgs<double> &, bool, bool, int, cudaStream_t);
template cudaError_t tile_ct<double>(const ColCTArgs<double> &, bool, int, cudaStream_t);
}
