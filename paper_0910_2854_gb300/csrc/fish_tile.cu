// fish_tile.cu -- launchers of the FP64 thread-per-cell sweep kernels of small
// boxes (fish_tile.cuh), compiled without FMA contraction like fish_f64.cu.
#include "fish_tile.cuh"

namespace fish {

// dynamic shared memory beyond 48 KB has to be asked for
template <class K> static cudaError_t tile_allow(K kernel, size_t bytes)
{
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <bool HSE, int GM, int LIM, bool FT1, bool NU>
static cudaError_t fluid_run(const ColFluidArgs<double> &A, int len, cudaStream_t s)
{
    const auto kernel = fluid_tile_kernel<HSE, GM, LIM, FT1, NU>;
    const size_t bytes = tile_fluid_smem<HSE, LIM < 0 && !HSE>(len);
    const cudaError_t e = tile_allow(kernel, bytes);
    if (e != cudaSuccess) return e;
    const long long cols = (long long)A.nf * A.no;
    const dim3 grid((unsigned)((cols + 31) / 32), (unsigned)((A.n + len - 1) / len));
    kernel<<<grid, 32 * (len + 6), bytes, s>>>(A, len);
    return cudaGetLastError();
}

template <bool HSE, int GM, bool FT1, bool NU>
static cudaError_t fluid_lim(const ColFluidArgs<double> &A, int len, cudaStream_t s)
{
    // (the limiter at compile time for the plain sweeps, as in the marches)
    if constexpr (!HSE && GM == 0 && !NU) {
        if (A.lim == LIM_VANLEER) return fluid_run<HSE, GM, LIM_VANLEER, FT1, NU>(A, len, s);
    }
    return fluid_run<HSE, GM, -1, FT1, NU>(A, len, s);
}

template <bool FT1> static cudaError_t fluid_ft(const ColFluidArgs<double> &A, bool hse, int len, cudaStream_t s)
{
    if (A.cfl_min || (A.sg && (hse || A.wd))) return cudaErrorInvalidValue;
    if (A.wd) {
        if (hse) return A.phi ? fluid_lim<true, 1, FT1, true>(A, len, s) : fluid_lim<true, 0, FT1, true>(A, len, s);
        return A.phi ? fluid_lim<false, 1, FT1, true>(A, len, s) : fluid_lim<false, 0, FT1, true>(A, len, s);
    }
    if (hse) return A.phi ? fluid_lim<true, 1, FT1, false>(A, len, s) : fluid_lim<true, 0, FT1, false>(A, len, s);
    if (A.phi && A.sg) return fluid_lim<false, 2, FT1, false>(A, len, s);
    return A.phi ? fluid_lim<false, 1, FT1, false>(A, len, s) : fluid_lim<false, 0, FT1, false>(A, len, s);
}

cudaError_t tile_fluid(const ColFluidArgs<double> &A, bool hse, bool ft1, int len, cudaStream_t s)
{
    return ft1 ? fluid_ft<true>(A, hse, len, s) : fluid_ft<false>(A, hse, len, s);
}

template <int LIM, bool FT1, bool NU> static cudaError_t ct_run(const ColCTArgs<double> &A, int len, cudaStream_t s)
{
    const dim3 grid((unsigned)((long long)((A.nf + 30) / 31) * A.no), (unsigned)((A.n + len - 1) / len));
    static_assert(tile_ct_smem(TILE_MAX) <= 48 * 1024, "no shared memory to ask for");
    ct_tile_kernel<LIM, FT1, NU><<<grid, 32 * (len + 8), tile_ct_smem(len), s>>>(A, len);
    return cudaGetLastError();
}

template <bool FT1> static cudaError_t ct_ft(const ColCTArgs<double> &A, int len, cudaStream_t s)
{
    if (A.wd) return ct_run<-1, FT1, true>(A, len, s);
    if (A.lim == LIM_VANLEER) return ct_run<LIM_VANLEER, FT1, false>(A, len, s);
    return ct_run<-1, FT1, false>(A, len, s);
}

cudaError_t tile_ct(const ColCTArgs<double> &A, bool ft1, int len, cudaStream_t s)
{
    return ft1 ? ct_ft<true>(A, len, s) : ct_ft<false>(A, len, s);
}

}  // namespace fish
