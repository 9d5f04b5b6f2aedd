// fish_f64.cu -- FP64 instantiation of the sweep kernels.  Compiled without
// FMA contraction (-fmad=false) so that every operation rounds like a plain
// IEEE double evaluation of the paper's formulas, in the order written.
#include "fish_col_impl.cuh"
#include "fish_launch.cuh"

namespace fish {
// the sweeps whose fast axis is t2 (FT1 = false) compile in fish_f64_t2.cu
#define FISH_F64_T2(HSE, GRAV, NU)                                                                                \
    extern template cudaError_t col_fluid_launch<double, HSE, GRAV, -1, false, NU>(const ColFluidArgs<double> &,  \
                                                                                   cudaStream_t);
FISH_F64_T2(false, 0, false)
FISH_F64_T2(false, 0, true)
FISH_F64_T2(false, 1, false)
FISH_F64_T2(false, 1, true)
FISH_F64_T2(true, 0, false)
FISH_F64_T2(true, 0, true)
FISH_F64_T2(true, 1, false)
FISH_F64_T2(true, 1, true)
FISH_F64_T2(false, 2, false)
#undef FISH_F64_T2
extern template cudaError_t col_fluid_launch<double, false, 0, LIM_VANLEER, false, false>(const ColFluidArgs<double> &,
                                                                                        cudaStream_t);
extern template cudaError_t col_ct_launch<double, LIM_VANLEER, false, false>(const ColCTArgs<double> &, cudaStream_t);
extern template cudaError_t col_ct_launch<double, -1, false, false>(const ColCTArgs<double> &, cudaStream_t);
extern template cudaError_t col_ct_launch<double, -1, false, true>(const ColCTArgs<double> &, cudaStream_t);
template struct Launch<double>;
template cudaError_t col_fluid<double>(const ColFluidArgs<double> &, bool, bool, cudaStream_t);
template cudaError_t col_ct<double>(const ColCTArgs<double> &, bool, cudaStream_t);
}

namespace fish {
cudaError_t launch_cfl_finish(unsigned long long *minbits, double k, double *dt, double *dt_copy,
                              cudaStream_t s)
{
    cfl_finish_kernel<<<1, 1, 0, s>>>(minbits, k, dt, dt_copy);
    return cudaGetLastError();
}

// Eight contiguous copies in one launch (blockIdx.y: the field), in units of U:
// the plane slabs of a ghost exchange are small, and a copy each costs more in
// launches than in traffic.
template <class U> struct Copy8Args {
    const U *src[8];
    U *dst[8];
    size_t n;
};
template <class U> static __global__ void __launch_bounds__(256) copy8_kernel(const Copy8Args<U> A)
{
    const U *src = A.src[blockIdx.y];
    U *dst = A.dst[blockIdx.y];
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < A.n; i += (size_t)gridDim.x * blockDim.x)
        dst[i] = src[i];
}
template <class U>
static cudaError_t copy8(const void *const src[8], void *const dst[8], size_t n, cudaStream_t s)
{
    Copy8Args<U> A;
    for (int f = 0; f < 8; ++f) {
        A.src[f] = (const U *)src[f];
        A.dst[f] = (U *)dst[f];
    }
    A.n = n / sizeof(U);
    const size_t blocks = (A.n + 1023) / 1024;
    copy8_kernel<U><<<dim3((unsigned)(blocks < 1 ? 1 : (blocks < 608 ? blocks : 608)), 8), 256, 0, s>>>(A);
    return cudaGetLastError();
}

cudaError_t launch_copy8(const void *const src[8], void *const dst[8], size_t n, cudaStream_t s)
{
    // 16 bytes at a time where every slab is so aligned, else words
    size_t al = n;
    for (int f = 0; f < 8; ++f) al |= (size_t)src[f] | (size_t)dst[f];
    if (al % 16 == 0) return copy8<uint4>(src, dst, n, s);
    if (al % 4 == 0) return copy8<unsigned>(src, dst, n, s);
    return copy8<unsigned char>(src, dst, n, s);
}

static __global__ void reset_min_kernel(unsigned long long *p) { *p = 0x7FF0000000000000ull; }

cudaError_t launch_reset_min(unsigned long long *minbits, cudaStream_t s)
{
    reset_min_kernel<<<1, 1, 0, s>>>(minbits);
    return cudaGetLastError();
}

cudaError_t launch_set_scalar(double *p, double v, cudaStream_t s)
{
    set_scalar_kernel<<<1, 1, 0, s>>>(p, v);
    return cudaGetLastError();
}

// FP64 pipe throughput probe: every thread runs eight independent chains of
// fused multiply-adds (x <- x a + b, |a| < 1, so the chains stay bounded) and
// writes its sum, so nothing is optimised away.  The FP64 sweeps are
// compared against this rate (their DADD, DMUL and DFMA each take one issue
// of the FP64 pipe).
static __global__ void __launch_bounds__(256) dfma_probe_kernel(double *out, int iters, double a, double b)
{
    double x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = 1.0 + 1e-3 * (threadIdx.x + k);
#pragma unroll 1
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = __fma_rn(x[k], a, b);
    }
    double sum = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) sum += x[k];
    out[(long long)blockIdx.x * blockDim.x + threadIdx.x] = sum;
}

cudaError_t launch_dfma_probe(double *out, int blocks, int iters, cudaStream_t s)
{
    dfma_probe_kernel<<<blocks, 256, 0, s>>>(out, iters, 0.9999999, 1e-7);
    return cudaGetLastError();
}
}  // namespace fish

