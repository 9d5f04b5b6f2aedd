// fish_col_impl.cuh -- launchers of the column-march kernels for one
// lane-vector type; included by the translation unit that instantiates them.
#pragma once

#include <type_traits>

#include "fish_column.cuh"

namespace fish {

static inline unsigned col_grid(long long work, int block)
{
    long long g = (work + block - 1) / block;
    return (unsigned)(g < 1 ? 1 : g);
}

// Whether the byte offsets of a sweep's FP32 fields fit in 32 bits.
template <class A_> static bool fits_u32(const A_ &A)
{
    return A.off + (long long)A.nf * A.no * A.n <= (1ll << 30);
}

// Length of the segments a sweep of n cells is cut into, for `blocks` column
// blocks of a kernel that keeps `slots` blocks on the GPU, `lone` of which
// already run without sharing a scheduler (FP32) or an FP64 pipe.  A segment
// of len cells costs len + `extra` march steps (its windows fill over the
// cells before it), so the number of segments S minimises
//   waves(blocks S) (ceil(n / S) + extra),
// a last wave of at most `lone` blocks counting `lone_cost` of a full one.
// Measured against every S from 1 to 64 on boxes from 32^3 to 1024^2 x 512:
// within 3 % of the best S.  L_d uncut and cut: 79 -> 36 us at 128^3 (FP32, four
// segments), 942 -> 215 us for the x sweep of 72 x 60 x 51 cells (FP64, six),
// 13.9 -> 12.4 ms at 256^3 (FP64, two: less of the last wave idle), 2.67 ->
// 2.52 ms at 640^3 (FP32, three).
static inline int col_segments(int n, long long blocks, int slots, int lone, double lone_cost, int extra)
{
    double best = 1e300;
    int len = n;
    for (int S = 1; S <= n; ++S) {
        const int l = (n + S - 1) / S;
        if ((n + l - 1) / l != S) continue;  // the same length as a smaller S
        const long long B = blocks * S;
        const long long full = B / slots, rem = B % slots;
        const double waves = (double)full + (rem == 0 ? 0.0 : (rem <= lone ? lone_cost : 1.0));
        const double cost = waves * (l + extra);
        if (cost < best * 0.999) {
            best = cost;
            len = l;
        }
        if (B > 64ll * slots) break;  // many waves: finer cuts only add steps
    }
    return len;
}

// Launch fluid_col_kernel over all columns: one thread per column group, the
// sweep in segments.
template <class V, bool HSE, int GRAV, int LIM, bool FT1, bool CFLF, bool NU, class IX>
static cudaError_t fluid_run(const ColFluidArgs<typename VT<V>::S> &A, cudaStream_t s)
{
    constexpr int T = fluid_threads<V>();
    const unsigned blocks = col_grid((long long)(A.nf / VT<V>::W) * A.no, T);
    const int sms = sm_count();
    constexpr int resident = fluid_resident<V, HSE>();
    const int len = VT<V>::F64 ? col_segments(A.n, blocks, resident * sms, 4 * sms, 0.6, 4)
                               : col_segments(A.n, blocks, resident * sms, sms, 0.7, 5);
    const dim3 grid(blocks, (unsigned)((A.n + len - 1) / len));
    fluid_col_kernel<V, HSE, GRAV, LIM, FT1, CFLF, NU, IX><<<grid, T, 0, s>>>(A, len);
    return cudaGetLastError();
}

// FP32 addresses by 32-bit byte offsets where they fit (boxes up to 1024^3),
// which need no 64-bit multiply-add per access: L_d 213 -> 199 us at 256^3 and
// 2690 -> 2541 us at 640^3 against int indices, B_d 170 -> 156 and 2285 ->
// 2139 us against 64-bit ones.
template <class V, bool HSE, int GRAV, int LIM, bool FT1, bool CFLF, bool NU>
static cudaError_t fluid_any(const ColFluidArgs<typename VT<V>::S> &A, cudaStream_t s)
{
    if constexpr (!VT<V>::F64) {
        if (fits_u32(A)) return fluid_run<V, HSE, GRAV, LIM, FT1, CFLF, NU, unsigned>(A, s);
    }
    return fluid_run<V, HSE, GRAV, LIM, FT1, CFLF, NU, long long>(A, s);
}

// (external linkage: the packed instantiations are spread over several
// translation units that compile in parallel)
template <class V, bool HSE, int GRAV, int LIM, bool FT1, bool NU = false>
cudaError_t col_fluid_launch(const ColFluidArgs<typename VT<V>::S> &A, cudaStream_t s)
{
    if constexpr (std::is_same<V, P2>::value && !NU) {
        if (A.cfl_min) return fluid_any<V, HSE, GRAV, LIM, FT1, true, false>(A, s);
    }
    if (A.cfl_min) return cudaErrorInvalidValue;  // only the two-column kernels carry the CFL epilogue
    return fluid_any<V, HSE, GRAV, LIM, FT1, false, NU>(A, s);
}

#ifndef FISH_F64_VL
#define FISH_F64_VL 1   // FP64 sweeps without gravity: compile-time Van Leer limiter
#endif

// GRAV: 0 no potential, 1 unsplit source terms, 2 split kicks in the march
// (uniform meshes; with an irregular mesh the kicks run as separate passes)
template <class V, bool HSE, int GRAV, bool FT1>
static cudaError_t col_fluid_lim(const ColFluidArgs<typename VT<V>::S> &A, cudaStream_t s)
{
    if constexpr (GRAV == 2) {
        if (A.wd) return cudaErrorInvalidValue;
    }
    if constexpr (std::is_same<V, P2>::value) {
        // compile-time limiters for the throughput path (an irregular mesh
        // with Van Leer; its other limiters run on the one-column kernels)
        if constexpr (HSE) {
            if (A.wd) return cudaErrorInvalidValue;
        } else if constexpr (GRAV != 2) {
            if (A.wd) {
                if (A.lim == LIM_VANLEER) return col_fluid_launch<V, HSE, GRAV, LIM_VANLEER, FT1, true>(A, s);
                return cudaErrorInvalidValue;
            }
        }
        if (A.lim == LIM_VANLEER) return col_fluid_launch<V, HSE, GRAV, LIM_VANLEER, FT1>(A, s);
        if (A.lim == LIM_MINMOD) return col_fluid_launch<V, HSE, GRAV, LIM_MINMOD, FT1>(A, s);
        if constexpr (!HSE) {
            if (A.lim == LIM_HYBRID) return col_fluid_launch<V, HSE, GRAV, LIM_HYBRID, FT1>(A, s);
        }
        return cudaErrorInvalidValue;
    } else {
        // irregular mesh: widths along d (limiter read at run time)
        if constexpr (GRAV != 2) {
            if (A.wd) return col_fluid_launch<V, HSE, GRAV, -1, FT1, true>(A, s);
        }
        if constexpr (std::is_same<V, float>::value && !HSE && GRAV == 0) {
            // the plain sweeps of odd fast extents with compile-time limiters
            if (A.lim == LIM_VANLEER) return col_fluid_launch<V, HSE, GRAV, LIM_VANLEER, FT1>(A, s);
            if (A.lim == LIM_MINMOD) return col_fluid_launch<V, HSE, GRAV, LIM_MINMOD, FT1>(A, s);
        }
        if constexpr (VT<V>::F64 && !HSE && GRAV == 0 && FISH_F64_VL) {
            // the plain FP64 sweeps with a compile-time Van Leer limiter
            if (A.lim == LIM_VANLEER) return col_fluid_launch<V, HSE, GRAV, LIM_VANLEER, FT1>(A, s);
        }
        return col_fluid_launch<V, HSE, GRAV, -1, FT1>(A, s);
    }
}

template <class V, bool FT1>
static cudaError_t col_fluid_ft(const ColFluidArgs<typename VT<V>::S> &A, bool hse, cudaStream_t s)
{
    if (hse && A.sg) return cudaErrorInvalidValue;  // split gravity and the correction exclude each other
    if (hse && A.phi) return col_fluid_lim<V, true, 1, FT1>(A, s);
    if (hse) return col_fluid_lim<V, true, 0, FT1>(A, s);  // correction with phi = 0
    if (A.phi && A.sg) return col_fluid_lim<V, false, 2, FT1>(A, s);
    if (A.phi) return col_fluid_lim<V, false, 1, FT1>(A, s);
    return col_fluid_lim<V, false, 0, FT1>(A, s);
}

template <class V>
cudaError_t col_fluid(const ColFluidArgs<typename VT<V>::S> &A, bool hse, bool ft1, cudaStream_t s)
{
    if constexpr (VT<V>::F64) {
        return ft1 ? col_fluid_ft<V, true>(A, hse, s) : col_fluid_ft<V, false>(A, hse, s);
    } else {
        if (!ft1) return cudaErrorInvalidValue;
        return col_fluid_ft<V, true>(A, hse, s);
    }
}

template <class V, int LIM, bool FT1, bool NU = false>
cudaError_t col_ct_launch(const ColCTArgs<typename VT<V>::S> &A, cudaStream_t s)
{
    // one warp per 31 W columns of a row (plus a halo lane); a block takes
    // one segment of ct_rows() consecutive rows
    const int segc = 31 * VT<V>::W;
    const long long blocks = (long long)((A.nf + segc - 1) / segc) * ((A.no + ct_rows<V>() - 1) / ct_rows<V>());
    const int sms = sm_count();
    constexpr int resident = ct_resident<V>();
    const int len = VT<V>::F64 ? col_segments(A.n, blocks, resident * sms, 4 * sms, 0.6, 6)
                               : col_segments(A.n, blocks, resident * sms, sms, 0.7, 8);
    const dim3 grid((unsigned)blocks, (unsigned)((A.n + len - 1) / len));
    if constexpr (!VT<V>::F64) {
        if (fits_u32(A)) {
            ct_col_kernel<V, LIM, FT1, NU, unsigned><<<grid, 32 * ct_rows<V>(), 0, s>>>(A, len);
            return cudaGetLastError();
        }
    }
    ct_col_kernel<V, LIM, FT1, NU><<<grid, 32 * ct_rows<V>(), 0, s>>>(A, len);
    return cudaGetLastError();
}

template <class V> cudaError_t col_ct(const ColCTArgs<typename VT<V>::S> &A, bool ft1, cudaStream_t s)
{
    const bool nu = A.wd != nullptr;
    if (nu && (!A.wf || !A.wo)) return cudaErrorInvalidValue;
    if constexpr (VT<V>::F64) {
        if (nu) return ft1 ? col_ct_launch<V, -1, true, true>(A, s) : col_ct_launch<V, -1, false, true>(A, s);
        if (FISH_F64_VL && A.lim == LIM_VANLEER)
            return ft1 ? col_ct_launch<V, LIM_VANLEER, true>(A, s) : col_ct_launch<V, LIM_VANLEER, false>(A, s);
        return ft1 ? col_ct_launch<V, -1, true>(A, s) : col_ct_launch<V, -1, false>(A, s);
    } else if constexpr (std::is_same<V, P2>::value) {
        if (nu) return cudaErrorInvalidValue;
        if (A.lim == LIM_VANLEER) return col_ct_launch<V, LIM_VANLEER, true>(A, s);
        if (A.lim == LIM_MINMOD) return col_ct_launch<V, LIM_MINMOD, true>(A, s);
        return cudaErrorInvalidValue;
    } else {
        if (nu && A.lim == LIM_VANLEER) return col_ct_launch<V, LIM_VANLEER, true, true>(A, s);
        if (nu) return col_ct_launch<V, -1, true, true>(A, s);
        // FP32: compile-time limiters for the throughput path
        if (A.lim == LIM_VANLEER) return col_ct_launch<V, LIM_VANLEER, true>(A, s);
        if (A.lim == LIM_MINMOD) return col_ct_launch<V, LIM_MINMOD, true>(A, s);
        return col_ct_launch<V, -1, true>(A, s);
    }
}

}  // namespace fish
