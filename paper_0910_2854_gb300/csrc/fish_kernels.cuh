// fish_kernels.cuh -- sm_103a kernels around FISH's operator-split sweep
// (Kaeppeli et al., arXiv:0910.2854), templated on the real type: the CFL
// reduction, the diagnostics, the layout change between sweep directions,
// the operator-split gravity and precision conversions.  The sweeps
// themselves (L_d and B_d) are the column marches of fish_column.cuh.
//
// Data layout: structure of arrays; fields rho, m_x, m_y, m_z, E, b_x, b_y,
// b_z, b_x[i,j,k] being the face average at x_{i+1/2} (eq0080-eq0080b), in
// one of two layouts (x fastest, or y fastest for the x sweeps; Geom says
// which).  No ghost cells are stored: the ghost layer of every sweep is an
// index map (periodic wrap or zeroth-order extrapolation).
#pragma once

#include "fish_math.cuh"
#include "fish_types.h"
#include "fish_vec.cuh"

namespace fish {

// ---------------------------------------------------------------------------
// CFL (eq0083-eq0084): min over cells and axes of h_d / (|v_d| + c_F,d)
// ---------------------------------------------------------------------------
template <class T> struct CFLArgs {
    const T *in[8];
    Geom g;
    double h[3];
    T gamma, gm1;
    unsigned long long *minbits;  // order-preserving bits of the positive minimum (double)
    unsigned *flags;
    const T *w[3] = {nullptr, nullptr, nullptr};  // irregular mesh: cell widths per axis (eq0420)
    int k0 = 0, nk = -1;  // z-planes k0 .. k0+nk-1 only (nk < 0: all)
};

// FP32 signal speeds along the three axes of one cell, sharing the
// primitives: out[d] = (|v_d| + c_F,d) / h_d (reading C-15), compensated
// pressure recovery as in the sweeps.
__device__ __forceinline__ float cfl_rate_f32(const float u[5], const float b[3], float gamma, float gm1,
                                              const float rh[3], unsigned &flags)
{
    const float ri = __fdividef(1.0f, u[0]);
    const float v[3] = {u[1] * ri, u[2] * ri, u[3] * ri};
    const float kin = 0.5f * (u[1] * v[0] + u[2] * v[1] + u[3] * v[2]);
    const float b2[3] = {b[0] * b[0], b[1] * b[1], b[2] * b[2]};
    const float mag = 0.5f * (b2[0] + b2[1] + b2[2]);
    const float p = gas_pressure<float>(gm1, u[4], kin, mag);
    const float a2 = gamma * p * ri;
    float best = 0.0f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float bn2 = b2[d] * ri;
        const float bt2 = (b2[(d + 1) % 3] + b2[(d + 2) % 3]) * ri;
        const float B2 = bn2 + bt2;
        const float disc = (a2 - B2) * (a2 - B2) + 4.0f * a2 * bt2;
        const float cf = sqrtf(0.5f * (a2 + B2 + sqrtf(disc)));
        best = fmaxf(best, (fabsf(v[d]) + cf) * rh[d]);
        if (cf != cf) flags |= FLAG_NAN;
    }
    if (!(u[0] > 0.0f)) flags |= FLAG_RHO;
    if (!(p > 0.0f)) flags |= FLAG_P;
    return best;
}

// Conversions that keep off the FP64 pipe, where GB300 converts: zeros and
// normal numbers by moving the exponent and mantissa.  `odd` collects whether
// an operand was something else, whose result is then not its value.
__device__ __forceinline__ double widen(double f, unsigned &) { return f; }
__device__ __forceinline__ double widen(float f, unsigned &odd)
{
    const unsigned u = __float_as_uint(f), top = u & 0x80000000u, m = u & 0x7fffffffu;
    odd |= m != 0u && m - 0x00800000u >= 0x7f000000u ? 1u : 0u;  // subnormal, infinite, NaN
    return __hiloint2double((int)(m ? top | ((m >> 3) + 0x38000000u) : top), (int)(m << 29));
}
// towards zero (1.2e-7 relative)
__device__ __forceinline__ float narrow(double d, unsigned &odd)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d), m = hi & 0x7fffffffu;
    odd |= m != 0u && m - 0x38100000u >= 0x0fe00000u ? 1u : 0u;  // outside the normal numbers of FP32
    return m ? __uint_as_float((hi & 0x80000000u) | ((m - 0x38000000u) << 3) | (lo >> 29)) : 0.0f;
}

// Upper bound of the FP64 path's largest rate (|v_d| + c_F,d) / h_d of a cell,
// in FP32 behind the FP64 pressure, with margins for the FP32 rounding: with
// c^2 = a^2 + B^2, t = a^2 / c^2 and s = b_t^2 / (rho c^2),
//   c_F^2 = c^2 (1 + sqrt((2 t - 1)^2 + 4 t s)) / 2.
// Infinite where an operand is no normal FP32 number or zero, NaN included, and
// where the density or the pressure is not positive by far more than rounding:
// the FP64 path, which such a cell then takes, finds whether they are.
__device__ __forceinline__ float cfl_bound_f64(const double u[5], const double b[3], double gamma, double gm1,
                                               const float rh[3])
{
    const double ri = rcp64(u[0]);
    const double v[3] = {u[1] * ri, u[2] * ri, u[3] * ri};
    const double k2 = u[1] * v[0] + u[2] * v[1] + u[3] * v[2];
    const double b2 = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
    const double e = __fma_rn(-0.5, b2, __fma_rn(-0.5, k2, u[4]));
    const double p = gm1 * e;
    const double g2 = gamma * p, s2 = g2 + b2;   // rho a^2, rho c^2
    unsigned odd = 0;
    const bool sure = pos64(u[0]) && narrow(e, odd) > 1e-12f * narrow(u[4], odd);
    const float s2f = narrow(s2, odd), f2 = narrow(b2, odd);
    const float c2 = narrow(s2 * ri, odd), rs = __fdividef(1.0f, s2f), t = narrow(g2, odd) * rs;
    float r = 0.0f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float bn = narrow(b[d], odd);
        const float s = fmaxf(f2 - bn * bn, 0.0f) * rs + 1e-6f;
        const float x = 2.0f * t - 1.0f;
        const float cf = sqrtf(0.5f * c2 * (1.0f + sqrtf(x * x + 4.0f * t * s)));
        r = fmaxf(r, (fabsf(narrow(v[d], odd)) + cf) * rh[d]);
    }
    // (b_n^2 against b^2 must not under- or overflow either)
    const bool ok = sure && !odd && s2f > 1e-30f && s2f < 1e30f && c2 > 1e-30f && r < 1e30f;
    return ok ? r * 1.00001f : __int_as_float(0x7f800000);
}

// CFL minimum over the box: a warp per row along the fastest memory axis (no
// per-cell index division; short rows leave no warp idle), per-block minimum,
// then one atomic on the order-preserving bits of the positive double.  Bound
// by HBM in FP32.  FP64 would be bound by its pipe (six square roots and 24
// quotients per cell, 9.8 ms at 256^3): a cell is evaluated in FP64 only if its
// bound above reaches the smallest step found so far, by the warp or, at the
// start of a row, by the whole grid.
// PAIR (FP32, even rows): a lane takes two adjacent cells with 8-byte loads.
template <class T, bool PAIR>
__global__ void __launch_bounds__(256) cfl_kernel(CFLArgs<T> A)
{
    const Geom &g = A.g;
    const bool yf = g.ord[0] == 1;  // y fastest (else x); z is the slowest axis of both layouts
    const int nf = yf ? g.n[1] : g.n[0], nm = yf ? g.n[0] : g.n[1], ns = g.n[2];
    const T *bxp = A.in[5], *byp = A.in[6], *bzp = A.in[7];
    const long long of0 = gmap(-1, nf, g.bc);  // to the lower neighbour of a row's first cell
    const int kb = A.nk < 0 ? 0 : A.k0;
    const long long rows = (long long)nm * (A.nk < 0 ? ns : A.nk);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double best = 1e300;   // min of h_d / (|v_d| + c_F,d)
    double sent = 1e300;   // FP64: the smallest minimum this thread has put into *minbits
    float fbest = 0.0f;    // FP32 path: max of (|v_d| + c_F,d) / h_d; FP64: a lower bound of 1 / best
    unsigned flags = 0;
    float rh[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) rh[d] = (float)(1.0 / A.h[d]);
    for (long long row = (long long)blockIdx.x * 8 + wid; row < rows; row += (long long)gridDim.x * 8) {
        const int m = (int)(row % nm), k = kb + (int)(row / nm);
        const long long rbase = ((long long)k * nm + m) * nf;
        // offsets to the lower neighbours: along the row, across the rows, across the planes
        const long long om = (long long)(gmap(m - 1, nm, g.bc) - m) * nf;
        const long long oz = (long long)(gmap(k - 1, ns, g.bc) - k) * nm * nf;
        if (A.w[0]) {
            // irregular mesh: this row's widths along the two slower axes
            if (yf) rh[0] = (float)(1.0 / (double)A.w[0][m]);
            else rh[1] = (float)(1.0 / (double)A.w[1][m]);
            rh[2] = (float)(1.0 / (double)A.w[2][k]);
        }
        if constexpr (sizeof(T) == 8)
            fbest = fmaxf(fbest, 0.999999f / (float)__longlong_as_double(*(volatile long long *)A.minbits));
        if constexpr (PAIR) {
            for (int f = 2 * lane; f < nf; f += 64) {
                const long long idx = rbase + f;
                const long long of = f > 0 ? -1 : of0;
                const T *bfp = yf ? byp : bxp, *bmp = yf ? bxp : byp;
                const P2 bf = vload<P2>(bfp, idx), bz = vload<P2>(bzp, idx) + vload<P2>(bzp, idx + oz);
                const P2 bfc = vshift_lo(__ldg(bfp + idx + of), bf) + bf;
                const P2 bmc = vload<P2>(bmp, idx) + vload<P2>(bmp, idx + om);
                P2 u[5];
#pragma unroll
                for (int i = 0; i < 5; ++i) u[i] = vload<P2>(A.in[i], idx);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    if (A.w[0]) {
                        if (yf) rh[1] = (float)(1.0 / (double)A.w[1][f + c]);
                        else rh[0] = (float)(1.0 / (double)A.w[0][f + c]);
                    }
                    const float uc[5] = {vget(u[0], c), vget(u[1], c), vget(u[2], c), vget(u[3], c), vget(u[4], c)};
                    const float bc[3] = {0.5f * vget(yf ? bmc : bfc, c), 0.5f * vget(yf ? bfc : bmc, c),
                                         0.5f * vget(bz, c)};
                    fbest = fmaxf(fbest, cfl_rate_f32(uc, bc, (float)A.gamma, (float)A.gm1, rh, flags));
                }
            }
            continue;
        }
        for (int fw = 0; fw < nf; fw += 32) {
            // (FP64: the lanes share their bound; the lanes past the row's end repeat its last cell)
            const int f = min(fw + lane, nf - 1);
            const long long idx = rbase + f;
            const long long of = f > 0 ? -1 : of0;
            if (A.w[0]) {
                if (yf) rh[1] = (float)(1.0 / (double)A.w[1][f]);
                else rh[0] = (float)(1.0 / (double)A.w[0][f]);
            }
            const T bc[3] = {T(0.5) * (__ldg(bxp + idx + (yf ? om : of)) + __ldg(bxp + idx)),
                             T(0.5) * (__ldg(byp + idx + (yf ? of : om)) + __ldg(byp + idx)),
                             T(0.5) * (__ldg(bzp + idx + oz) + __ldg(bzp + idx))};
            const T u0[5] = {__ldg(A.in[0] + idx), __ldg(A.in[1] + idx), __ldg(A.in[2] + idx), __ldg(A.in[3] + idx),
                             __ldg(A.in[4] + idx)};
            if constexpr (sizeof(T) == 8) {
                const float bound = cfl_bound_f64(u0, bc, A.gamma, A.gm1, rh);
                if (!(fbest > 1e-30f && bound < fbest)) {
                    // per axis in the paper's frame, the oracle's operation order
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const int t1 = (d + 1) % 3, t2 = (d + 2) % 3;
                        const T u[5] = {u0[0], u0[1 + d], u0[1 + t1], u0[1 + t2], u0[4]};
                        const T bb[3] = {bc[d], bc[t1], bc[t2]};
                        const T sp = signal_speed<T>(u, bb, A.gamma, A.gm1, flags);
                        // eq0420
                        const T hd = A.w[0] ? A.w[d][d == 2 ? k : ((d == 1) == yf ? f : m)] : T(A.h[d]);
                        const double r = (double)(hd / sp);
                        best = r < best ? r : best;
                    }
                    fbest = fmaxf(fbest, 0.999999f / (float)best);
                }
                fbest = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fbest)));
            } else {
                fbest = fmaxf(fbest, cfl_rate_f32(u0, bc, (float)A.gamma, (float)A.gm1, rh, flags));
            }
        }
        if constexpr (sizeof(T) == 8) {
            // the row's minimum, so that the other warps' bounds follow
            if (best > 0.0 && best < sent) {
                sent = best;
                atomicMin(A.minbits, (unsigned long long)__double_as_longlong(best));
            }
        }
    }
    if constexpr (sizeof(T) == 4) best = fbest > 0.0f ? 1.0 / (double)fbest : 1e300;
    // block minimum, then one atomic on the order-preserving bits
    for (int off = 16; off > 0; off >>= 1) {
        double o = __shfl_xor_sync(0xffffffffu, best, off);
        best = o < best ? o : best;
    }
    __shared__ double wmin[8];
    if (lane == 0) wmin[wid] = best;
    __syncthreads();
    if (wid == 0) {
        best = lane < (int)(blockDim.x >> 5) ? wmin[lane] : 1e300;
        for (int off = 16; off > 0; off >>= 1) {
            double o = __shfl_xor_sync(0xffffffffu, best, off);
            best = o < best ? o : best;
        }
        if (lane == 0) {
            if (best != best || best <= 0.0) {
                flags |= FLAG_NAN;
            } else {
                atomicMin(A.minbits, (unsigned long long)__double_as_longlong(best));
            }
        }
    }
    if (flags) atomicOr(A.flags, flags);
}

// dt = k * min; resets the minimum for the next reduction.
static __global__ void cfl_finish_kernel(unsigned long long *minbits, double k, double *dt_out, double *dt_copy)
{
    const double m = __longlong_as_double((long long)*minbits);
    const double dt = k * m;
    *dt_out = dt;
    if (dt_copy) *dt_copy = dt;
    *minbits = 0x7FF0000000000000ull;  // +inf
}

static __global__ void set_scalar_kernel(double *p, double v) { *p = v; }

// ---------------------------------------------------------------------------
// diagnostics: per-block FP64 partial sums (fixed order) and max |div b|
// ---------------------------------------------------------------------------
template <class T> struct DiagArgs {
    const T *in[8];
    Geom g;
    double h[3];
    double *partial;  // [gridDim.x][9]
    // irregular mesh: cell widths per axis; the sums are then volume-weighted
    // in the kernel and the divergence takes each cell's own widths
    const T *w[3] = {nullptr, nullptr, nullptr};
};

// A warp takes rows of the fastest memory axis (fixed by the grid, so the
// order of the sums is fixed).  Bound by the FP64 pipe: eight sums per cell and,
// for cells that may hold the maximum, the divergence with quotients behind
// shared reciprocals of the widths.
template <class T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 2) diag_kernel(DiagArgs<T> A)
{
    const Geom &g = A.g;
    const bool yf = g.ord[0] == 1;  // y fastest (else x)
    const int nf = yf ? g.n[1] : g.n[0], nm = yf ? g.n[0] : g.n[1], ns = g.n[2];
    const long long rows = (long long)nm * ns;
    const bool open = g.bc == BC_OUTFLOW;
    const long long of0 = gmap(-1, nf, g.bc);  // to the lower neighbour of a row's first cell
    double s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    long long dmax = 0;  // bits of the largest |div b|
    float dlow = 0.0f;   // FP32 states: a lower bound of the warp's largest
    double hx[3], ri[3];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        hx[ax] = A.h[ax];
        ri[ax] = rcp64(hx[ax]);
    }
    for (long long row = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); row < rows; row += (long long)gridDim.x * 8) {
        const int m = (int)(row % nm), k = (int)(row / nm);
        const long long base = row * nf;
        const long long om = (long long)(gmap(m - 1, nm, g.bc) - m) * nf;
        const long long oz = (long long)(gmap(k - 1, ns, g.bc) - k) * nm * nf;
        if (A.w[0]) {
            if (yf) ri[0] = rcp64(hx[0] = (double)A.w[0][m]);
            else ri[1] = rcp64(hx[1] = (double)A.w[1][m]);
            ri[2] = rcp64(hx[2] = (double)A.w[2][k]);
        }
        const bool skip_row = open && ((nm > 1 && m == 0) || (ns > 1 && k == 0));
        for (int f = threadIdx.x & 31; f < nf; f += 32) {
            const long long idx = base + f;
            const long long of = f > 0 ? -1 : of0;
            const T v[11] = {__ldg(A.in[0] + idx), __ldg(A.in[1] + idx), __ldg(A.in[2] + idx), __ldg(A.in[3] + idx),
                             __ldg(A.in[4] + idx), __ldg(A.in[5] + idx), __ldg(A.in[6] + idx), __ldg(A.in[7] + idx),
                             __ldg(A.in[5] + idx + (yf ? om : of)), __ldg(A.in[6] + idx + (yf ? of : om)),
                             __ldg(A.in[7] + idx + oz)};
            double q[11];
            unsigned odd = 0;
#pragma unroll
            for (int i = 0; i < 11; ++i) q[i] = widen(v[i], odd);
            if (odd) {
#pragma unroll
                for (int i = 0; i < 11; ++i) q[i] = (double)v[i];
            }
            if (A.w[0]) {
                if (yf) ri[1] = rcp64(hx[1] = (double)A.w[1][f]);
                else ri[0] = rcp64(hx[0] = (double)A.w[0][f]);
                const double vol = hx[0] * hx[1] * hx[2];
#pragma unroll
                for (int i = 0; i < 8; ++i) s[i] += q[i] * vol;
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) s[i] += q[i];
            }
            if (!skip_row && !(open && nf > 1 && f == 0)) {
                if constexpr (sizeof(T) == 4) {
                    // in FP32 first, with a bound of its rounding: only a
                    // cell that may exceed the maximum is evaluated in FP64
                    const float e0 = (float)(v[5] - v[8]) * (float)ri[0], e1 = (float)(v[6] - v[9]) * (float)ri[1],
                                e2 = (float)(v[7] - v[10]) * (float)ri[2];
                    const float top = fabsf(e0 + e1 + e2) + 1e-6f * (fabsf(e0) + fabsf(e1) + fabsf(e2));
                    if (dlow > 1e-30f && top < dlow) continue;
                }
                const double dv = quot64(q[5] - q[8], hx[0], ri[0]) + quot64(q[6] - q[9], hx[1], ri[1]) +
                                  quot64(q[7] - q[10], hx[2], ri[2]);
                // (a NaN counts as none, as in fmax)
                const long long d = __double_as_longlong(fabs(dv));
                if (d <= 0x7ff0000000000000ll) dmax = max(dmax, d);
                if constexpr (sizeof(T) == 4) dlow = fmaxf(dlow, 0.999999f * (float)__longlong_as_double(dmax));
            }
        }
        if constexpr (sizeof(T) == 4)
            dlow = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(dlow)));
    }
    __shared__ double red[256][9];
    for (int f = 0; f < 8; ++f) red[threadIdx.x][f] = s[f];
    red[threadIdx.x][8] = __longlong_as_double(dmax);
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            for (int f = 0; f < 8; ++f) red[threadIdx.x][f] += red[threadIdx.x + w][f];
            red[threadIdx.x][8] = fmax(red[threadIdx.x][8], red[threadIdx.x + w][8]);
        }
        __syncthreads();
    }
    if (threadIdx.x < 9) A.partial[(long long)blockIdx.x * 9 + threadIdx.x] = red[0][threadIdx.x];
}

// ---------------------------------------------------------------------------
// layout change: per z-plane 2-D transpose of every field between
// [z][y][x] (x fastest) and [z][x][y] (y fastest) -- the paper's data
// rotation between sweeps (Sec. 3) as a tiled shared-memory transpose with
// coalesced reads and writes.  src rows have length nr, there are nc rows.
// ---------------------------------------------------------------------------
template <class T> struct TransArgs {
    const T *src[8];
    T *dst[8];
    int nr, nc;          // source: nc rows of nr elements; destination: nr rows of nc
    int nf;              // number of fields (1..8)
    int fb;              // fields per block (blocks of one tile along gridDim.z: ceil(nf / fb))
    long long plane;     // elements per z-plane
};

// Tiles of FISH_TR_ROWS source rows x 32 elements: a thread keeps
// FISH_TR_ROWS/8 loads in flight, and the loads of field f+1 are issued
// before field f is stored (two tiles, one barrier per field: a tile is
// rewritten two fields later, after every thread has passed the barrier
// between).
#ifndef FISH_TR_ROWS
#define FISH_TR_ROWS 64
#endif
// FP32 transpose with 16-byte accesses: tiles of 64 x 64 elements, each
// thread moves four float4 of a field per tile (source rows of 256 bytes
// read whole, destination rows of 256 bytes written whole), the next
// field's float4 loads in flight while the current tile is stored.  Needs
// nr and nc multiples of 4 (16-byte aligned rows).  Grid: ceil(nr/64) x
// ceil(nc/64) x nz, 256 threads.
template <class T>
__global__ void __launch_bounds__(256) transpose4_kernel(TransArgs<T> A)
{
    static_assert(sizeof(T) == 4, "16-byte accesses of four 4-byte elements");
    __shared__ T tile[2][64][65];
    const int r0 = blockIdx.x * 64, c0 = blockIdx.y * 64;
    // a grid of few tiles splits the fields over blocks: a block moves one
    // field after the other, each a round trip to memory
    const int nb = (A.nf + A.fb - 1) / A.fb, fs = (int)(blockIdx.z % nb) * A.fb, fe = min(fs + A.fb, A.nf);
    const long long zoff = (long long)(blockIdx.z / nb) * A.plane;
    const int t = threadIdx.x;
    const int lr = t >> 4, l4 = (t & 15) * 4;  // row within a 16-row band, first element of the float4
    float4 v[4];
    auto load = [&](const T *src) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = c0 + lr + 16 * k, r = r0 + l4;
            v[k] = (c < A.nc && r < A.nr) ? __ldg(reinterpret_cast<const float4 *>(src + zoff + (long long)c * A.nr + r))
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    load(A.src[fs]);
#pragma unroll 1
    for (int f = fs; f < fe; ++f) {
        const int b = f & 1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            T *row = &tile[b][lr + 16 * k][l4];
            row[0] = v[k].x;
            row[1] = v[k].y;
            row[2] = v[k].z;
            row[3] = v[k].w;
        }
        __syncthreads();
        if (f + 1 < fe) load(A.src[f + 1]);
        T *__restrict__ dst = A.dst[f] + zoff;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // destination row r0 + lr + 16k holds source column r0 + lr + 16k
            const int rl = lr + 16 * k, r = r0 + rl, c = c0 + l4;
            if (r < A.nr && c < A.nc) {
                float4 o;
                o.x = tile[b][l4 + 0][rl];
                o.y = tile[b][l4 + 1][rl];
                o.z = tile[b][l4 + 2][rl];
                o.w = tile[b][l4 + 3][rl];
                *reinterpret_cast<float4 *>(dst + (long long)r * A.nc + c) = o;
            }
        }
    }
}

// tile height: FP64 tiles stay within the 48 KB of static shared memory
template <class T> constexpr int tr_rows() { return sizeof(T) == 8 && FISH_TR_ROWS > 64 ? 64 : FISH_TR_ROWS; }
template <class T>
__global__ void __launch_bounds__(256) transpose_kernel(TransArgs<T> A)
{
    constexpr int TR = tr_rows<T>(), KL = TR / 8;
    __shared__ T tile[2][TR][33];
    const int r0 = blockIdx.x * 32, c0 = blockIdx.y * TR;
    const int nb = (A.nf + A.fb - 1) / A.fb, fs = (int)(blockIdx.z % nb) * A.fb, fe = min(fs + A.fb, A.nf);
    const long long zoff = (long long)(blockIdx.z / nb) * A.plane;
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    const int rl = r0 + tx;
    T v[KL];
#pragma unroll
    for (int k = 0; k < KL; ++k) {
        const int c = c0 + ty + 8 * k;
        v[k] = (rl < A.nr && c < A.nc) ? A.src[fs][zoff + (long long)c * A.nr + rl] : T(0);
    }
#pragma unroll 1
    for (int f = fs; f < fe; ++f) {
        const int b = f & 1;
#pragma unroll
        for (int k = 0; k < KL; ++k) tile[b][ty + 8 * k][tx] = v[k];
        __syncthreads();
        if (f + 1 < fe) {
            const T *__restrict__ src = A.src[f + 1] + zoff;
#pragma unroll
            for (int k = 0; k < KL; ++k) {
                const int c = c0 + ty + 8 * k;
                v[k] = (rl < A.nr && c < A.nc) ? src[(long long)c * A.nr + rl] : T(0);
            }
        }
        T *__restrict__ dst = A.dst[f] + zoff;
#pragma unroll
        for (int k = 0; k < KL; ++k) {
            const int idx = ty + 8 * k;  // destination row r0 + (idx & 31), column block idx >> 5
            const int r = r0 + (idx & 31), cl = tx + 32 * (idx >> 5), c = c0 + cl;
            if (r < A.nr && c < A.nc) dst[(long long)r * A.nc + c] = tile[b][cl][idx & 31];
        }
    }
}

// ---------------------------------------------------------------------------
// operator-split gravity G_d(tau) (eq025111-eq02513): in place on the current
// state, m_d -= tau rho dphi/dx_d with the centred potential difference, and
// E changes by the kinetic energy change (reading C-22), tau = frac * dt.
// FP64 reads the cell potential in the current layout; FP32 the differences
// to the next cell along d (formed in FP64), phi_{i+1} - phi_{i-1} = D_i +
// D_{i-1} with D_{-1} = 0 at an outflow boundary.
// ---------------------------------------------------------------------------
template <class T> struct GravArgs {
    const T *rho;
    T *md, *E;
    const T *phi;
    const double *dt;
    double frac;
    Geom g;                 // layout; d is not its fastest axis
    int d;
    double h;
    const T *wd = nullptr;  // irregular mesh: cell widths along d (centre span, reading C-26)
};

// One block per row of the fastest memory axis at a time (grid-stride over
// rows): the coordinate along d, the neighbour offsets and the centre span
// are constant along a row, so the per-cell work is the kick alone.
template <class T>
__global__ void __launch_bounds__(256) gravity_kernel(GravArgs<T> A)
{
    const Geom &g = A.g;
    const int f0 = g.ord[0], f1 = g.ord[1], f2 = g.ord[2];
    const int nf = g.n[f0], nm = g.n[f1];
    const long long rows = (long long)nm * g.n[f2];
    const int n = g.n[A.d];
    const double tau = A.frac * *A.dt;
    for (long long row = blockIdx.x; row < rows; row += gridDim.x) {
        const int m = (int)(row % nm), k = (int)(row / nm);
        const long long base = (long long)m * g.st[f1] + (long long)k * g.st[f2];
        const int s = A.d == f1 ? m : k;
        const long long sd = g.st[A.d];
        const long long op = (long long)(gmap(s + 1, n, g.bc) - s) * sd;
        const long long om = (long long)(gmap(s - 1, n, g.bc) - s) * sd;
        if constexpr (sizeof(T) == 8) {
            const double span = A.wd ? 0.5 * A.wd[gmap(s - 1, n, g.bc)] + A.wd[s] + 0.5 * A.wd[gmap(s + 1, n, g.bc)]
                                     : 2.0 * A.h;
            for (int f = threadIdx.x; f < nf; f += blockDim.x) {
                const long long i = base + f;
                const double dphi = (A.phi[i + op] - A.phi[i + om]) / span;
                const double rho = A.rho[i];
                const double mo = A.md[i];
                const double mn = mo - tau * rho * dphi;
                A.md[i] = mn;
                A.E[i] = A.E[i] + 0.5 * (mn * mn - mo * mo) / rho;
            }
        } else {
            // phi_{s+1} - phi_{s-1} = D_s + D_{s-1}; D_{-1} = 0 at an outflow boundary
            const bool lower = s > 0 || g.bc == BC_PERIODIC;
            float rspan;
            if (A.wd) {
                rspan = 1.0f / (0.5f * (float)A.wd[gmap(s - 1, n, g.bc)] + (float)A.wd[s] +
                                0.5f * (float)A.wd[gmap(s + 1, n, g.bc)]);
            } else {
                rspan = (float)(0.5 / A.h);
            }
            const float ftau = (float)tau;
            for (int f = threadIdx.x; f < nf; f += blockDim.x) {
                const long long i = base + f;
                const float dm1 = lower ? A.phi[i + om] : 0.0f;
                const float dphi = (A.phi[i] + dm1) * rspan;
                const float rho = A.rho[i];
                const float mo = A.md[i];
                const float dm = -(ftau * rho) * dphi;
                A.md[i] = mo + dm;
                A.E[i] = A.E[i] + __fdividef(dm * (mo + 0.5f * dm), rho);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// precision conversion of one field
// ---------------------------------------------------------------------------
template <class S, class D>
__global__ void convert_kernel(const S *__restrict__ src, D *__restrict__ dst, long long n)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        dst[i] = (D)src[i];
}

}  // namespace fish
