// fish_column.cuh -- column-march kernels of FISH's fluid operator L_d and
// magnetic operator B_d (Kaeppeli et al., arXiv:0910.2854, Sec. 2-3).
//
// Geometry.  A sweep runs along axis d with element stride sd.  The two
// transverse axes are the "fast" axis (element stride 1, the fastest memory
// axis of the current layout) and the "other" axis (stride so).  A thread
// owns W adjacent columns along the fast axis (V = P2: two FP32 columns
// advanced together with packed FP32x2 arithmetic and 64-bit accesses;
// V = float or double: one column) and marches them along d, so every global
// access of a warp is coalesced.  In the x-fastest layout this serves the y
// and z sweeps; the x sweeps run on the y-fastest copy of the state.
//
// The march is the paper's pipelined loop (Sec. 3) held in registers: raw
// cell r enters, predicted cell r-1 is formed, corrected cell r-3 leaves.
// Windows are indexed by r mod 4 (unrolled by four) so they rotate without
// moves.  Ghost cells (periodic wrap or zeroth-order extrapolation, no ghost
// storage) are an index map of the loads.
//
// A thread marches a segment [a, b) of its columns: the raw cells a-3 .. b+2
// enter and the updated cells a .. b-1 leave.  One loop serves the start of a
// segment, its interior and its end: a step evaluates every stage, and only
// the old state's loads and the result's stores wait for the windows to fill.
// So the code of a kernel is four copies of the step (it was 23 with separate
// prologue, interior and tail), which a short march would otherwise fetch
// from L2 once per step, and a box with few columns is cut into segments until
// it fills the GPU (col_segments in fish_col_impl.cuh).
//
// Both operators read the current buffers and write the other ones.
#pragma once

#include <type_traits>

#include "fish_math.cuh"
#include "fish_types.h"
#include "fish_vec.cuh"

namespace fish {

// ---------------------------------------------------------------------------
// arguments
// ---------------------------------------------------------------------------
template <class S> struct ColFluidArgs {
    using Real = S;
    const S *u[5];          // rho, m_d, m_t1, m_t2, E of the current buffer (sweep frame)
    const S *bd, *bt1, *bt2;  // face fields b_d, b_t1, b_t2 (sweep frame)
    S *uo[5];               // outputs, sweep frame
    const S *phi;           // potential or nullptr; FP32: phi(next cell along d) - phi(cell), from FP64
    const double *dt;
    long long off;          // element offset of the box in the field arrays (batches; else 0)
    long long sd, so;       // strides along the sweep and the other transverse axis
    int n, nf, no;          // cells along the sweep, the fast and the other axis
    int bc;
    int lim;                // limiter (kernels with LIM < 0 read it at run time)
    S gamma, gm1, alpha;
    double h;               // cell width along d
    unsigned *flags;
    // CFL of the updated state (kernels built with CFLF): the maximum over the
    // output cells of (|v_a| + c_F,a) / h_a over the three axes a in the frame
    // order (d, t1, t2) goes to *cfl_min as the order-preserving bits of its
    // reciprocal (atomic minimum)
    unsigned long long *cfl_min;
    S rh[3];
    const S *wd = nullptr;  // irregular mesh (kernels built with NU): the n cell widths along d
    int sg = 0;             // 1: phi drives operator-split kicks G_d(dt/2) around the sweep, not source terms
};

template <class S> struct ColCTArgs {
    using Real = S;
    const S *rho, *md;      // density and momentum along d (unchanged by B_d)
    const S *bd, *bf, *bo;  // b_d and the face fields of the fast and other transverse axes
    S *bdo, *bfo, *boo;     // outputs (other buffer)
    const double *dt;
    long long off;          // element offset of the box in the field arrays (batches; else 0)
    long long sd, so;
    int n, nf, no;
    int bc;
    int lim;
    double h, hf, ho;       // cell widths along d, the fast and the other axis
    // irregular mesh (kernels built with NU): cell widths along d, fast, other
    const S *wd = nullptr, *wf = nullptr, *wo = nullptr;
};

// ---------------------------------------------------------------------------
// per-cell arithmetic (frame: component 0 along d)
// ---------------------------------------------------------------------------
template <class V> struct CCell {
    V u[5];
    V F[5];
    V d;                 // freezing speed |v_d| + c_F (label 0111)
    V p, cs, cf, vn;     // used by the hydrostatic correction only
};

// running checks for reading C-16.  FP32: min rho, min p, and a sum of c_F
// that turns NaN if any evaluated cell has none (a maximum of speeds drops a
// NaN, so this is the only trace of one); FP64: FLAG_* by the bits
template <class V> struct Checks {
    V mn_rho, mn_p, nsum;
    int hi;
};

template <class V> __device__ __forceinline__ void checks_init(Checks<V> &k)
{
    k.mn_rho = vb<V>(3.0e38f);
    k.mn_p = vb<V>(3.0e38f);
    k.nsum = vb<V>(0.0f);
    k.hi = 0;
}

template <class V> __device__ __forceinline__ unsigned checks_flags(const Checks<V> &k)
{
    if constexpr (VT<V>::F64) return (unsigned)k.hi;
    unsigned f = 0;
#pragma unroll
    for (int i = 0; i < VT<V>::W; ++i) {
        const auto r = vget(k.mn_rho, i), p = vget(k.mn_p, i), s = vget(k.nsum, i);
        if (!(r > 0)) f |= FLAG_RHO;
        if (!(p > 0)) f |= FLAG_P;
        if (s != s) f |= FLAG_NAN;
    }
    return f;
}

// E - (kin + mag) with the rounding error of kin + mag carried by an
// error-free two-sum (Knuth), so the cancellation against E costs no more
// than the rounding of its inputs (the FP32 compensated island).
__device__ __forceinline__ float eint_comp(float E, float kin, float mag)
{
    const float s = __fadd_rn(kin, mag);
    const float bp = __fsub_rn(s, kin);
    const float es = __fadd_rn(__fsub_rn(kin, __fsub_rn(s, bp)), __fsub_rn(mag, bp));
    return __fsub_rn(__fsub_rn(E, s), es);
}
__device__ __forceinline__ P2 eint_comp(P2 E, P2 kin, P2 mag)
{
    const P2 s = kin + mag;
    const P2 bp = s - kin;
    const P2 es = (kin - (s - bp)) + (mag - bp);
    return (E - s) - es;
}

// Primitives, flux vector (eq0100) and freezing speed (label 0111) of a cell
// with conserved state u and cell-centred field bb (reading C-1 for c_F).
template <class V>
__device__ __forceinline__ void ceval(const V u[5], const V bb[3], V gamma, V gm1, CCell<V> &c, Checks<V> &k)
{
    const V rho = u[0];
#pragma unroll
    for (int i = 0; i < 5; ++i) c.u[i] = u[i];
    V v0, v1, v2, p, a2, bn2, bt2, mag;
    if constexpr (VT<V>::F64) {
        const V ri = rcp64(rho);
        v0 = quot64(u[1], rho, ri);
        v1 = quot64(u[2], rho, ri);
        v2 = quot64(u[3], rho, ri);
        // kin = k2 / 2 and mag (here b^2, the factor 1/2 in the operations
        // that use it, whose products with it are exact)
        const V k2 = u[1] * v0 + u[2] * v1 + u[3] * v2;
        mag = bb[0] * bb[0] + bb[1] * bb[1] + bb[2] * bb[2];
        p = gm1 * __fma_rn(-0.5, mag, __fma_rn(-0.5, k2, u[4]));
        a2 = quot64(gamma * p, rho, ri);
        bn2 = quot64(bb[0] * bb[0], rho, ri);
        bt2 = quot64(bb[1] * bb[1] + bb[2] * bb[2], rho, ri);
    } else {
        const V half = vb<V>(0.5f);
        const V ri = vrcp(rho);
        v0 = u[1] * ri;
        v1 = u[2] * ri;
        v2 = u[3] * ri;
        const V kin = half * vfma(u[3], v2, vfma(u[2], v1, u[1] * v0));
        const V bb2 = bb[2] * bb[2];
        const V bt = vfma(bb[1], bb[1], bb2);
        const V bn = bb[0] * bb[0];
        mag = half * (bn + bt);
        p = gm1 * eint_comp(u[4], kin, mag);
        a2 = gamma * p * ri;
        bn2 = bn * ri;
        bt2 = bt * ri;
    }
    V ptot;
    if constexpr (VT<V>::F64) ptot = __fma_rn(0.5, mag, p);
    else ptot = p + mag;
    const V B2 = bn2 + bt2;
    V disc;
    if constexpr (VT<V>::F64) disc = __fma_rn(4.0, a2 * bt2, (a2 - B2) * (a2 - B2));
    else disc = vfma(a2 - B2, a2 - B2, vb<V>(4.0f) * a2 * bt2);
    c.cf = vsqrt(vb<V>(0.5f) * (a2 + B2 + vsqrt(disc)));
    c.cs = vsqrt(a2);
    c.p = p;
    c.vn = v0;
    c.d = vabs(v0) + c.cf;
    if constexpr (VT<V>::F64) {
        const V bv = bb[0] * v0 + bb[1] * v1 + bb[2] * v2;
        c.F[0] = u[1];
        c.F[1] = u[1] * v0 + ptot - bb[0] * bb[0];
        c.F[2] = u[2] * v0 - bb[0] * bb[1];
        c.F[3] = u[3] * v0 - bb[0] * bb[2];
        c.F[4] = (u[4] + ptot) * v0 - bb[0] * bv;
    } else {
        const V bv = vfma(bb[2], v2, vfma(bb[1], v1, bb[0] * v0));
        const V nb0 = -bb[0];
        c.F[0] = u[1];
        c.F[1] = vfma(nb0, bb[0], vfma(u[1], v0, ptot));
        c.F[2] = vfma(nb0, bb[1], u[2] * v0);
        c.F[3] = vfma(nb0, bb[2], u[3] * v0);
        c.F[4] = vfma(nb0, bv, (u[4] + ptot) * v0);
    }
    if constexpr (VT<V>::F64) {
        if (nonpos64(rho)) k.hi |= FLAG_RHO;
        if (nonpos64(p)) k.hi |= FLAG_P;
        if ((__double2hiint(c.cf) & 0x7fffffff) > 0x7ff00000) k.hi |= FLAG_NAN;
    } else {
        k.mn_rho = vmin(k.mn_rho, rho);
        k.mn_p = vmin(k.mn_p, p);
        k.nsum = k.nsum + c.cf;
    }
}

// Potential difference phi_b - phi_a across the interface a|b.  FP64 takes
// the difference of the cell potentials; the FP32 kernels read, per cell,
// the difference to the next cell along the sweep (formed in FP64 when the
// potential is set), so phia already holds phi_b - phi_a.
template <class V> __device__ __forceinline__ V pdiff(V phia, V phib)
{
    if constexpr (VT<V>::F64) return phib - phia;
    else return phia;
}

// hydrostatic estimate g (eq0321) and the HSE-corrected difference (eq0323).
// FP32 island: g = s * fac is split into its rounded value and the exact
// rounding error (TwoProduct with an FMA), both subtracted from du, so the
// cancellation du - g near equilibrium adds no product rounding.
template <class V>
__device__ __forceinline__ void chse(const CCell<V> &a, const CCell<V> &b, V phia, V phib, V du[5], V ddu[5])
{
    // -g = (xi_a + xi_b)/2 fac with xi = -(rho, m, E + p); the factor 1/2 goes
    // into fac (exact)
    const V fac = vb<V>(0.5f) * vdiv(pdiff(phia, phib), a.cs * b.cs);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const V s = i < 4 ? b.u[i] + a.u[i] : (b.u[4] + b.p) + (a.u[4] + a.p);
        du[i] = b.u[i] - a.u[i];
        if constexpr (VT<V>::F64) {
            ddu[i] = vminmod(du[i] + s * fac, du[i]);
        } else {
            const V ghi = s * fac;
            const V glo = vfma(s, fac, -ghi);
            ddu[i] = vminmod((du[i] + ghi) + glo, du[i]);
        }
    }
}

// first-order interface flux: eq0140 with D = alpha max(d_a, d_b) (eq0150),
// or the HSE-corrected form eq0324 (reading C-3).  Fluxes are carried doubled:
// the 1/2 of the mean and of the dissipation, exact, goes into dt/dx.
constexpr double FLUX_SCALE = 0.5;
template <class V, bool HSE>
__device__ __forceinline__ void cflux1(const CCell<V> &a, const CCell<V> &b, V phia, V phib, V alpha, V F[5])
{
    if constexpr (!HSE) {
        const V D = alpha * vmax(a.d, b.d);
        if constexpr (VT<V>::F64) {
#pragma unroll
            for (int i = 0; i < 5; ++i) F[i] = (a.F[i] + b.F[i]) - D * (b.u[i] - a.u[i]);
        } else {
#pragma unroll
            for (int i = 0; i < 5; ++i) F[i] = vfma(-D, b.u[i] - a.u[i], a.F[i] + b.F[i]);
        }
    } else {
        V du[5], ddu[5];
        const V Dadv = alpha * vmax(vabs(a.vn), vabs(b.vn));
        const V Dac = alpha * vmax(a.cf, b.cf);
        chse(a, b, phia, phib, du, ddu);
#pragma unroll
        for (int i = 0; i < 5; ++i) F[i] = vfma(-Dac, ddu[i], vfma(-Dadv, du[i], a.F[i] + b.F[i]));
    }
}

// second-order TVD flux at the interface c1|c2 from predicted cells c0..c3
// (eq0160-eq0230; one freezing speed per interface, reading C-2; HSE form of
// the slope differences, reading C-19, from the jumps du, dd of chse at the
// three interfaces of the stencil).  The hybrid limiter is taken only by
// the one-column kernels with the limiter read at run time.
// NU (irregular mesh, reading C-25): each one-sided difference is divided
// by the distance of the centres it joins and the limited slope carried
// over half the width of its own cell (w1 for F+, w2 for F-).
template <class V, bool HSE, int LIM, bool NU = false>
__device__ __forceinline__ void cflux2(const CCell<V> &c0, const CCell<V> &c1, const CCell<V> &c2, const CCell<V> &c3,
                                       const V du0[5], const V dd0[5], const V du1[5], const V dd1[5],
                                       const V du2[5], const V dd2[5], V F[5], int lim, V w0 = V(), V w1 = V(),
                                       V w2 = V(), V w3 = V())
{
    V gl = w0, gc = w1, gr = w2;
    if constexpr (NU) {
        const V half = vb<V>(0.5f);
        gl = half * (w0 + w1);
        gc = half * (w1 + w2);
        gr = half * (w2 + w3);
    }
    if constexpr (LIM < 0 && VT<V>::W == 1) {
        // hybrid limiter (Sec. 2.2): minmod where either cell of the
        // interface moves faster than its sound speed, else Van Leer (reading C-21)
        if (lim == LIM_HYBRID)
            lim = (vabs(c1.vn) > c1.cs || vabs(c2.vn) > c2.cs) ? LIM_MINMOD : LIM_VANLEER;
    }
    // compile-time hybrid (LIM = LIM_HYBRID, packed kernels): per lane,
    // sup > 0 where either cell is supersonic (|v| - c_S > 0 iff |v| > c_S)
    V sup = vb<V>(0.0f);
    if constexpr (LIM == LIM_HYBRID) sup = vmax(vabs(c1.vn) - c1.cs, vabs(c2.vn) - c2.cs);
    if constexpr (!HSE && !VT<V>::F64) {
        // FP32: 2 F = F_e + F_{e+1} - D du_e + [phi(+) - phi(-)]/2 with the
        // split-flux slopes written as dF +- D du (each one multiply-add)
        const V D = vmax(c1.d, c2.d);
        const V nD = -D;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const V df0 = c1.F[i] - c0.F[i], du0 = c1.u[i] - c0.u[i];
            const V df1 = c2.F[i] - c1.F[i], du1 = c2.u[i] - c1.u[i];
            const V df2 = c3.F[i] - c2.F[i], du2 = c3.u[i] - c2.u[i];
            V slp, slm;
            if constexpr (NU) {
                slp = w1 * vlimit_half<LIM>(vdiv(vfma(D, du0, df0), gl), vdiv(vfma(D, du1, df1), gc), lim);
                slm = w2 * vlimit_half<LIM>(vdiv(vfma(nD, du1, df1), gc), vdiv(vfma(nD, du2, df2), gr), lim);
            } else if constexpr (LIM == LIM_HYBRID) {
                const V ap = vfma(D, du0, df0), bp = vfma(D, du1, df1);
                const V am = vfma(nD, du1, df1), bm = vfma(nD, du2, df2);
                slp = vsel_pos(sup, vhalf(vminmod(ap, bp)), vvanleer_half(ap, bp));
                slm = vsel_pos(sup, vhalf(vminmod(am, bm)), vvanleer_half(am, bm));
            } else {
                slp = vlimit_half<LIM>(vfma(D, du0, df0), vfma(D, du1, df1), lim);
                slm = vlimit_half<LIM>(vfma(nD, du1, df1), vfma(nD, du2, df2), lim);
            }
            F[i] = vfma(nD, du1, c1.F[i] + c2.F[i]) + (slp - slm);
        }
    } else if constexpr (!HSE) {
        const V D = vmax(c1.d, c2.d);
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            // twice the split fluxes F+ and F- (eq0130)
            const V d1 = D * c1.u[i], d2 = D * c2.u[i];
            const V fp0 = c0.F[i] + D * c0.u[i];
            const V fp1 = c1.F[i] + d1;
            const V fp2 = c2.F[i] + d2;
            const V fm1 = c1.F[i] - d1;
            const V fm2 = c2.F[i] - d2;
            const V fm3 = c3.F[i] - D * c3.u[i];
            V slp, slm;  // half of twice the limited slopes
            if constexpr (NU) {
                slp = w1 * vlimit_half<LIM>((fp1 - fp0) / gl, (fp2 - fp1) / gc, lim);
                slm = w2 * vlimit_half<LIM>((fm2 - fm1) / gc, (fm3 - fm2) / gr, lim);
            } else {
                slp = vlimit_half<LIM>(fp1 - fp0, fp2 - fp1, lim);
                slm = vlimit_half<LIM>(fm2 - fm1, fm3 - fm2, lim);
            }
            F[i] = fp1 + fm2 + (slp - slm);
        }
    } else {
        const V Dadv = vmax(vabs(c1.vn), vabs(c2.vn));
        const V Dac = vmax(c1.cf, c2.cf);
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const V q0 = Dadv * du0[i] + Dac * dd0[i];
            const V q1 = Dadv * du1[i] + Dac * dd1[i];
            const V q2 = Dadv * du2[i] + Dac * dd2[i];
            // twice the one-sided differences of F+ and F-, and half their limited slopes
            const V fp_l = (c1.F[i] - c0.F[i]) + q0;
            const V fp_r = (c2.F[i] - c1.F[i]) + q1;
            const V fm_l = (c2.F[i] - c1.F[i]) - q1;
            const V fm_r = (c3.F[i] - c2.F[i]) - q2;
            V slp, slm;
            if constexpr (NU) {
                slp = w1 * vlimit_half<LIM>(vdiv(fp_l, gl), vdiv(fp_r, gc), lim);
                slm = w2 * vlimit_half<LIM>(vdiv(fm_l, gc), vdiv(fm_r, gr), lim);
            } else {
                slp = vlimit_half<LIM>(fp_l, fp_r, lim);
                slm = vlimit_half<LIM>(fm_l, fm_r, lim);
            }
            F[i] = (c1.F[i] + c2.F[i]) - q1 + (slp - slm);
        }
    }
}

// Largest (|v_a| + c_F,a) / h_a over the three axes of the frame (eq0083-
// eq0084, reading C-15) for a cell with conserved state u and cell-centred
// field b; the primitives are shared between the axes (FP32 path).
template <class V>
__device__ __forceinline__ V cfl_rate3(const V u[5], const V b[3], V gamma, V gm1, const V rh[3])
{
    const V half = vb<V>(0.5f);
    const V ri = vrcp(u[0]);
    const V v0 = u[1] * ri, v1 = u[2] * ri, v2 = u[3] * ri;
    const V kin = half * vfma(u[3], v2, vfma(u[2], v1, u[1] * v0));
    const V q0 = b[0] * b[0], q1 = b[1] * b[1], q2 = b[2] * b[2];
    const V mag = half * (q0 + q1 + q2);
    const V p = gm1 * eint_comp(u[4], kin, mag);
    const V a2 = gamma * p * ri;
    const V B2 = (q0 + q1 + q2) * ri;
    const V am = a2 - B2;
    const V c0 = am * am;
    const V aB = a2 + B2;
    const V f4a2 = vb<V>(4.0f) * a2;
    const V r0 = (vabs(v0) + vsqrt(half * (aB + vsqrt(vfma(f4a2, (q1 + q2) * ri, c0))))) * rh[0];
    const V r1 = (vabs(v1) + vsqrt(half * (aB + vsqrt(vfma(f4a2, (q0 + q2) * ri, c0))))) * rh[1];
    const V r2 = (vabs(v2) + vsqrt(half * (aB + vsqrt(vfma(f4a2, (q0 + q1) * ri, c0))))) * rh[2];
    return vmax(vmax(r0, r1), r2);
}

// ---------------------------------------------------------------------------
// L_d: fluid column march
// ---------------------------------------------------------------------------
template <class V> struct FRaw {
    V u[5];
    V bd;      // b_d at the cell's own (upper) face
    V bdm;     // b_d at the lower face
    V bf;      // fast-axis transverse face field at the cell's own faces
    V bo, bom; // other-axis transverse face field at own / lower face
    V phi;
    typename VT<V>::S bfm;  // fast-axis field at the face below the first column
    typename VT<V>::S w;    // cell width along d (irregular mesh; the same for all columns of a group)
};

template <class V> struct FMarch {
    FRaw<V> R;           // raw input of the next cell (prefetched)
    CCell<V> C[2];       // evaluated raw cells r-1, r (slot r & 1)
    V bb[2][3];          // their cell-centred field
    V ph[2];             // their potential
    V F1[2][5];          // predictor fluxes at (r-2, r-1), (r-1, r)
    CCell<V> P[4];       // predicted cells (slot index mod 4)
    V q[4];              // their potential
    V F2[2][5];          // corrector fluxes
    V hu[2][5], hd[2][5];  // HSE: jumps of the predicted cells at (r-3, r-2), (r-2, r-1) (slot r & 1)
    V phm2;              // potential of raw cell r-2
    Checks<V> chk;
    V cflr;              // largest CFL rate of the output cells (CFLF)
    typename VT<V>::S w0, w1, w2, w3, w4;  // irregular mesh: widths of raw cells r, r-1, .. r-4
    V dprev;             // split gravity: potential (FP64) or its difference (FP32) of raw cell r-1
};

// stride along the sweep as an IX (AR: the argument type, ColFluidArgs or
// ColCTArgs or, in the batch, a view with their members)
template <class IX, class AR> __device__ __forceinline__ IX ix_sd(const AR &A)
{
    return (IX)A.sd * ix_unit<typename AR::Real, IX>();
}

// IX: how elements are addressed, long long indices or (unsigned) 32-bit byte
// offsets where all fit.
template <class S, class IX = long long> struct FCtx {
    IX base;             // offset of cell 0 of the first column
    IX ofm;              // offset of the fast-axis face below the first column
    IX oom;              // offset of the other-axis face below (mapped)
};

// L2 prefetch of one cell of a warp's march with a single instruction: lane
// l takes field row l / 2 (u0..u4, b_d, b_f, b_o, b_o of the row below, the
// potential) and the (l % 2)-th 128-byte line of the warp's span of it in
// cell 0, shifted by whole cells along the sweep (when the stride along the
// sweep is not a multiple of a line the lines drift by less than one line:
// it is a hint).
#ifndef FISH_FL_PF_WARP
#define FISH_FL_PF_WARP 1
#endif
template <class S, class IX> struct FPf {
    const S *p;   // the lane's line in cell 0 (nullptr: lane idle); cell c: p + c * sd
};

template <class S, class IX, class AR>
__device__ __forceinline__ void fpf_setup(const AR &A, const S *bfp, const S *bop, IX base0, IX oom0,
                                          int span, bool grav, int lane, FPf<S, IX> &P)
{
    P.p = nullptr;
    const int r = lane >> 1;
    if (r >= (grav ? 10 : 9)) return;
    const S *f = r < 5 ? A.u[r] : (r == 5 ? A.bd : (r == 6 ? bfp : (r == 9 ? A.phi : bop)));
    const IX r0 = base0 + (r == 8 ? oom0 : (IX)0);
    constexpr IX un = ix_unit<S, IX>();
    const IX line = (r0 & ~((IX)31 * un)) + (IX)(32 * (lane & 1)) * un;
    if (line <= r0 + (IX)(span - 1) * un) P.p = ix_at(f, line);
}

template <class S, class IX, class AR>
__device__ __forceinline__ void fpf_step(const AR &A, const FPf<S, IX> &P, int c)
{
    if (P.p) pf_l2(ix_at(P.p, (IX)c * ix_sd<IX>(A)));
}

// load raw cell s (any s): every index through the boundary map; a ghost
// cell copies the mapped cell as a whole, its lower b_d face included
template <class V, bool GRAV, bool FT1, class IX = long long, class AR>
__device__ __forceinline__ void fload_mapped(const AR &A,
                                             const FCtx<typename VT<V>::S, IX> &X, int s, FRaw<V> &R)
{
    const int cc = gmap(s, A.n, A.bc);
    const IX i = X.base + (IX)cc * ix_sd<IX>(A);
    const IX im = X.base + (IX)gmap(cc - 1, A.n, A.bc) * ix_sd<IX>(A);
    const auto *bfp = FT1 ? A.bt1 : A.bt2;
    const auto *bop = FT1 ? A.bt2 : A.bt1;
#pragma unroll
    for (int k = 0; k < 5; ++k) R.u[k] = vget_at<V>(A.u[k], i);
    R.bd = vget_at<V>(A.bd, i);
    R.bdm = vget_at<V>(A.bd, im);
    R.bf = vget_at<V>(bfp, i);
    R.bfm = __ldg(ix_at(bfp, i + X.ofm));
    R.bo = vget_at<V>(bop, i);
    R.bom = vget_at<V>(bop, i + X.oom);
    if (GRAV) {
        // FP32 reads the difference to the next cell: zero between the copies
        // of an outflow boundary cell (and across its face)
        R.phi = vget_at<V>(A.phi, i);
        if constexpr (!VT<V>::F64)
            if (A.bc == BC_OUTFLOW && (s < 0 || s >= A.n)) R.phi = vb<V>(0.0f);
    }
    // a ghost has the width of the cell it copies (reading C-23)
    if (A.wd) R.w = A.wd[cc];
}

// Cell of the box that raw cell c stands for (c up to four cells outside the
// box, which may be thinner than that).
__device__ __forceinline__ int wrap_cell(int c, int n, int bc)
{
    if ((unsigned)c < (unsigned)n) return c;
    if (bc == BC_PERIODIC) {
        while (c < 0) c += n;
        while (c >= n) c -= n;
        return c;
    }
    return c < 0 ? 0 : n - 1;
}

// Load raw cell c, the one after the cell whose raw data R holds: its lower
// b_d face is that cell's upper one, and for the ghosts above an outflow box,
// which copy cell n-1 as a whole, that of cell n-1.
template <class V, bool PHI, bool FT1, bool NU, class IX = long long, class AR>
__device__ __forceinline__ void fload_next(const AR &A,
                                           const FCtx<typename VT<V>::S, IX> &X, int c, FRaw<V> &R)
{
    const auto *bfp = FT1 ? A.bt1 : A.bt2;
    const auto *bop = FT1 ? A.bt2 : A.bt1;
    const int cc = wrap_cell(c, A.n, A.bc);
    const IX i = X.base + (IX)cc * ix_sd<IX>(A);
    if (!(c >= A.n && A.bc == BC_OUTFLOW)) R.bdm = R.bd;
#pragma unroll
    for (int k = 0; k < 5; ++k) R.u[k] = vget_at<V>(A.u[k], i);
    R.bd = vget_at<V>(A.bd, i);
    R.bf = vget_at<V>(bfp, i);
    R.bfm = __ldg(ix_at(bfp, i + X.ofm));
    R.bo = vget_at<V>(bop, i);
    R.bom = vget_at<V>(bop, i + X.oom);
    if constexpr (PHI) {
        R.phi = vget_at<V>(A.phi, i);
        if constexpr (!VT<V>::F64)
            if (c != cc && A.bc == BC_OUTFLOW) R.phi = vb<V>(0.0f);
    }
    if constexpr (NU) R.w = A.wd[cc];
}

// L2 prefetch distance of the fluid march (cells ahead of the load): four in
// long segments (2552 -> 2513 us at 640^3), two in short ones, which belong to
// boxes that fit in L2 and would fetch the next segment's cells.
__device__ __forceinline__ int pf_dist(int len) { return len >= 96 ? 4 : 2; }

#ifndef FISH_FL_PF_NEIGH
#define FISH_FL_PF_NEIGH 1   // also the lower other-axis face (a neighbour row)
#endif
// prefetch into L2 the fields the fluid march will load for interior cell i
template <class V, bool GRAV, bool FT1, class IX = long long, class AR>
__device__ __forceinline__ void fprefetch(const AR &A,
                                          const FCtx<typename VT<V>::S, IX> &X, IX i)
{
    const auto *bfp = FT1 ? A.bt1 : A.bt2;
    const auto *bop = FT1 ? A.bt2 : A.bt1;
#pragma unroll
    for (int k = 0; k < 5; ++k) pf_l2(ix_at(A.u[k], i));
    pf_l2(ix_at(A.bd, i));
    pf_l2(ix_at(bfp, i));
    pf_l2(ix_at(bop, i));
#if FISH_FL_PF_NEIGH
    pf_l2(ix_at(bop, i + X.oom));
#endif
    if (GRAV) pf_l2(ix_at(A.phi, i));
}

// Stages of a march step: the evaluation of the raw cell alone, with the
// predictor flux behind it, or everything.
enum : int { ST_RAW = 0, ST_FLUX = 1, ST_ALL = 2 };
// (stage flags of the ring march)
enum : int { ST_F1 = 1, ST_PRED = 2, ST_F2 = 4, ST_OUT = 8 };

// Operator-split gravity kick G_d(tau) of one cell (eq02512, reading C-22):
// m_d -= tau rho dphi, E changes by the kinetic energy change; FP64 in the
// oracle's operation order.
template <class V> __device__ __forceinline__ void sg_kick(V u[5], V dk, V tau)
{
    if constexpr (VT<V>::F64) {
        const V mo = u[1];
        const V mn = mo - tau * u[0] * dk;
        u[1] = mn;
        u[4] = u[4] + 0.5 * (mn * mn - mo * mo) / u[0];
    } else {
        const V mo = u[1];
        const V dm = -(tau * u[0]) * dk;
        u[1] = mo + dm;
        const V dE = dm * vfma(vb<V>(0.5f), dm, mo);
        // (one column: the quotient unrounded in the sum, as earlier versions had it)
        if constexpr (VT<V>::W == 1) u[4] = vfma(dE, vrcp(u[0]), u[4]);
        else u[4] = u[4] + vdiv(dE, u[0]);
    }
}

// Centred potential difference (eq02513) of the image cell of ghost r (its
// copy along d): FP64 from the potential, FP32 from the stored differences
// D_c = phi_{c+1} - phi_c (D_{-1} = 0 at an outflow boundary).
template <class V, class IX = long long, class AR>
__device__ __forceinline__ V sg_image_dk(const AR &A,
                                         const FCtx<typename VT<V>::S, IX> &X, int r, V rtwoh)
{
    const int cc = gmap(r, A.n, A.bc);
    if constexpr (VT<V>::F64) {
        const V pp = vget_at<V>(A.phi, X.base + (IX)gmap(cc + 1, A.n, A.bc) * ix_sd<IX>(A));
        const V pm = vget_at<V>(A.phi, X.base + (IX)gmap(cc - 1, A.n, A.bc) * ix_sd<IX>(A));
        return (pp - pm) / (2.0 * A.h);
    } else {
        const V dc = vget_at<V>(A.phi, X.base + (IX)cc * ix_sd<IX>(A));
        V dl = vb<V>(0.0f);
        if (cc > 0 || A.bc == BC_PERIODIC) dl = vget_at<V>(A.phi, X.base + (IX)gmap(cc - 1, A.n, A.bc) * ix_sd<IX>(A));
        return (dc + dl) * rtwoh;
    }
}

// GM: gravity mode, 0 none, 1 unsplit source terms (eq0253-eq0255), 2
// operator-split kicks G_d(dt/2) folded into the march (eq025111): the raw
// cell is kicked as it is consumed, the output cell's old state before its
// update and the result after it (reading C-22 for the kick).
// The ring of the packed kernels with the CFL epilogue (blocks of 128
// threads): the cell-centred fields of a thread's raw cells r .. r-3, slot
// r mod 4, component k at [(slot * 3 + k) * 128 + thread]; only the kernels
// that use it allocate it.
static __shared__ float2 cfl_bb_ring[4 * 3 * 128];

// One step of the march for raw cell r (K = slot of cell r in the windows).
// The raw data of cell r is in M.R on entry (loaded by the previous step); the
// step loads raw cell r+1 into M.R.  a: first output cell of the segment, so
// that cell r-3 is an output cell from r = a+3 on.  FT1: the fast axis is t1
// (else t2).  NU: irregular mesh along d (eq037): the cells' own widths
// replace h (the widths of raw cells r .. r-4 ride along in M.w0 .. M.w4).
template <class V, bool HSE, int GM, int LIM, bool FT1, bool CFLF, bool NU, int K, int ST, class IX = long long,
          bool PFW = FISH_FL_PF_WARP != 0, class AR>
__device__ __forceinline__ void fstep(const AR &A, const FCtx<typename VT<V>::S, IX> &X,
                                      FMarch<V> &M, int r, int a, int pfd, V lam, V lamh, V hdt, V dt, V rtwoh,
                                      const FPf<typename VT<V>::S, IX> &PF)
{
    constexpr bool GRAV = GM == 1, SG = GM == 2, PHI = GM != 0;
    constexpr int k2 = K & 1, p2 = (K + 1) & 1;
    const V half = vb<V>(0.5f);
    // consume the raw input of cell r
    V bbr[3];
    V ur[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) ur[k] = M.R.u[k];
    bbr[0] = half * (M.R.bdm + M.R.bd);
    const V bfc = half * (vshift_lo(M.R.bfm, M.R.bf) + M.R.bf);
    const V boc = half * (M.R.bom + M.R.bo);
    if constexpr (FT1) {
        bbr[1] = bfc;
        bbr[2] = boc;
    } else {
        bbr[1] = boc;
        bbr[2] = bfc;
    }
    const V phr = PHI ? M.R.phi : vb<V>(0.0f);  // no potential: phi = 0
    if constexpr (CFLF) {
        // keep the cell-centred field of raw cell r for the CFL rate of its
        // update three steps later (b is unchanged by L_d)
        static_assert(VT<V>::W == 2, "the CFL epilogue is built for the packed kernels");
        const int t = threadIdx.x & 127;
#pragma unroll
        for (int k = 0; k < 3; ++k) cfl_bb_ring[((K & 3) * 3 + k) * 128 + t] = bbr[k].v;
    }
    if constexpr (NU) {
        M.w4 = M.w3;
        M.w3 = M.w2;
        M.w2 = M.w1;
        M.w1 = M.w0;
        M.w0 = M.R.w;
    }
    // load raw cell r+1
    fload_next<V, PHI, FT1, NU, IX>(A, X, r + 1, M.R);
    if constexpr (ST == ST_ALL) {
        const int pf = min(r + 1 + pfd, A.n - 1);
        if constexpr (PFW) fpf_step(A, PF, pf);
        else fprefetch<V, PHI, FT1, IX>(A, X, X.base + (IX)pf * ix_sd<IX>(A));
    }
    // old state of the output cell o = r-3
    const int o = r - 3;
    const bool out = ST == ST_ALL && o >= a;
    const IX io = X.base + (IX)o * ix_sd<IX>(A);
    V un[5];
    if constexpr (ST == ST_ALL) {
#pragma unroll
        for (int k = 0; k < 5; ++k) un[k] = ur[k];
        if (out) {
#pragma unroll
            for (int k = 0; k < 5; ++k) un[k] = vget_at<V>(A.u[k], io);
        }
    }
    if constexpr (SG) {
        // kick of raw cell r with its centred potential difference (a ghost
        // takes its image cell's), and of the output cell's old state
        V dk;
        if (A.bc == BC_OUTFLOW && (r < 0 || r >= A.n)) {
            dk = sg_image_dk<V, IX>(A, X, r, rtwoh);
        } else if constexpr (VT<V>::F64) {
            dk = (M.R.phi - M.dprev) / (2.0 * A.h);  // phi_{r+1} - phi_{r-1}
        } else {
            dk = (phr + M.dprev) * rtwoh;            // D_r + D_{r-1}
        }
        M.dprev = phr;
        sg_kick<V>(ur, dk, hdt);
        M.ph[k2] = dk;
        if constexpr (ST == ST_ALL) sg_kick<V>(un, M.q[(K + 1) & 3], hdt);
    }
    ceval<V>(ur, bbr, vb<V>(A.gamma), vb<V>(A.gm1), M.C[k2], M.chk);
#pragma unroll
    for (int k = 0; k < 3; ++k) M.bb[k2][k] = bbr[k];
    if (!SG && (GRAV || HSE)) M.ph[k2] = phr;
    if constexpr (ST >= ST_FLUX) {
        // predictor flux at (r-1, r) (eq0140 / eq0324)
        cflux1<V, HSE>(M.C[p2], M.C[k2], M.ph[p2], phr, vb<V>(A.alpha), M.F1[k2]);
    }
    if constexpr (ST == ST_ALL) {
        // predicted half step of cell r-1 (eq0253; source eq0254, reading C-6)
        const CCell<V> &cp = M.C[p2];
        V up[5];
        V lh = lamh;
        if constexpr (NU) {
            if constexpr (VT<V>::F64) lh = FLUX_SCALE * (dt / (2.0 * M.w1));
            else lh = vdiv(vb<V>(0.5f) * hdt, vb<V>(M.w1));
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            if constexpr (VT<V>::F64) up[k] = cp.u[k] - lh * (M.F1[k2][k] - M.F1[p2][k]);
            else up[k] = vfma(-lh, M.F1[k2][k] - M.F1[p2][k], cp.u[k]);
        }
        if (GRAV) {
            // centred difference phi_r - phi_{r-2} (eq02513; NU: over the
            // centre span, reading C-26)
            V dphi;
            if constexpr (NU) {
                const V span = vb<V>(0.5f) * vb<V>(M.w2) + vb<V>(M.w1) + vb<V>(0.5f) * vb<V>(M.w0);
                if constexpr (VT<V>::F64) dphi = (phr - M.phm2) / span;
                else dphi = vdiv(M.ph[p2] + M.phm2, span);
            } else if constexpr (VT<V>::F64) {
                dphi = (phr - M.phm2) / (2.0 * A.h);
            } else {
                dphi = (M.ph[p2] + M.phm2) * rtwoh;
            }
            up[1] = up[1] - hdt * cp.u[0] * dphi;
            up[4] = up[4] - hdt * cp.u[1] * dphi;
        }
        constexpr int s3 = (K + 3) & 3;  // slot of cell r-1
        ceval<V>(up, M.bb[p2], vb<V>(A.gamma), vb<V>(A.gm1), M.P[s3], M.chk);
        if (PHI || HSE) M.q[s3] = M.ph[p2];
        // corrector flux at (r-3, r-2) from predicted cells r-4 .. r-1 (eq0230)
        constexpr int s0 = K & 3, s1 = (K + 1) & 3, s2 = (K + 2) & 3;
        // (the jumps of its two older interfaces are those of the last two steps)
        V du2[5], dd2[5];
        if constexpr (HSE) chse(M.P[s2], M.P[s3], M.q[s2], M.q[s3], du2, dd2);
        if (!VT<V>::F64 || r >= a + 2)  // (FP64, bound by its pipe, skips the fluxes no output cell uses)
            cflux2<V, HSE, LIM, NU>(M.P[s0], M.P[s1], M.P[s2], M.P[s3], M.hu[k2], M.hd[k2], M.hu[p2], M.hd[p2], du2,
                                    dd2, M.F2[k2], A.lim, vb<V>(M.w4), vb<V>(M.w3), vb<V>(M.w2), vb<V>(M.w1));
        if constexpr (HSE) {
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                M.hu[k2][k] = du2[k];
                M.hd[k2][k] = dd2[k];
            }
        }
        V lo = lam;
        if constexpr (NU) {
            if constexpr (VT<V>::F64) lo = FLUX_SCALE * (dt / M.w3);
            else lo = vdiv(hdt, vb<V>(M.w3));
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            if constexpr (VT<V>::F64) un[k] = un[k] - lo * (M.F2[k2][k] - M.F2[p2][k]);
            else un[k] = vfma(-lo, M.F2[k2][k] - M.F2[p2][k], un[k]);
        }
        if (GRAV) {
            // corrector source from the predicted state (eq0255)
            V dphi;
            if constexpr (NU) {
                const V span = vb<V>(0.5f) * vb<V>(M.w4) + vb<V>(M.w3) + vb<V>(0.5f) * vb<V>(M.w2);
                if constexpr (VT<V>::F64) dphi = (M.q[s2] - M.q[s0]) / span;
                else dphi = vdiv(M.q[s0] + M.q[s1], span);
            } else if constexpr (VT<V>::F64) {
                dphi = (M.q[s2] - M.q[s0]) / (2.0 * A.h);
            } else {
                dphi = (M.q[s0] + M.q[s1]) * rtwoh;
            }
            un[1] = un[1] - dt * M.P[s1].u[0] * dphi;
            un[4] = un[4] - dt * M.P[s1].u[1] * dphi;
        }
        if constexpr (SG) sg_kick<V>(un, M.q[s1], hdt);  // output cell: second half kick
        if (out) {
#pragma unroll
            for (int k = 0; k < 5; ++k) vstore(ix_at(A.uo[k], io), 0, un[k]);
            if constexpr (CFLF) {
                // CFL rate of the updated cell with its cell-centred field,
                // formed when the cell entered as raw cell o = r-3 (slot
                // (r-3) mod 4 of the ring)
                V bc[3];
                const int t = threadIdx.x & 127;
#pragma unroll
                for (int k = 0; k < 3; ++k) bc[k].v = cfl_bb_ring[(((K + 1) & 3) * 3 + k) * 128 + t];
                const V rh[3] = {vb<V>(A.rh[0]), vb<V>(A.rh[1]), vb<V>(A.rh[2])};
                M.cflr = vmax(M.cflr, cfl_rate3<V>(un, bc, vb<V>(A.gamma), vb<V>(A.gm1), rh));
            }
        }
    }
    if (GRAV) M.phm2 = M.ph[p2];
}

#ifndef FISH_COL_MINB
#define FISH_COL_MINB 2
#endif
#ifndef FISH_COL_MINB1
#define FISH_COL_MINB1 3   // one-column FP32 kernels
#endif

// The march of thread cid (column group cid of the box described by A) over
// the output cells a .. b-1.
// PFW: L2 prefetch of the next cells by one instruction per warp over the
// warp's span of its first row (the single-box sweeps, whose rows hold a
// multiple of 32 column groups), or per lane and field (the batch, whose
// short rows leave warps that straddle two rows)
template <class V, bool HSE, int GRAV, int LIM, bool FT1, bool CFLF, bool NU = false, class IX = long long,
          bool PFW = FISH_FL_PF_WARP != 0, class AR>
__device__ __forceinline__ void fluid_columns(const AR &A, long long cid, int a, int b)
{
    using S = typename VT<V>::S;
    constexpr int W = VT<V>::W;
    const int cols = A.nf / W;
    if (cid >= (long long)cols * A.no) return;
    const int fp = (int)(cid % cols), ob = (int)(cid / cols);
    const int f0 = fp * W;
    FCtx<S, IX> X;
    constexpr IX un = ix_unit<S, IX>();
    X.base = ((IX)A.off + (IX)f0 + (IX)ob * (IX)A.so) * un;
    X.ofm = (IX)(gmap(f0 - 1, A.nf, A.bc) - f0) * un;
    X.oom = (IX)(gmap(ob - 1, A.no, A.bc) - ob) * (IX)A.so * un;
    // per-warp L2 prefetch over the span of the warp's first lane (32 groups
    // of W columns; a warp that crosses a row end prefetches its first row)
    FPf<S, IX> PF;
    PF.p = nullptr;
    if constexpr (PFW) {
        const unsigned am = __activemask();
        const int l0 = __ffs(am) - 1;
        const IX b0 = __shfl_sync(am, X.base, l0);
        const IX m0 = __shfl_sync(am, X.oom, l0);
        const int span = min(32 * W, A.nf - (int)(b0 / un - (IX)A.off) % A.nf);
        fpf_setup(A, FT1 ? A.bt1 : A.bt2, FT1 ? A.bt2 : A.bt1, b0, m0, span, GRAV != 0, (int)(threadIdx.x & 31), PF);
    }
    const double dtd = *A.dt;
    const V dt = vb<V>(S(dtd));
    const V lam = vb<V>(S(FLUX_SCALE * (dtd / A.h)));
    const V lamh = vb<V>(S(FLUX_SCALE * (dtd / (2.0 * A.h))));
    const V hdt = vb<V>(S(0.5 * dtd));
    const V rtwoh = vb<V>(S(1.0 / (2.0 * A.h)));

    const int pfd = pf_dist(b - a);
    FMarch<V> M;
    checks_init(M.chk);
    const V zero = vb<V>(0.0f);
    M.cflr = M.phm2 = M.dprev = M.ph[0] = M.ph[1] = zero;
    M.w0 = M.w1 = M.w2 = M.w3 = M.w4 = typename VT<V>::S(1);
    // the windows behind the first output cell are zero until they fill: the
    // fluxes formed from them are not used
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        M.q[i] = zero;
        M.P[i].d = M.P[i].p = M.P[i].cs = M.P[i].cf = M.P[i].vn = zero;
#pragma unroll
        for (int k = 0; k < 5; ++k) M.P[i].u[k] = M.P[i].F[k] = M.F2[i & 1][k] = M.hu[i & 1][k] = M.hd[i & 1][k] = zero;
    }
    fload_mapped<V, GRAV != 0, FT1, IX>(A, X, a - 3, M.R);
    if constexpr (GRAV == 2) {
        // potential data of the cell before the first (its centred difference)
        FRaw<V> R0;
        fload_mapped<V, true, FT1, IX>(A, X, a - 4, R0);
        M.dprev = R0.phi;
    }
    if constexpr (PFW) {
        // the first cells, so that their loads do not each wait for memory
#pragma unroll
        for (int c = -2; c < 2; ++c) fpf_step(A, PF, max(min(a + c, A.n - 1), 0));
    }
    fstep<V, HSE, GRAV, LIM, FT1, CFLF, NU, 1, ST_RAW, IX, PFW>(A, X, M, a - 3, a, pfd, lam, lamh, hdt, dt, rtwoh, PF);
    fstep<V, HSE, GRAV, LIM, FT1, CFLF, NU, 2, ST_FLUX, IX, PFW>(A, X, M, a - 2, a, pfd, lam, lamh, hdt, dt, rtwoh, PF);
    const int last = b + 2;
#pragma unroll 1
    for (int r = a - 1;; r += 4) {
        fstep<V, HSE, GRAV, LIM, FT1, CFLF, NU, 3, ST_ALL, IX, PFW>(A, X, M, r, a, pfd, lam, lamh, hdt, dt, rtwoh, PF);
        if (r >= last) break;
        fstep<V, HSE, GRAV, LIM, FT1, CFLF, NU, 0, ST_ALL, IX, PFW>(A, X, M, r + 1, a, pfd, lam, lamh, hdt, dt, rtwoh, PF);
        if (r + 1 >= last) break;
        fstep<V, HSE, GRAV, LIM, FT1, CFLF, NU, 1, ST_ALL, IX, PFW>(A, X, M, r + 2, a, pfd, lam, lamh, hdt, dt, rtwoh, PF);
        if (r + 2 >= last) break;
        fstep<V, HSE, GRAV, LIM, FT1, CFLF, NU, 2, ST_ALL, IX, PFW>(A, X, M, r + 3, a, pfd, lam, lamh, hdt, dt, rtwoh, PF);
        if (r + 3 >= last) break;
    }
    const unsigned fl = checks_flags(M.chk);
    if (fl) atomicOr(A.flags, fl);
    if constexpr (CFLF) {
        // warp maximum of the rates (order-preserving bits of non-negative
        // floats), then one atomic minimum of 1/rate per warp
        float m = 0.0f;
#pragma unroll
        for (int i = 0; i < VT<V>::W; ++i) m = fmaxf(m, (float)vget(M.cflr, i));
        const unsigned mask = __activemask();
        const unsigned wm = __reduce_max_sync(mask, __float_as_uint(m));
        if ((threadIdx.x & 31) == __ffs(mask) - 1) {
            const float mx = __uint_as_float(wm);
            if (mx > 0.0f && mx == mx) {
                atomicMin(A.cfl_min, (unsigned long long)__double_as_longlong(1.0 / (double)mx));
            } else {
                atomicOr(A.flags, FLAG_NAN);
            }
        }
    }
}

// Threads of a block.  FP64 is bound by the FP64 pipe of each SM quarter,
// which one warp nearly fills, so its blocks are single warps that spread
// evenly (L_x of 72 x 60 x 51 cells: 215 us with one-warp blocks, 248 us with
// four-warp blocks, 942 us with the columns uncut).
template <class V> constexpr int fluid_threads() { return VT<V>::F64 ? 32 : 128; }
// Blocks per SM the kernels are compiled for.
template <class V, bool HSE> constexpr int fluid_resident()
{
    return VT<V>::F64 ? 8 : (VT<V>::W == 2 ? FISH_COL_MINB : FISH_COL_MINB1);
}

// Grid: column blocks x segments of `len` cells.
template <class V, bool HSE, int GRAV, int LIM, bool FT1, bool CFLF = false, bool NU = false, class IX = long long>
__global__ void __launch_bounds__(fluid_threads<V>(), fluid_resident<V, HSE>())
    fluid_col_kernel(const ColFluidArgs<typename VT<V>::S> A, int len)
{
    const int a = blockIdx.y * len;
    fluid_columns<V, HSE, GRAV, LIM, FT1, CFLF, NU, IX>(A, (long long)blockIdx.x * blockDim.x + threadIdx.x, a,
                                                        min(A.n, a + len));
}

// ---------------------------------------------------------------------------
// B_d: constrained transport column march (eq0330-eq0364, signs of C-5)
// ---------------------------------------------------------------------------
// Rolling state of one face pencil (windows indexed by cell s mod 4 or 2).
template <class V> struct CFace {
    V vt[4];   // face velocity (eq0361) at s
    V vh[4];   // smoothed velocity (eq0362) at s-1
    V bf[4];   // face field at s
    V w[2];    // cell product v b at s-1
    V dw[2];   // FP64: differences of the predicted products, w_{s-2} - w_{s-3} (slot s & 1)
    unsigned up;  // FP64: bit k: edge velocity > 0 at interface (s-2-k)'
    V f1[2];   // predictor flux at interface (s-2)'
    V wp[4];   // predicted product at s-2
    V f[2];    // corrector flux at interface (s-4)'
};

// Widths along d of cells s, s-1 .. s-5 (irregular mesh).
template <class V> struct CWid {
    V w0, w1, w2, w3, w4, w5;
};

// Sign of the edge velocity between cells a and b of a face pencil (eq0364):
// of the sum, or with NU of the linear interpolation to the interface (reading
// C-27), whose positive denominator is left out.
template <class V, bool NU> __device__ __forceinline__ V cedge(V va, V vb_, V wa, V wb)
{
    if constexpr (!NU) return va + vb_;
    else return vfma(wb, va, wa * vb_);
}

// B_d: the velocities a face pencil is advanced with are eight times the
// smoothed ones (the 1/2 of the mean eq0361 and the 1/4 of the smoothing eq0362
// are left out, exactly), and so are its products and fluxes; the factors dt/dx
// carry an eighth.
constexpr double CT_SCALE = 0.125;

// Advance a face pencil by cell s (K = s mod 4) with face velocity vt and
// field bf.  With OUT, bnew receives the updated face field of cell s-4 and
// f[K & 1] holds the corrector flux at (s-4)'.  NU: irregular mesh along d
// (widths in cw, eq037 and reading C-25/C-27; dt for the per-cell factors).
// fin: the newest product difference of a float pencil takes its product
// unrounded (see ct_rounding).
template <class V, int LIM, int K, bool OUT, bool NU = false>
__device__ __forceinline__ void cface(CFace<V> &P, V vt, V bf, V lamh, V lam, V &bnew, int lim, bool live,
                                      const CWid<V> &cw = CWid<V>(), V dt = V(), bool fin = false)
{
    constexpr int k1 = (K + 3) & 3, k2 = (K + 2) & 3, kp = (K + 1) & 3;
    constexpr int e = K & 1, o = (K + 1) & 1;
    if constexpr (VT<V>::F64) {
        // The upwind sides are kept as bits and the differences of the
        // predicted products in registers; the upwind operands are selected
        // before the one limiter.
        const V vh = __fma_rn(2.0, P.vt[k1], vt) + P.vt[k2];
        P.vh[k1] = vh;
        P.w[o] = vh * P.bf[k1];
        V vbar;
        if constexpr (NU) vbar = cw.w1 * P.vh[k2] + cw.w2 * vh;  // (positive weights over their sum: the sign)
        else vbar = P.vh[k2] + vh;
        const bool pos = pos64(vbar);
        P.up = P.up << 1 | (pos ? 1u : 0u);
        P.f1[e] = pos ? P.w[e] : P.w[o];
        V lh = lamh;
        if constexpr (NU) lh = CT_SCALE * (dt / (2.0 * cw.w2));
        const V bp = P.bf[k2] - lh * (P.f1[e] - P.f1[o]);
        P.wp[k2] = P.vh[k2] * bp;
        const V d2 = P.wp[k2] - P.wp[kp];
        if (live) {
            const bool u = (P.up & 4u) != 0;  // interface (s-4)'
            V la = u ? P.dw[e] : P.dw[o], lb = u ? P.dw[o] : d2;
            if constexpr (NU) {
                la = la / (0.5 * (u ? cw.w5 + cw.w4 : cw.w4 + cw.w3));
                lb = lb / (0.5 * (u ? cw.w4 + cw.w3 : cw.w3 + cw.w2));
            }
            V sl = vlimit_half<LIM>(la, lb, lim);
            if constexpr (NU) sl = (u ? cw.w4 : cw.w3) * sl;
            P.f[e] = (u ? P.wp[K] : P.wp[kp]) + (u ? sl : -sl);
            if constexpr (OUT) {
                V lo = lam;
                if constexpr (NU) lo = CT_SCALE * (dt / cw.w4);
                bnew = P.bf[K] - lo * (P.f[e] - P.f[o]);
            }
        }
        P.dw[e] = d2;
        P.bf[K] = bf;
        P.vt[K] = vt;
        return;
    }
    // smoothed face velocity at s-1 (eq0362) and the cell product w_{s-1}
    const V vh = vfma(vb<V>(2.0f), P.vt[k1], vt) + P.vt[k2];
    P.vh[k1] = vh;
    P.w[o] = vmul(vh, P.bf[k1]);
    {
        // first-order upwind flux at (s-2)' (eq0363, edge velocity eq0364;
        // tie v = 0 takes the right cell, reading C-7)
        const V vbar = cedge<V, NU>(P.vh[k2], vh, cw.w2, cw.w1);
        P.f1[e] = vsel_pos(vbar, P.w[e], P.w[o]);
    }
    V bp;
    {
        // predictor half step of the face field at s-2
        V lh = lamh;
        if constexpr (NU) lh = vdiv(vb<V>(float(0.5 * CT_SCALE)) * dt, cw.w2);
        bp = vfma(-lh, P.f1[e] - P.f1[o], P.bf[k2]);
        P.wp[k2] = vmul(P.vh[k2], bp);
    }
    {
        // corrector flux at q' = (s-4)': piecewise-linear TVD about the
        // upwind cell (reading C-10)
        const V vbar = cedge<V, NU>(P.vh[K], P.vh[kp], cw.w4, cw.w3);
        const V wm = P.wp[k1], w0 = P.wp[K], w1 = P.wp[kp], w2 = P.wp[k2];
        if constexpr (NU) {
            // slopes per unit length over the centre distances, carried over
            // half the upwind cell (reading C-25)
            const V half = vb<V>(0.5f);
            const V gl = half * (cw.w5 + cw.w4), gc = half * (cw.w4 + cw.w3), gr = half * (cw.w3 + cw.w2);
            {
                const V d1 = vdiv(w1 - w0, gc);
                const V dx = vdiv(vsel_pos(vbar, w0 - wm, w2 - w1), vsel_pos(vbar, gl, gr));
                const V base = vsel_pos(vbar, w0, w1);
                const V sg = vsel_pos(vbar, cw.w4, -cw.w3);
                P.f[e] = vfma(sg, vlimit_half<LIM>(d1, dx, lim), base);
            }
        } else {
            // the upwind side's operands, then one limiter: both sides limit
            // the middle difference against their outer one
            V d2 = w2 - w1;
            if constexpr (std::is_same<V, float>::value) d2 = fin ? fmaf(P.vh[k2], bp, -w1) : d2;
            const V dx = vsel_pos(vbar, w0 - wm, d2);
            const V base = vsel_pos(vbar, w0, w1);
            const V sg = vsel_pos(vbar, vb<V>(1.0f), vb<V>(-1.0f));
            P.f[e] = vfma(sg, vlimit_half<LIM>(w1 - w0, dx, lim), base);
        }
        if constexpr (OUT) {
            V lo = lam;
            if constexpr (NU) lo = vdiv(vb<V>(float(CT_SCALE)) * dt, cw.w4);
            bnew = vfma(-lo, P.f[e] - P.f[o], P.bf[K]);
        }
    }
    P.bf[K] = bf;
    P.vt[K] = vt;
}

// ---------------------------------------------------------------------------
// B_d column march.  A warp owns 31 W consecutive columns of one row of the
// other axis (lanes 1..31) plus a halo lane 0 holding the W columns below:
// every lane marches the face pencils above its columns along the fast axis
// (PF) and along the other axis (PO), and the pencil below along the other
// axis (PO-).  The fast-axis pencil below a column is the PF pencil of the
// lane beneath it, whose edge flux arrives by a warp shuffle.  Raw inputs of
// cell s+1 are loaded while cell s is computed.
// ---------------------------------------------------------------------------
// IX: how elements are addressed, long long indices or (unsigned) 32-bit byte
// offsets where all fit.
template <class S, class IX = long long> struct CTCtx {
    IX base;             // element offset of the lane's first column in cell 0
    IX ofp;              // offset to the fast-axis column above the lane's last column
    IX oom, oop;         // offsets to the other-axis rows below / above (mapped)
    bool active;         // lane stores its columns
    bool edge_lo, edge_hi;  // first / last row of the block
    bool fixy;           // halo lane at an outflow edge: its upper column is a copy of the lower
    int fused, fin;      // see ct_rounding
    S wfa, wfb;          // irregular mesh: widths of the lane's column and the one above (fast axis)
    S woa, wop, wom;     // widths of the lane's row and the rows above / below (other axis)
};

template <class V> struct CTRaw {
    V rc, mc, ro, mo, rm, mm;   // rho, m_d of the lane's columns in this, the next and the previous row
    typename VT<V>::S rf, mf;   // rho, m_d of the column above the lane's last column
    V bF, bO, bOm;              // fast-axis faces; other-axis faces of this and the previous row
    V bdo;                      // b_d of the output cell s-4
    V w;                        // width along d of cell s (irregular mesh)
};

template <class V> __device__ __forceinline__ void fixy_(V &a, bool f)
{
    if constexpr (VT<V>::W == 2) {
        if (f) a.v.y = a.v.x;
    }
}

// Load the raw inputs of cell s (any s up to four cells outside the box) and
// b_d of the cell s-4 that leaves when s enters (clamped to the box: before
// the segment's first output cell, and in the load behind its last step, it is
// not used).
template <class V, bool NU, class IX = long long, class AR>
__device__ __forceinline__ void ctload(const AR &A, const CTCtx<typename VT<V>::S, IX> &X,
                                       int s, CTRaw<V> &R)
{
    const int sm = wrap_cell(s, A.n, A.bc);
    const IX i = X.base + (IX)sm * ix_sd<IX>(A);
    if constexpr (NU) R.w = A.wd[sm];  // a ghost has the width of its image (reading C-23)
    R.rc = vget_at<V>(A.rho, i);
    R.mc = vget_at<V>(A.md, i);
    R.ro = vget_at<V>(A.rho, i + X.oop);
    R.mo = vget_at<V>(A.md, i + X.oop);
    R.rm = vget_at<V>(A.rho, i + X.oom);
    R.mm = vget_at<V>(A.md, i + X.oom);
    R.rf = __ldg(ix_at(A.rho, i + X.ofp));
    R.mf = __ldg(ix_at(A.md, i + X.ofp));
    R.bF = vget_at<V>(A.bf, i);
    R.bO = vget_at<V>(A.bo, i);
    R.bOm = vget_at<V>(A.bo, i + X.oom);
    if constexpr (VT<V>::W == 2) {
        if (X.fixy) {
            fixy_(R.rc, true); fixy_(R.mc, true); fixy_(R.ro, true); fixy_(R.mo, true);
            fixy_(R.rm, true); fixy_(R.mm, true); fixy_(R.bF, true); fixy_(R.bO, true); fixy_(R.bOm, true);
        }
    }
    R.bdo = vget_at<V>(A.bd, X.base + (IX)max(min(s - 4, A.n - 1), 0) * ix_sd<IX>(A));
}

// prefetch into L2 the fields of interior cell i; the neighbour rows by the
// warps at the edges of a block only, the others' are their siblings' own rows
#ifndef FISH_CT_PF_DIST
#define FISH_CT_PF_DIST 2   // against 1: 156 -> 148 us at 256^3, 2161 -> 2035 us at 640^3
#endif
template <class V, class IX = long long, class AR>
__device__ __forceinline__ void ctprefetch(const AR &A,
                                           const CTCtx<typename VT<V>::S, IX> &X, IX i)
{
    pf_l2(ix_at(A.rho, i));
    pf_l2(ix_at(A.md, i));
    if (X.edge_lo) {
        pf_l2(ix_at(A.rho, i + X.oom));
        pf_l2(ix_at(A.md, i + X.oom));
        pf_l2(ix_at(A.bo, i + X.oom));
    }
    if (X.edge_hi) {
        pf_l2(ix_at(A.rho, i + X.oop));
        pf_l2(ix_at(A.md, i + X.oop));
    }
    pf_l2(ix_at(A.bf, i));
    pf_l2(ix_at(A.bo, i));
    pf_l2(ix_at(A.bd, i));
}

// FP32 one-column CT (uniform mesh): the two face pencils above a column,
// along the fast and the other axis, have the same update; they advance
// together as one packed pencil (component x: fast axis, y: other axis),
// so one FP32x2 instruction serves both.
#ifndef FISH_CT_PACK
#define FISH_CT_PACK 1
#endif
template <class V, bool NU> constexpr bool ct_packs() { return FISH_CT_PACK && std::is_same<V, float>::value && !NU; }

template <class V> struct CTMarch {
    CFace<V> PF, PO, POm;   // fast-axis faces above, other-axis faces above / below
    CFace<P2> PFO;          // packed PF (x) and PO (y) of the FP32 one-column march
    CTRaw<V> R;             // raw inputs of the next cell
    CWid<V> cw;             // irregular mesh: widths along d of cells s-1 .. s-5
};

template <class V> __device__ __forceinline__ V shfl_up1(V a)
{
    if constexpr (VT<V>::W == 2) return {make_float2(__shfl_up_sync(0xffffffffu, a.v.x, 1),
                                                     __shfl_up_sync(0xffffffffu, a.v.y, 1))};
    else return __shfl_up_sync(0xffffffffu, a, 1);
}

// Where the one-column FP32 march rounds.  At a change of sign of an edge
// velocity one rounding picks another upwind cell, so the results stay those
// of earlier versions (of a run that is continued, of a study compared with
// one) only if every rounding does; these are where earlier kernels had them:
// - the sum of two velocities takes the neighbour's quotient m / rho as the
//   unrounded product of one multiply-add in the cells -1 .. fused - 1 and
//   `fin`, and rounded in the others (of a sweep of fewer than eight cells: in
//   all but cell -1), but in cell -4 the sum across the other-axis face takes
//   the cell's own quotient so;
// - the lower other-axis pencil takes its newest product unrounded in the
//   difference formed at cell `fin` (a cell no march reaches if there is none).
// The loop has a copy of its steps for the cells in the middle, where only the
// first holds: 137.3 -> 139.2 us at 256^3 and 1954 -> 1969 us at 640^3 against
// one form for all cells, 142.2 and 2008 us with the choice made in each step.
// A batch, whose short marches take both copies in most work items, makes the
// choice in each step: 808 us per double step of 12 boxes of 32 to 96 cells,
// 817 us with the copy, 799 us with one form.
__device__ __forceinline__ void ct_rounding(int n, int &fused, int &fin)
{
    fused = n >= 8 ? (n - 1) / 4 * 4 : 0;
    fin = n >= 8 && n % 4 == 0 ? n + 3 : n + 4;
}

// One cell s of the CT march (K = slot of cell s in the windows); the raw
// inputs of s are in M.R, the step loads those of s+1.  a: first output cell of
// the segment, so that cell s-4 is an output cell from s = a+4 on (the stages
// before work on windows that are still zero and their results are not used).
// MID: s is one of the cells 0 .. fused - 1 of ct_rounding.
template <class V, int LIM, bool FT1, bool NU, int K, bool MID, class IX = long long, class AR>
__device__ __forceinline__ void ctstep(const AR &A, const CTCtx<typename VT<V>::S, IX> &X,
                                       CTMarch<V> &M, int s, int a, V lamh, V lam, V lamf, V lamo, V dt)
{
    // widths of cells s .. s-5 for this step (the width of cell s arrived
    // with its raw inputs)
    if constexpr (NU) {
        M.cw.w5 = M.cw.w4;
        M.cw.w4 = M.cw.w3;
        M.cw.w3 = M.cw.w2;
        M.cw.w2 = M.cw.w1;
        M.cw.w1 = M.cw.w0;
        M.cw.w0 = M.R.w;
    }
    // consume the raw inputs of cell s
    constexpr bool PK = ct_packs<V, NU>();
    const V vc = vquot(M.R.mc, M.R.rc);
    V vop, vom, vfp, vtF, vtO, vtOm;
    if constexpr (PK) {
        // the sums of the velocities across the three faces (see ct_rounding)
        const float rf = srcp(M.R.rf), ro = srcp(M.R.ro), rm = srcp(M.R.rm);
        if (MID || (s >= -1 && s < X.fused) || s == X.fin) {
            vtF = fmaf(M.R.mf, rf, vc);
            vtO = fmaf(M.R.mo, ro, vc);
            vtOm = fmaf(M.R.mm, rm, vc);
        } else {
            vtF = vc + __fmul_rn(M.R.mf, rf);
            vtO = vc + __fmul_rn(M.R.mo, ro);
            vtOm = vc + __fmul_rn(M.R.mm, rm);
            if (s == -4) vtO = fmaf(M.R.mc, srcp(M.R.rc), __fmul_rn(M.R.mo, ro));
        }
    } else {
        vop = vquot(M.R.mo, M.R.ro);
        vom = vquot(M.R.mm, M.R.rm);
    }
    if constexpr (PK) {
    } else if constexpr (VT<V>::F64) vfp = vquot(M.R.mf, M.R.rf);
    else if constexpr (VT<V>::W == 2) vfp = vshift_hi(vc, __fdividef(M.R.mf, M.R.rf));
    else vfp = vdiv(V(M.R.mf), V(M.R.rf));
    const V bF = M.R.bF, bO = M.R.bO, bOm = M.R.bOm;
    const V bdo = M.R.bdo;
    // load cell s+1
    ctload<V, NU, IX>(A, X, s + 1, M.R);
    ctprefetch<V, IX>(A, X, X.base + (IX)max(min(s + 1 + FISH_CT_PF_DIST, A.n - 1), 0) * ix_sd<IX>(A));
    // twice the face velocities (see CT_SCALE; eq0361): the mean of the two
    // cells across the face, or on an irregular mesh their linear
    // interpolation to it (reading C-27)
    if constexpr (PK) {
    } else if constexpr (!NU) {
        vtF = vc + vfp;
        vtO = vc + vop;
        vtOm = vom + vc;
    } else if constexpr (VT<V>::F64) {
        vtF = 2.0 * ((X.wfb * vc + X.wfa * vfp) / (X.wfa + X.wfb));
        vtO = 2.0 * ((X.wop * vc + X.woa * vop) / (X.woa + X.wop));
        vtOm = 2.0 * ((X.woa * vom + X.wom * vc) / (X.wom + X.woa));
    } else {
        const V two = vb<V>(2.0f);
        vtF = two * vdiv(vfma(V(X.wfb), vc, V(X.wfa) * vfp), V(X.wfa + X.wfb));
        vtO = two * vdiv(vfma(V(X.wop), vc, V(X.woa) * vop), V(X.woa + X.wop));
        vtOm = two * vdiv(vfma(V(X.woa), vom, V(X.wom) * vc), V(X.wom + X.woa));
    }
    V nF, nO, dummy;
    // (FP64, bound by its pipe, skips the corrector until its fluxes are used)
    const bool live = s >= a + 3;
    if constexpr (PK) {
        P2 n2;
        cface<P2, LIM, K, true, false>(M.PFO, P2{make_float2(vtF, vtO)}, P2{make_float2(bF, bO)}, vb<P2>(lamh),
                                       vb<P2>(lam), n2, A.lim, live);
        nF = n2.v.x;
        nO = n2.v.y;
    } else {
        cface<V, LIM, K, true, NU>(M.PF, vtF, bF, lamh, lam, nF, A.lim, live, M.cw, dt);
        cface<V, LIM, K, true, NU>(M.PO, vtO, bO, lamh, lam, nO, A.lim, live, M.cw, dt);
    }
    cface<V, LIM, K, false, NU>(M.POm, vtOm, bOm, lamh, lam, dummy, A.lim, live, M.cw, dt, PK && !MID && s == X.fin);
    {
        constexpr int e = K & 1;
        // edge flux of the fast-axis face below: the upper pencil of the lane beneath
        V fup, fpo;
        if constexpr (PK) {
            fup = M.PFO.f[e].v.x;
            fpo = M.PFO.f[e].v.y;
        } else {
            fup = M.PF.f[e];
            fpo = M.PO.f[e];
        }
        const V sh = shfl_up1(fup);
        V fdn;
        if constexpr (VT<V>::W == 2) fdn = vshift_lo(sh.v.y, fup);
        else fdn = sh;
        if (X.active && s - 4 >= a) {
            const IX io = X.base + (IX)(s - 4) * ix_sd<IX>(A);
            vstore(ix_at(A.bfo, io), 0, nF);
            vstore(ix_at(A.boo, io), 0, nO);
            const V tF = fup - fdn, tO = fpo - M.POm.f[e];
            V r;
            if constexpr (VT<V>::F64) {
                if constexpr (FT1) r = bdo + lamf * tF + lamo * tO;
                else r = bdo + lamo * tO + lamf * tF;
            } else {
                r = vfma(lamo, tO, vfma(lamf, tF, bdo));
            }
            vstore(ix_at(A.bdo, io), 0, r);
        }
    }
}

#ifndef FISH_CT_MINB
#define FISH_CT_MINB 4
#endif

// B_d over all columns (eq0350 advection of the transverse components,
// eq0360 constraint update of b_d from the same edge fluxes).  Every lane of
// a warp takes the same steps (shuffles); lanes without columns of their
// own repeat a valid column and store nothing.
// The march of warp gw (31 W columns of one row) of the box described by A
// over the output cells a .. b-1.
// COPY: with a copy of the steps for the cells in the middle (see ct_rounding)
template <class V, int LIM, bool FT1, bool NU = false, class IX = long long, bool COPY = true, class AR>
__device__ __forceinline__ void ct_columns(const AR &A, long long gw, int lane, int a, int b,
                                           bool edge_lo, bool edge_hi)
{
    using S = typename VT<V>::S;
    constexpr int W = VT<V>::W;
    constexpr int SEGC = 31 * W;  // output columns per warp
    const int nseg = (A.nf + SEGC - 1) / SEGC;
    if (gw >= (long long)nseg * A.no) return;  // whole warps only
    const int seg = (int)(gw % nseg), ob = (int)(gw / nseg);
    int cl = seg * SEGC + (lane - 1) * W;       // first logical column of the lane
    CTCtx<S, IX> X;
    X.edge_lo = edge_lo;
    X.edge_hi = edge_hi || ob + 1 == A.no;
    X.active = lane >= 1 && cl < A.nf;
    if (lane >= 1 && cl >= A.nf) cl = A.nf - W;  // idle lane: repeat a valid column
    int cb;                                      // physical first column
    X.fixy = false;
    if (cl >= 0) {
        cb = cl;
    } else if (A.bc == BC_PERIODIC) {
        cb = cl + A.nf;
    } else {
        cb = 0;
        X.fixy = W == 2;
    }
    ct_rounding(A.n, X.fused, X.fin);
    const int cfp = gmap(cl + W, A.nf, A.bc);
    constexpr IX un = ix_unit<S, IX>();
    X.base = ((IX)A.off + (IX)cb + (IX)ob * (IX)A.so) * un;
    X.ofp = (IX)(cfp - cb) * un;
    X.oom = (IX)(gmap(ob - 1, A.no, A.bc) - ob) * (IX)A.so * un;
    X.oop = (IX)(gmap(ob + 1, A.no, A.bc) - ob) * (IX)A.so * un;
    const double dtd = *A.dt;
    const V dtv = vb<V>(S(dtd));
    constexpr double sc = CT_SCALE;
    const V lamh = vb<V>(S(sc * (dtd / (2.0 * A.h))));
    const V lam = vb<V>(S(sc * (dtd / A.h)));
    V lamf = vb<V>(S(sc * (dtd / A.hf)));
    V lamo = vb<V>(S(sc * (dtd / A.ho)));
    if constexpr (NU) {
        // irregular mesh: widths of the lane's column and its neighbours (a
        // halo or ghost column has the width of its image), and the
        // constraint factors of b_d over the cell's own transverse widths
        X.wfa = A.wf[cb];
        X.wfb = A.wf[cfp];
        X.woa = A.wo[ob];
        X.wop = A.wo[gmap(ob + 1, A.no, A.bc)];
        X.wom = A.wo[gmap(ob - 1, A.no, A.bc)];
        lamf = vb<V>(S(sc * (dtd / (double)X.wfa)));
        lamo = vb<V>(S(sc * (dtd / (double)X.woa)));
    }
    CTMarch<V> M;
    {
        CFace<V> z;
#pragma unroll
        for (int k = 0; k < 4; ++k) z.vt[k] = z.vh[k] = z.bf[k] = z.wp[k] = vb<V>(0.0f);
        z.w[0] = z.w[1] = z.f1[0] = z.f1[1] = z.f[0] = z.f[1] = z.dw[0] = z.dw[1] = vb<V>(0.0f);
        z.up = 0;
        M.PF = M.PO = M.POm = z;
        CFace<P2> z2;
#pragma unroll
        for (int k = 0; k < 4; ++k) z2.vt[k] = z2.vh[k] = z2.bf[k] = z2.wp[k] = vb<P2>(0.0f);
        z2.w[0] = z2.w[1] = z2.f1[0] = z2.f1[1] = z2.f[0] = z2.f[1] = vb<P2>(0.0f);
        M.PFO = z2;
    }
    M.cw.w0 = M.cw.w1 = M.cw.w2 = M.cw.w3 = M.cw.w4 = M.cw.w5 = vb<V>(1.0f);
    ctload<V, NU, IX>(A, X, a - 4, M.R);
    const int last = b + 3;
    // four steps; whether the last one was among them
    const auto four = [&](auto mid, int s) {
        constexpr bool MID = decltype(mid)::value;
        ctstep<V, LIM, FT1, NU, 0, MID, IX>(A, X, M, s, a, lamh, lam, lamf, lamo, dtv);
        if (s >= last) return true;
        ctstep<V, LIM, FT1, NU, 1, MID, IX>(A, X, M, s + 1, a, lamh, lam, lamf, lamo, dtv);
        if (s + 1 >= last) return true;
        ctstep<V, LIM, FT1, NU, 2, MID, IX>(A, X, M, s + 2, a, lamh, lam, lamf, lamo, dtv);
        if (s + 2 >= last) return true;
        ctstep<V, LIM, FT1, NU, 3, MID, IX>(A, X, M, s + 3, a, lamh, lam, lamf, lamo, dtv);
        return s + 3 >= last;
    };
#pragma unroll 1
    for (int s = a - 4;; s += 4) {
        if (!ct_packs<V, NU>() || (COPY && s >= 0 && s + 3 < X.fused)) {
            if (four(std::true_type{}, s)) break;
        } else {
            if (four(std::false_type{}, s)) break;
        }
    }
}

// The warps of a block take the same segment of ct_rows() consecutive
// rows of the other axis, so the neighbour-row loads of each warp (rho, m_d
// of rows o-1 and o+1, the other-axis face of row o-1) are mostly the
// own-row loads of its sibling warps, served from L1; FP64, bound by its pipe
// and not by loads, takes one warp per block.  Grid: (column segments x
// ceil(no / ct_rows())) x segments of `len` cells along the sweep.
template <class V> constexpr int ct_rows() { return VT<V>::F64 ? 1 : 8; }
// Blocks per SM the kernels are compiled for.
template <class V> constexpr int ct_resident() { return (VT<V>::F64 ? 8 : FISH_CT_MINB * 4) / ct_rows<V>(); }

template <class V, int LIM, bool FT1, bool NU = false, class IX = long long>
__global__ void __launch_bounds__(32 * ct_rows<V>(), ct_resident<V>())
    ct_col_kernel(const ColCTArgs<typename VT<V>::S> A, int len)
{
    constexpr int SEGC = 31 * VT<V>::W;
    const long long nseg = (A.nf + SEGC - 1) / SEGC;
    const long long seg = blockIdx.x % nseg, ob = (blockIdx.x / nseg) * ct_rows<V>() + (threadIdx.x >> 5);
    const int a = blockIdx.y * len;
    const int row = threadIdx.x >> 5;
    ct_columns<V, LIM, FT1, NU, IX>(A, ob * nseg + seg, threadIdx.x & 31, a, min(A.n, a + len), row == 0,
                                    row == ct_rows<V>() - 1);
}

// ---------------------------------------------------------------------------
// launchers (defined in fish_col_impl.cuh, instantiated per lane-vector type
// in their own translation units so they compile in parallel)
// ---------------------------------------------------------------------------
static inline int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        return 152;
    return sms;
}

// L_d with the lane-vector type V: hse selects the hydrostatic correction,
// ft1 says whether the fast axis is t1 (FP32 callers always order the frame
// so that it is).  Limiter from A.lim.
template <class V>
cudaError_t col_fluid(const ColFluidArgs<typename VT<V>::S> &A, bool hse, bool ft1, cudaStream_t s);
// B_d with the lane-vector type V.
template <class V> cudaError_t col_ct(const ColCTArgs<typename VT<V>::S> &A, bool ft1, cudaStream_t s);
// L_d fed by a shared-memory ring of bulk copies (fish_ring.cu): FP32 pairs,
// t1 fast, no potential, uniform mesh, Van Leer / minmod / hybrid limiter,
// nf % 4 == 0 and 16-byte aligned rows.  cudaErrorNotSupported where it
// does not apply (the caller then runs the column kernel).
cudaError_t ring_fluid(const ColFluidArgs<float> &A, cudaStream_t s);

}  // namespace fish
