// fish_tile.cuh -- FP64 L_d and B_d of small boxes: a thread per cell.
//
// The column marches (fish_column.cuh) want segments of a dozen cells or more
// to keep the steps that fill their windows cheap, and a box of a few thousand
// columns has too few of those to occupy the FP64 pipes of the GPU: at 32^3 the
// best cut, segments of two cells, computes most things three times.  Here a
// block takes 32 columns (a warp's lanes) and a segment [a, b) of the sweep,
// one warp per cell of the segment and of its ghosts; the warps form the same
// quantities as a march step does, all cells at once, and pass them to their
// neighbours through shared memory in four rounds.  The arithmetic is the
// marches' own (ceval, cflux1, cflux2, the kicks, cface's formulas), so results
// are bitwise theirs.  Bound by the FP64 pipe: a tile of eight cells does 1.4
// times the operations of eight cells.  The times of both stand beside the rule
// that chooses (tile_cells in fish_launch.cuh); FP32 gains nothing (10.3 us
// either way at 32^3, most of it launches).
#pragma once

#include "fish_column.cuh"

namespace fish {

constexpr int TILE_MAX = 8;  // output cells of a tile: at most 16 warps with the ghosts

// values of a cell its neighbours read: u, F and the speeds a variant needs
template <bool HSE, bool HYB> constexpr int tile_vals() { return HSE ? 15 : (HYB ? 13 : 11); }

template <bool HSE, bool HYB>
__device__ __forceinline__ void tile_put(double *sm, int slot, int rows, int lane, const CCell<double> &c)
{
    // [value][slot][lane]
    double *p = sm + slot * 32 + lane;
    const int st = rows * 32;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        p[k * st] = c.u[k];
        p[(5 + k) * st] = c.F[k];
    }
    p[10 * st] = c.d;
    if constexpr (HSE || HYB) {
        p[11 * st] = c.vn;
        p[12 * st] = c.cs;
    }
    if constexpr (HSE) {
        p[13 * st] = c.cf;
        p[14 * st] = c.p;
    }
}
template <bool HSE, bool HYB>
__device__ __forceinline__ void tile_get(const double *sm, int slot, int rows, int lane, CCell<double> &c)
{
    const double *p = sm + slot * 32 + lane;
    const int st = rows * 32;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        c.u[k] = p[k * st];
        c.F[k] = p[(5 + k) * st];
    }
    c.d = p[10 * st];
    c.vn = c.cs = c.cf = c.p = 0.0;
    if constexpr (HSE || HYB) {
        c.vn = p[11 * st];
        c.cs = p[12 * st];
    }
    if constexpr (HSE) {
        c.cf = p[13 * st];
        c.p = p[14 * st];
    }
}

// L_d.  Grid: ceil(nf no / 32) x segments of `len` cells, 32 (len + 6) threads;
// dynamic shared memory of tile_fluid_smem.  GM as in the march.
template <bool HSE, int GM, int LIM, bool FT1, bool NU>
__global__ void __launch_bounds__(32 * (TILE_MAX + 6)) fluid_tile_kernel(const ColFluidArgs<double> A, int len)
{
    constexpr bool GRAV = GM == 1, SG = GM == 2, PHI = GM != 0, HYB = LIM < 0 && !HSE;
    constexpr int NV = tile_vals<HSE, HYB>();
    extern __shared__ __align__(16) unsigned char tile_smem[];
    double *cells = reinterpret_cast<double *>(tile_smem);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, rows = len + 6;
    double *flux = cells + NV * rows * 32, *pots = flux + 5 * rows * 32;
    const int a = blockIdx.y * len, b = min(A.n, a + len), r = a - 3 + w;
    const long long cols = (long long)A.nf * A.no, cid = (long long)blockIdx.x * 32 + lane;
    const bool col = cid < cols, cell = col && r <= b + 2;
    const long long cc = col ? cid : cols - 1;
    const int f0 = (int)(cc % A.nf), ob = (int)(cc / A.nf);
    FCtx<double> X;
    X.base = A.off + f0 + ob * A.so;
    X.ofm = (long long)(gmap(f0 - 1, A.nf, A.bc) - f0);
    X.oom = (long long)(gmap(ob - 1, A.no, A.bc) - ob) * A.so;
    const double dtd = *A.dt;
    const double dt = dtd, hdt = 0.5 * dtd, rtwoh = 1.0 / (2.0 * A.h), half = 0.5;
    double lam = FLUX_SCALE * (dtd / A.h), lamh = FLUX_SCALE * (dtd / (2.0 * A.h));
    Checks<double> chk;
    checks_init(chk);
    // round 1: the raw cells
    double u[5], bb[3], pot = 0.0, dk = 0.0;
    CCell<double> C, P;
    double wm = 1.0, w0 = 1.0, wp = 1.0, wq = 1.0;  // widths of cells r-1, r, r+1, r+2
    if (cell) {
        FRaw<double> R;
        fload_mapped<double, PHI, FT1>(A, X, r, R);
#pragma unroll
        for (int k = 0; k < 5; ++k) u[k] = R.u[k];
        bb[0] = half * (R.bdm + R.bd);
        bb[FT1 ? 1 : 2] = half * (R.bfm + R.bf);
        bb[FT1 ? 2 : 1] = half * (R.bom + R.bo);
        if constexpr (PHI) pot = R.phi;
        if constexpr (SG) {
            dk = sg_image_dk<double>(A, X, r, rtwoh);
            sg_kick<double>(u, dk, hdt);
        }
        if constexpr (NU) {
            wm = A.wd[gmap(r - 1, A.n, A.bc)];
            w0 = A.wd[gmap(r, A.n, A.bc)];
            wp = A.wd[gmap(r + 1, A.n, A.bc)];
            wq = A.wd[gmap(r + 2, A.n, A.bc)];
            lamh = FLUX_SCALE * (dt / (2.0 * w0));
            lam = FLUX_SCALE * (dt / w0);
        }
        ceval<double>(u, bb, A.gamma, A.gm1, C, chk);
        tile_put<HSE, HYB>(cells, w, rows, lane, C);
        if constexpr (GRAV || HSE) pots[w * 32 + lane] = pot;
    }
    __syncthreads();
    // round 2: predicted cells r = a-2 .. b+1
    const bool pred = cell && w >= 1 && r <= b + 1;
    double dphi = 0.0, potm = 0.0, potp = 0.0;
    if (pred) {
        CCell<double> Cm, Cp;
        tile_get<HSE, HYB>(cells, w - 1, rows, lane, Cm);
        tile_get<HSE, HYB>(cells, w + 1, rows, lane, Cp);
        if constexpr (GRAV || HSE) {
            potm = pots[(w - 1) * 32 + lane];
            potp = pots[(w + 1) * 32 + lane];
        }
        double Fm[5], Fp[5], up[5];
        cflux1<double, HSE>(Cm, C, potm, pot, A.alpha, Fm);
        cflux1<double, HSE>(C, Cp, pot, potp, A.alpha, Fp);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            up[k] = C.u[k] - lamh * (Fp[k] - Fm[k]);
        }
        if constexpr (GRAV) {
            // centred difference (eq02513; NU: over the centre span, reading C-26)
            if constexpr (NU) dphi = (potp - potm) / (0.5 * wm + w0 + 0.5 * wp);
            else dphi = (potp - potm) / (2.0 * A.h);
            up[1] = up[1] - hdt * C.u[0] * dphi;
            up[4] = up[4] - hdt * C.u[1] * dphi;
        }
        ceval<double>(up, bb, A.gamma, A.gm1, P, chk);
    }
    __syncthreads();
    if (pred) tile_put<HSE, HYB>(cells, w, rows, lane, P);
    __syncthreads();
    // round 3: corrector fluxes at (r, r+1), r = a-1 .. b-1
    double F2[5];
    if (cell && w >= 2 && r <= b - 1) {
        CCell<double> Pm, Pp, Pq;
        tile_get<HSE, HYB>(cells, w - 1, rows, lane, Pm);
        tile_get<HSE, HYB>(cells, w + 1, rows, lane, Pp);
        tile_get<HSE, HYB>(cells, w + 2, rows, lane, Pq);
        double du0[5], dd0[5], du1[5], dd1[5], du2[5], dd2[5];
        if constexpr (HSE) {
            chse(Pm, P, potm, pot, du0, dd0);
            chse(P, Pp, pot, potp, du1, dd1);
            chse(Pp, Pq, potp, pots[(w + 2) * 32 + lane], du2, dd2);
        }
        cflux2<double, HSE, LIM, NU>(Pm, P, Pp, Pq, du0, dd0, du1, dd1, du2, dd2, F2, A.lim, wm, w0, wp, wq);
#pragma unroll
        for (int k = 0; k < 5; ++k) flux[(k * rows + w) * 32 + lane] = F2[k];
    }
    __syncthreads();
    // round 4: the update of cells a .. b-1
    if (cell && w >= 3 && r < b) {
        double un[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            un[k] = u[k] - lam * (F2[k] - flux[(k * rows + w - 1) * 32 + lane]);
        }
        if constexpr (GRAV) {
            un[1] = un[1] - dt * P.u[0] * dphi;
            un[4] = un[4] - dt * P.u[1] * dphi;
        }
        if constexpr (SG) sg_kick<double>(un, dk, hdt);
        const long long io = X.base + r * A.sd;
#pragma unroll
        for (int k = 0; k < 5; ++k) A.uo[k][io] = un[k];
    }
    const unsigned fl = checks_flags(chk);
    if (fl) atomicOr(A.flags, fl);
}

template <bool HSE, bool HYB> constexpr size_t tile_fluid_smem(int len)
{
    return sizeof(double) * 32 * (size_t)(len + 6) * (tile_vals<HSE, HYB>() + 6);
}

// B_d.  A warp's lanes are a halo column and 31 columns of one row, as in the
// march; grid: (column segments x rows) x segments of `len` cells, 32 (len + 8)
// threads.  Pencils 0: fast-axis faces above the lane's column, 1: other-axis
// faces above it, 2: other-axis faces below it.
template <int LIM, bool FT1, bool NU>
__global__ void __launch_bounds__(32 * (TILE_MAX + 8)) ct_tile_kernel(const ColCTArgs<double> A, int len)
{
    extern __shared__ __align__(16) unsigned char tile_smem[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, rows = len + 8, st = rows * 32;
    double *X0 = reinterpret_cast<double *>(tile_smem) + w * 32 + lane;  // face velocities, then predicted products
    double *X1 = X0 + 3 * st;                                       // smoothed velocities
    double *X2 = X1 + 3 * st;                                       // products, then corrector fluxes
    const int a = blockIdx.y * len, b = min(A.n, a + len), s = a - 4 + w;
    const int nseg = (A.nf + 30) / 31, seg = (int)(blockIdx.x % nseg), ob = (int)(blockIdx.x / nseg);
    int cl = seg * 31 + lane - 1;
    const bool active = lane >= 1 && cl < A.nf;
    if (cl >= A.nf) cl = A.nf - 1;  // idle lane: repeat a valid column
    const int cb = cl >= 0 ? cl : (A.bc == BC_PERIODIC ? cl + A.nf : 0);
    const int cfp = gmap(cl + 1, A.nf, A.bc), obm = gmap(ob - 1, A.no, A.bc), obp = gmap(ob + 1, A.no, A.bc);
    const long long base = A.off + cb + ob * A.so, ofp = cfp - cb;
    const long long oom = (obm - ob) * A.so, oop = (obp - ob) * A.so;
    const double dtd = *A.dt;
    const double dt = dtd;
    double lamh = (CT_SCALE * (dtd / (2.0 * A.h))), lam = (CT_SCALE * (dtd / A.h));
    double lamf = (CT_SCALE * (dtd / A.hf)), lamo = (CT_SCALE * (dtd / A.ho));
    // widths along d of cells s-1 .. s+2
    double wm = 1.0, w0 = 1.0, wp = 1.0, wq = 1.0;
    if constexpr (NU) {
        lamf = (CT_SCALE * (dtd / (double)A.wf[cb]));
        lamo = (CT_SCALE * (dtd / (double)A.wo[ob]));
        wm = A.wd[gmap(s - 1, A.n, A.bc)];
        w0 = A.wd[gmap(s, A.n, A.bc)];
        wp = A.wd[gmap(s + 1, A.n, A.bc)];
        wq = A.wd[gmap(s + 2, A.n, A.bc)];
        lamh = CT_SCALE * (dt / (2.0 * w0));
        lam = CT_SCALE * (dt / w0);
    }
    const bool in = s <= b + 3;
    double vt[3], bf[3], vh[3], ww[3], f[3];
    if (in) {
        // face velocities (eq0361), FP64 doubled (see cface)
        const long long i = base + (long long)wrap_cell(s, A.n, A.bc) * A.sd;
        const double vc = vquot(__ldg(A.md + i), __ldg(A.rho + i));
        const double vfp = vquot(__ldg(A.md + i + ofp), __ldg(A.rho + i + ofp));
        const double vop = vquot(__ldg(A.md + i + oop), __ldg(A.rho + i + oop));
        const double vom = vquot(__ldg(A.md + i + oom), __ldg(A.rho + i + oom));
        bf[0] = __ldg(A.bf + i);
        bf[1] = __ldg(A.bo + i);
        bf[2] = __ldg(A.bo + i + oom);
        if constexpr (!NU) {
            vt[0] = vc + vfp;
            vt[1] = vc + vop;
            vt[2] = vom + vc;
        } else {
            const double wfa = A.wf[cb], wfb = A.wf[cfp], woa = A.wo[ob], wop = A.wo[obp], wom = A.wo[obm];
            vt[0] = 2.0 * ((wfb * vc + wfa * vfp) / (wfa + wfb));
            vt[1] = 2.0 * ((wop * vc + woa * vop) / (woa + wop));
            vt[2] = 2.0 * ((woa * vom + wom * vc) / (wom + woa));
        }
#pragma unroll
        for (int p = 0; p < 3; ++p) X0[p * st] = vt[p];
    }
    __syncthreads();
    // smoothed velocities (eq0362) and cell products, s = a-3 .. b+2
    const bool sm = in && w >= 1 && s <= b + 2;
    if (sm) {
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            // (eight times the velocity, see cface)
            vh[p] = __fma_rn(2.0, vt[p], X0[p * st + 32]) + X0[p * st - 32];
            ww[p] = vh[p] * bf[p];
            X1[p * st] = vh[p];
            X2[p * st] = ww[p];
        }
    }
    __syncthreads();
    // first-order upwind fluxes on both sides (eq0363, eq0364) and the
    // predicted products, s = a-2 .. b+1
    const bool pr = in && w >= 2 && s <= b + 1;
    double vhp[3];
    bool pos[3] = {false, false, false};
    if (pr) {
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            const double vhm = X1[p * st - 32], wwm = X2[p * st - 32], wwp = X2[p * st + 32];
            vhp[p] = X1[p * st + 32];
            double em, ep;
            if constexpr (NU) {
                em = w0 * vhm + wm * vh[p];
                ep = wp * vh[p] + w0 * vhp[p];
            } else {
                em = vhm + vh[p];
                ep = vh[p] + vhp[p];
            }
            pos[p] = pos64(ep);
            const double fm = pos64(em) ? wwm : ww[p], fp = pos[p] ? ww[p] : wwp;
            X0[p * st] = vh[p] * (bf[p] - lamh * (fp - fm));
        }
    }
    __syncthreads();
    // corrector fluxes at s' (reading C-10), s = a-1 .. b-1
    const bool co = in && w >= 3 && s <= b - 1;
    if (co) {
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            const double q0 = X0[p * st], qm = X0[p * st - 32], q1 = X0[p * st + 32], q2 = X0[p * st + 64];
            const double d0 = q0 - qm, d1 = q1 - q0, d2 = q2 - q1;
            const bool u = pos[p];
            double la = u ? d0 : d1, lb = u ? d1 : d2;
            if constexpr (NU) {
                la = la / (0.5 * (u ? wm + w0 : w0 + wp));
                lb = lb / (0.5 * (u ? w0 + wp : wp + wq));
            }
            double sl = vlimit_half<LIM>(la, lb, A.lim);
            const double q = u ? q0 : q1;
            if constexpr (NU) sl = (u ? w0 : wp) * sl;
            f[p] = q + (u ? sl : -sl);
            X2[p * st] = f[p];
        }
    }
    __syncthreads();
    if (in && w >= 4 && s < b) {
        const double fdn = __shfl_up_sync(0xffffffffu, f[0], 1);
        if (active) {
            const long long io = base + s * A.sd;
            double nb[2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                nb[p] = bf[p] - lam * (f[p] - X2[p * st - 32]);
            }
            A.bfo[io] = nb[0];
            A.boo[io] = nb[1];
            const double tF = f[0] - fdn, tO = f[1] - f[2], bd = __ldg(A.bd + io);
            A.bdo[io] = FT1 ? bd + lamf * tF + lamo * tO : bd + lamo * tO + lamf * tF;
        }
    }
}

constexpr size_t tile_ct_smem(int len) { return sizeof(double) * 32 * (size_t)(len + 8) * 9; }

// launchers (fish_tile.cu): `len` output cells per tile, at most TILE_MAX
cudaError_t tile_fluid(const ColFluidArgs<double> &A, bool hse, bool ft1, int len, cudaStream_t s);
cudaError_t tile_ct(const ColCTArgs<double> &A, bool ft1, int len, cudaStream_t s);

}  // namespace fish
