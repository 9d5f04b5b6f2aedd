"""The FP32 sweeps address by 32-bit byte offsets up to 2^30 cells, beyond them
by 64-bit indices, or in a batch by 32-bit ones.  No test has boxes that large:
here the kernels of all three forms run on one small box and give the same
bits."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "fish_col_impl.cuh"
using namespace fish;

template <class IX> static cudaError_t sweep(int which, float **f, const float *phi, const double *dt, int nf, int no,
                                             int n, int bc, unsigned *flags)
{
    if (which < 3) {
        ColFluidArgs<float> A;
        for (int k = 0; k < 5; ++k) {
            A.u[k] = f[k];
            A.uo[k] = f[8 + k];
        }
        A.bd = f[5];
        A.bt1 = f[6];
        A.bt2 = f[7];
        A.phi = which ? phi : nullptr;
        A.sg = which == 2;
        A.dt = dt;
        A.off = 0;
        A.sd = (long long)nf * no;
        A.so = nf;
        A.n = n;
        A.nf = nf;
        A.no = no;
        A.bc = bc;
        A.lim = LIM_VANLEER;
        A.gamma = 1.5f;
        A.gm1 = 0.5f;
        A.alpha = 1.0f;
        A.h = 0.125;
        A.flags = flags;
        A.cfl_min = nullptr;
        A.rh[0] = A.rh[1] = A.rh[2] = 8.0f;
        if (which == 0) return fluid_run<P2, false, 0, LIM_VANLEER, true, false, false, IX>(A, 0);
        if (which == 1) return fluid_run<P2, true, 1, LIM_VANLEER, true, false, false, IX>(A, 0);
        return fluid_run<float, false, 2, -1, true, false, false, IX>(A, 0);
    }
    ColCTArgs<float> A;
    A.rho = f[0];
    A.md = f[1];
    A.bd = f[5];
    A.bf = f[6];
    A.bo = f[7];
    A.bdo = f[8];
    A.bfo = f[9];
    A.boo = f[10];
    A.dt = dt;
    A.off = 0;
    A.sd = (long long)nf * no;
    A.so = nf;
    A.n = n;
    A.nf = nf;
    A.no = no;
    A.bc = bc;
    A.lim = LIM_VANLEER;
    A.h = A.hf = A.ho = 0.125;
    const int R = ct_rows<float>(), len = 7;
    const dim3 grid((nf + 30) / 31 * ((no + R - 1) / R), (n + len - 1) / len);
    ct_col_kernel<float, LIM_VANLEER, true, false, IX><<<grid, 32 * R>>>(A, len);
    return cudaGetLastError();
}
extern "C" int run(int form, int which, float **f, const float *phi, const double *dt, int nf, int no, int n, int bc,
                   unsigned *flags)
{
    cudaError_t e = form == 0   ? sweep<unsigned>(which, f, phi, dt, nf, no, n, bc, flags)
                    : form == 1 ? sweep<int>(which, f, phi, dt, nf, no, n, bc, flags)
                                : sweep<long long>(which, f, phi, dt, nf, no, n, bc, flags);
    return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_0910_2854_gb300 import build
    d = tmp_path_factory.mktemp("index")
    src, lib = d / "index.cu", d / "libindex.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), "-shared", "-o", str(lib), str(src)] + build.ARCH + build.COMMON +
                   build.UNITS["fish_p2.cu"], check=True)
    f = ctypes.CDLL(str(lib)).run
    f.argtypes = [ctypes.c_int] * 2 + [ctypes.c_void_p] * 3 + [ctypes.c_int] * 4 + [ctypes.c_void_p]
    return f


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("nf,no,n", [(2, 1, 1), (34, 5, 9), (70, 33, 21), (128, 40, 64)])
def test_index_forms_agree(run, nf, no, n, bc):
    import torch
    rng = np.random.RandomState(31)
    u = rng.random_sample((9, n, no, nf)).astype(np.float32)
    u[0] = 1.0 + 0.25 * u[0]
    u[1:4] = 0.5 * (u[1:4] - 0.5)
    u[4] = 2.0 + 0.25 * u[4]
    u[5:8] = 0.25 * (u[5:8] - 0.5)
    u[8] = 0.01 * (u[8] - 0.5)
    src = torch.as_tensor(u, device="cuda")
    dt = torch.full((1,), 0.01, dtype=torch.float64, device="cuda")
    flags = torch.zeros(1, dtype=torch.int32, device="cuda")
    for which, outs in ((0, 5), (1, 5), (2, 5), (3, 3)):
        got = []
        for form in range(3):
            out = torch.full((8, n, no, nf), float("nan"), device="cuda")
            ptrs = (ctypes.c_void_p * 16)(*([src[k].data_ptr() for k in range(8)] +
                                            [out[k].data_ptr() for k in range(8)]))
            torch.cuda.synchronize()
            assert run(form, which, ptrs, src[8].data_ptr(), dt.data_ptr(), nf, no, n, bc, flags.data_ptr()) == 0
            got.append(out[:outs].cpu().numpy())
            assert np.isfinite(got[-1]).all(), (which, form)
        assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2]), which
    assert flags.item() == 0
