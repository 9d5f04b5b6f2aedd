"""The FP64 sweeps' quotient (fish_vec.cuh: reciprocal by one Newton step,
quotient corrected by its residual) and bitwise minmod against CUDA's own
division and the plain formula, over the exponents the sweeps meet."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "fish_vec.cuh"
using namespace fish;
__global__ void k(const double *a, const double *b, double *q, double *d, double *m, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    q[i] = quot64(a[i], b[i], rcp64(b[i]));
    d[i] = a[i] / b[i];
    m[i] = vminmod(a[i], b[i]);
}
extern "C" int run(const double *a, const double *b, double *q, double *d, double *m, int n)
{
    k<<<(n + 255) / 256, 256>>>(a, b, q, d, m, n);
    return (int)cudaDeviceSynchronize();
}
"""


def test_quotient_and_minmod(tmp_path):
    import torch
    from paper_0910_2854_gb300 import build
    src, lib = tmp_path / "quot.cu", tmp_path / "libquot.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), "-shared", "-o", str(lib), str(src)] + build.ARCH + build.COMMON +
                   build.UNITS["fish_f64.cu"], check=True)
    rng = np.random.RandomState(5)
    n = 1 << 22
    a = rng.uniform(1, 2, n) * 2.0 ** rng.randint(-200, 200, n) * rng.choice([-1.0, 1.0], n)
    b = rng.uniform(1, 2, n) * 2.0 ** rng.randint(-200, 200, n) * rng.choice([-1.0, 1.0], n)
    a[:1000] = 0.0
    b[1000:2000] = 2.0 ** rng.randint(-100, 100, 1000)
    ta, tb = torch.as_tensor(a, device="cuda"), torch.as_tensor(b, device="cuda")
    q, d, m = (torch.empty_like(ta) for _ in range(3))
    torch.cuda.synchronize()
    f = ctypes.CDLL(str(lib)).run
    f.argtypes = [ctypes.c_void_p] * 5 + [ctypes.c_int]
    assert f(ta.data_ptr(), tb.data_ptr(), q.data_ptr(), d.data_ptr(), m.data_ptr(), n) == 0
    q, d, m = (t.cpu().numpy() for t in (q, d, m))
    # one rounding: never more than a unit in the last place off, and off at
    # all only where the quotient lies within 2^-30 ulp of a rounding boundary
    assert np.all(np.abs(q - d) <= np.spacing(np.abs(d)))
    assert np.mean(q != d) <= 1e-6
    assert np.array_equal(m, 0.5 * (np.sign(a) + np.sign(b)) * np.minimum(np.abs(a), np.abs(b)))
