"""The FP64 sweeps' quotient (fish_vec.cuh: reciprocal by one Newton step,
quotient corrected by its residual), Van Leer limiter and bitwise minmod
against CUDA's own division and the plain formulas, over the exponents the
sweeps meet."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "fish_vec.cuh"
using namespace fish;
__global__ void k(const double *a, const double *b, double *q, double *d, double *m, double *l, double *w,
                  int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    q[i] = quot64(a[i], b[i], rcp64(b[i]));
    d[i] = a[i] / b[i];
    m[i] = vminmod(a[i], b[i]);
    l[i] = 2.0 * vvanleer_half(a[i], b[i]);
    w[i] = a[i] * b[i] > 0.0 ? 2.0 * a[i] * b[i] / (a[i] + b[i]) : 0.0;
}
extern "C" int run(const double *a, const double *b, double *q, double *d, double *m, double *l, double *w, int n)
{
    k<<<(n + 255) / 256, 256>>>(a, b, q, d, m, l, w, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    from paper_0910_2854_gb300 import build
    d = tmp_path_factory.mktemp("quot")
    src, lib = d / "quot.cu", d / "libquot.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), "-shared", "-o", str(lib), str(src)] + build.ARCH + build.COMMON +
                   build.UNITS["fish_f64.cu"], check=True)
    f = ctypes.CDLL(str(lib)).run
    f.argtypes = [ctypes.c_void_p] * 7 + [ctypes.c_int]

    def call(a, b):
        """quot64, a / b, vminmod, the Van Leer limiter and its plain formula"""
        ta, tb = torch.as_tensor(a, device="cuda"), torch.as_tensor(b, device="cuda")
        out = [torch.empty_like(ta) for _ in range(5)]
        torch.cuda.synchronize()
        assert f(ta.data_ptr(), tb.data_ptr(), *[t.data_ptr() for t in out], a.size) == 0
        return [t.cpu().numpy() for t in out]
    return call


def test_quotient_and_minmod(run):
    rng = np.random.RandomState(5)
    n = 1 << 22
    a = rng.uniform(1, 2, n) * 2.0 ** rng.randint(-200, 200, n) * rng.choice([-1.0, 1.0], n)
    b = rng.uniform(1, 2, n) * 2.0 ** rng.randint(-200, 200, n) * rng.choice([-1.0, 1.0], n)
    a[:1000] = 0.0
    b[1000:2000] = 2.0 ** rng.randint(-100, 100, 1000)
    q, d, m, _, _ = run(a, b)
    # one rounding: never more than a unit in the last place off, and off at
    # all only where the quotient lies within 2^-30 ulp of a rounding boundary:
    # 0.004 of these pairs are expected to
    assert np.all(np.abs(q - d) <= np.spacing(np.abs(d)))
    assert np.count_nonzero(q != d) <= 1
    assert np.array_equal(m, 0.5 * (np.sign(a) + np.sign(b)) * np.minimum(np.abs(a), np.abs(b)))


def test_van_leer(run):
    """The limiter: pairs of like size, which share a slope, of any size, and
    what it has to return zero for (opposite signs, a sum of zero, zeros of
    either sign, a product that underflows)."""
    rng = np.random.RandomState(6)
    n = 1 << 21
    a = rng.uniform(1, 2, n) * 2.0 ** rng.randint(-100, 100, n) * rng.choice([-1.0, 1.0], n)
    b = a * rng.uniform(0.1, 10.0, n)
    b[: n // 4] = rng.uniform(1, 2, n // 4) * 2.0 ** rng.randint(-100, 100, n // 4) * np.sign(a[: n // 4])
    _, _, _, l, w = run(a, b)
    # the product is rounded alike (the factor 2 is exact) and so is the quotient, see above
    assert np.all(np.abs(l - w) <= np.spacing(np.abs(w)))
    assert np.count_nonzero(l != w) <= 1
    none = np.array([(1.5, -1.5), (1.5, -0.25), (-3.0, 2.0), (0.0, 1.0), (-0.0, 1.0), (1.0, -0.0), (0.0, 0.0),
                     (-0.0, -0.0), (0.0, -0.0), (1e-200, 1e-200), (-1e-250, -1e-100), (1e300, -1e300),
                     (5e-324, 5e-324), (-5e-324, 5e-324)])
    _, _, _, l, w = run(np.ascontiguousarray(none[:, 0]), np.ascontiguousarray(none[:, 1]))
    assert np.all(l == 0.0) and np.all(w == 0.0)
