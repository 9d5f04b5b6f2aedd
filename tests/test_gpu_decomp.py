"""GPU: the z-slab decomposition (``decomp.py``) driving the CUDA library.
One rank on a periodic box exchanges its ghost planes with itself through
fish_get_planes / fish_set_planes on device memory and must give the
single-box result: bitwise in FP64 (built without multiply-add contraction),
within 2e-6 of each field's largest magnitude in FP32, where a cell may sit
in the march prologue of one box and the steady loop of the other and the
compiler may contract the two instantiations differently.  Ranks on several GPUs are covered by the gloo tests on
CPU; on one GPU the multi-rank exchange is not run."""
import numpy as np
import pytest

from paper_0910_2854_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import torch
    assert torch.cuda.is_available()
    from paper_0910_2854_gb300 import build
    build.build()
    import paper_0910_2854_gb300 as mod
    mod.load()
    return mod


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_single_rank_slab_equals_single_box(F, precision):
    import torch
    from paper_0910_2854_gb300 import decomp
    w = W.random_smooth(24, 20, 18, seed=91, h=(0.04, 0.05, 0.055))
    nx, ny, nz = w.dims
    k0, nk, lo, hi = decomp.slab_extent(nz, 0, 1, True)
    assert (k0, nk, lo, hi) == (0, nz, decomp.HALO, decomp.HALO)
    st = np.zeros((8, lo + nk + hi, ny, nx))
    st[:, lo:lo + nk] = w.state
    box = F.Box(nx, ny, lo + nk + hi, w.gamma, precision=precision, h=w.h)
    box.set_state(st)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    run = decomp.SlabRun(box, nx, ny, nz, 0, 1, periodic=True, dist=None, device="cuda", dtype=dtype)
    ref = F.Box(*w.dims, w.gamma, precision=precision, h=w.h)
    ref.set_state(w.state)
    for _ in range(3):
        dt = run.step_cfl(0.5, 1)
        want = ref.cfl_dt(0.5)
        assert dt == want if precision == "fp64" else abs(dt - want) <= 1e-6 * want
        ref.step(dt)
    got, exp = box.get_state()[:, lo:lo + nk], ref.get_state()
    if precision == "fp64":
        assert np.array_equal(got, exp)
    else:
        scale = np.max(np.abs(exp), axis=(1, 2, 3), keepdims=True)
        assert float(np.max(np.abs(got - exp) / scale)) <= 2e-6
    box.close()
    ref.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_slab_beside_other_work_on_the_current_stream(F, precision):
    """The ghost exchange does not depend on when torch's current stream gets
    to it: a step queued behind other work there gives the same bits."""
    import torch
    from paper_0910_2854_gb300.decomp import SlabRun, slab_extent
    w = W.random_smooth(24, 20, 16, seed=15)
    nx, ny, nz = w.dims
    dt = torch.float32 if precision == "fp32" else torch.float64
    _, _, lo, hi = slab_extent(nz, 0, 1, True)
    st = torch.as_tensor(np.concatenate([w.state[:, nz - lo:], w.state, w.state[:, :hi]], axis=1), device="cuda").to(dt)
    out = []
    for busy in (False, True):
        box = F.Box(nx, ny, nz + lo + hi, w.gamma, bc=w.bc, precision=precision, h=w.h)
        run = SlabRun(box, nx, ny, nz, 0, 1, True, device="cuda", dtype=dt)
        box.set_state(st)
        for _ in range(2):
            if busy:
                torch.cuda._sleep(50_000_000)  # (clocks: some 25 ms)
            run.step_cfl(0.4, 1)
        torch.cuda.synchronize()
        out.append(box.get_state()[:, lo:lo + nz])
        box.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dims", [(5, 3, 7), (8, 4, 6), (33, 1, 9)])
def test_planes_to_device_host_and_unaligned_buffers(F, precision, dims):
    """Plane slabs through a device buffer (one kernel, 16-byte units or, from
    an odd offset or odd planes, words) and a host buffer (copies) are the
    state's planes, and write back to where they came from."""
    import torch
    w = W.random_smooth(*dims, seed=12)
    dt = torch.float32 if precision == "fp32" else torch.float64
    box = F.Box(*dims, w.gamma, bc=w.bc, precision=precision, h=w.h)
    box.set_state(w.state)
    ref = torch.as_tensor(box.get_state()).to(dt)
    nx, ny, nz = dims
    for k0, nk in ((0, 1), (1, 2), (nz - 1, 1), (0, nz), (2, 0)):
        n = 8 * nk * nx * ny
        for buf in (torch.zeros(n + 1, dtype=dt, device="cuda")[:n], torch.zeros(n + 1, dtype=dt, device="cuda")[1:],
                    torch.zeros(n, dtype=dt).pin_memory()):
            if n == 0 and buf.data_ptr() == 0:
                continue
            torch.cuda.synchronize()
            box.get_planes(k0, nk, buf)
            box.sync()
            assert torch.equal(buf.cpu().reshape(8, nk, ny, nx), ref[:, k0:k0 + nk])
            buf.mul_(2.0)
            torch.cuda.synchronize()
            box.set_planes(k0, nk, buf)
            box.sync()
            got = torch.as_tensor(box.get_state()).to(dt)
            assert torch.equal(got[:, k0:k0 + nk], 2.0 * ref[:, k0:k0 + nk])
            box.set_state(w.state)
    box.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_planes_are_x_fastest_after_set_and_get_state(F, precision):
    """The state is kept y fastest after fish_set_state_device and
    fish_get_state_device where the x sweeps come first; plane copies behind
    them still move x-fastest planes, operators and reads see the same state,
    whatever was needed first after the last upload."""
    import torch
    dims = (6, 10, 5)
    w = W.random_smooth(*dims, seed=13)
    dt = torch.float32 if precision == "fp32" else torch.float64
    dev = torch.as_tensor(w.state, device="cuda").to(dt)
    nx, ny, nz = dims
    box = F.Box(*dims, w.gamma, bc=w.bc, precision=precision, h=w.h)
    out, pl = torch.empty_like(dev), torch.empty(8 * 2 * nx * ny, dtype=dt, device="cuda")
    ref = None
    for first in ("planes", "x", "y", "planes", "get", "step", "y", "x", "planes"):
        box.set_state(dev)
        if first == "planes":
            box.get_planes(1, 2, pl)
            box.sync()
            assert torch.equal(pl.reshape(8, 2, ny, nx), dev[:, 1:3])
            box.set_planes(1, 2, pl)
        elif first == "get":
            assert torch.equal(box.get_state_device(out), dev)
        if first in ("x", "y"):
            box.fluid(0 if first == "x" else 1, 1e-3)
            box.set_state(dev)
        box.step(1e-3)
        got = box.get_state_device(out).clone()
        ref = got if ref is None else ref
        assert torch.equal(got, ref), first
        box.get_planes(1, 2, pl)
        box.sync()
        assert torch.equal(pl.reshape(8, 2, ny, nx), ref[:, 1:3]), first
        assert np.array_equal(box.get_state(), ref.double().cpu().numpy())
    box.close()


@pytest.mark.parametrize("dims,sweep", [((2, 4, 65535), 2), ((2, 4, 65536), 2), ((4200001, 2, 1), 1),
                                        ((2, 4200001, 1), 1), ((1, 4200001, 1), 1)])
def test_state_of_a_box_longer_than_a_launch_grid(F, dims, sweep):
    """A layout change takes a grid layer per z-plane (at most 65535) and a row
    of blocks per tile along x or y (as many); state uploads and downloads of
    longer boxes, and the sweeps along y and z, do without one."""
    import torch
    u = np.random.RandomState(3).random_sample((8, dims[2], dims[1], dims[0]))
    dev = torch.as_tensor(u, device="cuda").float().mul_(0.1)
    dev[0] += 1.0
    dev[4] += 1.0
    box = F.Box(*dims, 1.4, bc=W.BC_PERIODIC, precision="fp32", h=(0.1, 0.1, 0.1))
    box.set_state(dev)
    assert torch.equal(box.get_state_device(torch.empty_like(dev)), dev)
    box.fluid(sweep, 1e-3)
    box.ct(sweep, 1e-3)
    assert torch.isfinite(box.get_state_device(torch.empty_like(dev))).all()
    box.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_state_in_a_buffer_not_aligned_to_its_elements(F, precision):
    """Such a device buffer (a C caller's) is copied; only an aligned one is
    turned by a kernel."""
    import ctypes
    import torch
    dims = (6, 10, 5)
    w = W.random_smooth(*dims, seed=14)
    dt = torch.float32 if precision == "fp32" else torch.float64
    dev = torch.as_tensor(w.state, device="cuda").to(dt)
    raw = dev.reshape(-1).view(torch.uint8)
    code = F.FISH_F32 if precision == "fp32" else F.FISH_F64
    box, ref = (F.Box(*dims, w.gamma, bc=w.bc, precision=precision, h=w.h) for _ in range(2))
    ref.set_state(dev)
    ref.step(1e-3)
    want = ref.get_state_device(torch.empty_like(dev))
    for shift in (1, 2, dev.element_size() // 2 + 1):
        buf = torch.zeros(raw.numel() + 16, dtype=torch.uint8, device="cuda")
        buf[shift:shift + raw.numel()] = raw
        torch.cuda.synchronize()
        p = ctypes.c_void_p(buf.data_ptr() + shift)
        box._check(box._lib.fish_set_state_device(box.ctx, p, code), "set")
        box.step(1e-3)
        box._check(box._lib.fish_get_state_device(box.ctx, p, code), "get")
        box.sync()
        assert torch.equal(buf[shift:shift + raw.numel()].clone().view(dt).reshape(dev.shape), want)
    box.close()
    ref.close()
