"""FP32 results stay, bit for bit, those of the column marches before they were
cut into segments: at a change of sign of an edge velocity one rounding picks
another upwind cell of the field, so that two versions that round differently
part by far more than round-off within a few steps.

The digests are of states those kernels gave on a GB300 (FP32 quotients and
square roots are the hardware's approximations), from inputs that need no
library function."""
import hashlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BATCH = ((8, 2, 33), (66, 4, 7), (34, 32, 36), (4, 6, 3), (10, 12, 8))
# extents along the sweeps: fewer than eight cells, multiples of four and none
BOXES = ((8, 6, 16), (33, 21, 9), (4, 5, 7))
LIMITERS = {"vanleer": 0, "minmod": 1, "none": 2, "hybrid": 3}


def state(dims, seed):
    """Random values with a positive pressure, to FP32 exactly."""
    nx, ny, nz = dims
    u = np.random.RandomState(seed).random_sample((8, nz, ny, nx))
    q = np.empty_like(u)
    q[0] = 1.0 + 0.25 * u[0]
    q[1:4] = 0.5 * (u[1:4] - 0.5)
    q[4] = 2.0 + 0.25 * u[4]
    q[5:] = 0.25 * (u[5:] - 0.5)
    return q.astype(np.float32).astype(np.float64)


def digest(states):
    h = hashlib.sha256()
    for s in states:
        h.update((np.asarray(s).astype(np.float32) + np.float32(0.0)).astype("<f4").tobytes())  # (-0 is 0)
    return h.hexdigest()[:16]


def batch_states(F, bc, limiter):
    b = F.Batch(BATCH, [5.0 / 3.0] * len(BATCH), [bc] * len(BATCH), limiter=LIMITERS[limiter])
    for k, d in enumerate(BATCH):
        b.set_state(k, state(d, 300 + k))
    b.step(0.4, 3)
    out = [b.get_state(k) for k in range(len(BATCH))]
    b.close()
    return out


def box_states(F, bc, limiter, split):
    out = []
    for k, d in enumerate(BOXES):
        box = F.Box(*d, 5.0 / 3.0, bc=bc, precision="fp32", limiter=LIMITERS[limiter],
                    gravity="split" if split else "unsplit")
        q = state(d, 400 + k)
        box.set_state(q)
        if split:
            box.set_potential(0.25 * q[0])
        box.step_cfl(0.4, 3)
        out.append(box.get_state())
        box.close()
    return out


BATCH_DIGESTS = {
    (0, "vanleer"): "e0f09076048a518a",
    (0, "minmod"): "0a46fe6928da4cf2",
    (1, "vanleer"): "d07252c7b1777fcd",
    (1, "minmod"): "bc61826c96861f8f",
}
BOX_DIGESTS = {
    (0, "vanleer", False): "70ec0b5a8b837ab4",
    (0, "vanleer", True): "dc5e3b1cbff1bd80",
    (0, "minmod", False): "cc1fd4b01dfe6717",
    (0, "minmod", True): "dff98d4ed0825b79",
    (0, "none", False): "11b4b7a57532351b",
    (0, "none", True): "8f7c1a149a9bac83",
    (0, "hybrid", False): "70ec0b5a8b837ab4",
    (0, "hybrid", True): "dc5e3b1cbff1bd80",
    (1, "vanleer", False): "d28e7a3d6ec3a6a1",
    (1, "vanleer", True): "e6eb61ac5464a89f",
    (1, "minmod", False): "8f144a8088f714e5",
    (1, "minmod", True): "af0ea4b10be9df28",
    (1, "none", False): "28ef4cae04cc3e10",
    (1, "none", True): "49716440b9cd8afa",
    (1, "hybrid", False): "d28e7a3d6ec3a6a1",
    (1, "hybrid", True): "e6eb61ac5464a89f",
}


@pytest.fixture(scope="module")
def F():
    from paper_0910_2854_gb300 import build
    build.build()
    import paper_0910_2854_gb300 as F
    return F


@pytest.mark.parametrize("bc,limiter", sorted(BATCH_DIGESTS))
def test_batch(F, bc, limiter):
    assert digest(batch_states(F, bc, limiter)) == BATCH_DIGESTS[bc, limiter]


@pytest.mark.parametrize("bc,limiter,split", sorted(BOX_DIGESTS))
def test_box(F, bc, limiter, split):
    assert digest(box_states(F, bc, limiter, split)) == BOX_DIGESTS[bc, limiter, split]
