"""lb_cg_step(n) keeps the two colours' populations out of memory between the
steps of one call: its result is bit for bit that of n calls of one step, at
box remainders and one-node extents, with and without near-contact forces."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lb():
    import torch
    assert torch.cuda.is_available()
    from paper_2304_06437_gb300 import build
    build.build()
    import paper_2304_06437_gb300 as P
    return P


CASES = [("D2Q9", (1, 9, 1)), ("D2Q9", (37, 1, 1)), ("D2Q9", (67, 41, 1)), ("D2Q9", (256, 8, 1)),
         ("D3Q19", (1, 1, 1)), ("D3Q19", (5, 33, 2)), ("D3Q19", (33, 17, 19))]


@pytest.mark.parametrize("lat,dims", CASES)
@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("nci", [False, True])
def test_runs_equal_single_steps(lb, lat, dims, storage, nci):
    d = 2 if lat == "D2Q9" else 3
    n = int(np.prod(dims))
    if nci and min(dims[:d]) < 4:
        pytest.skip("the near-contact distance does not fit this extent")
    rng = np.random.default_rng(7)
    # droplets of both signs a few nodes apart: thin films everywhere
    z, y, x = np.meshgrid(*(np.arange(m) for m in dims[::-1]), indexing="ij")
    wave = np.cos(2 * np.pi * x / 7) + np.cos(2 * np.pi * y / 9) + (np.cos(2 * np.pi * z / 8) if d == 3 else 0)
    phi = np.tanh(2 * wave.ravel() + 0.2 * rng.standard_normal(n))
    _, u, _ = synth.smooth_random_state(dims, d, seed=5, du=0.02)
    outs = []
    for calls in ([5, 4, 1], [1] * 10):
        with lb.CGSolver(lat, dims, 0.8, 0.02, 0.7, storage=storage) as s:
            if nci:
                s.set_nci(0.02, 0.1875, 2)
            s.init((1 + phi) / 2, (1 - phi) / 2, np.ascontiguousarray(u))
            for k in calls:
                s.step(k)
            outs.append(s.get_populations())
    for a, b in zip(*outs):
        assert np.isfinite(a).all() and np.array_equal(a, b)
