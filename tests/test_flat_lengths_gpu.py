"""lb_step(n) of 2D domains for every short length and for odd lengths on
domains large enough that single steps are the cheapest launches: the
populations are bit for bit those of n calls of one step, alone and in a batch."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

FACES = [1, 1, 1, 2, 0, 0]
WALL_U = [[0.0] * 3] * 3 + [[0.05, 0.0, 0.0]] + [[0.0] * 3] * 2


@pytest.fixture(scope="module")
def lb():
    import torch
    assert torch.cuda.is_available()
    from paper_2304_06437_gb300 import build
    build.build()
    import paper_2304_06437_gb300 as pkg
    return pkg


def _solver(lb, dims, storage, state):
    s = lb.Solver("D2Q9", dims, 0.57, faces=FACES, wall_u=WALL_U, storage=storage, force=(1e-5, 0.0, 0.0))
    s.init_moments(*state)
    return s


def _state(dims):
    rho, u, pi = synth.smooth_random_state(dims, 2, seed=23, du=0.03)
    return rho, np.ascontiguousarray(u), np.ascontiguousarray(pi)


def _singles(lb, dims, storage, state, lengths):
    """Populations after each of the lengths, one step per call."""
    want = {}
    with _solver(lb, dims, storage, state) as s:
        for k in range(1, max(lengths) + 1):
            s.step(1)
            if k in lengths:
                want[k] = s.get_populations()
    return want


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("dims,lengths", [((64, 64, 1), range(4, 41)), ((256, 256, 1), (5, 9, 13, 17, 21, 25)),
                                          ((700, 256, 1), (5, 9, 13, 17, 21, 25)),
                                          ((1024, 1024, 1), (5, 9, 13, 17, 21, 25))])
def test_runs_of_every_length(lb, dims, lengths, storage):
    state = _state(dims)
    want = _singles(lb, dims, storage, state, set(lengths))
    for n in lengths:
        with _solver(lb, dims, storage, state) as s:
            s.step(n)
            assert np.array_equal(s.get_populations(), want[n]), n


def test_members_of_a_batch(lb):
    """A member large enough to run on its own, FP64, for lengths that single
    steps would serve best."""
    dims = (700, 256, 1)
    state = _state(dims)
    want = _singles(lb, dims, "f64", state, {9, 22})
    with _solver(lb, dims, "f64", state) as s, lb.Batch([s]) as b:
        b.step(9)
        b.sync()
        assert np.array_equal(s.get_populations(), want[9])
        b.step(13)
        b.sync()
        assert np.array_equal(s.get_populations(), want[22])
