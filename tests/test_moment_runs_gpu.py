"""Runs of several steps in moment form (lb_step(n), n >= 4): bit for bit the
populations of n single-step launches, at the edges of the compiled tiles
(partial tiles, one-plane and one-node domains, sweeps shorter than the load
ring), for every boundary kind, and with the state that a following single
step reads (the shell) in order."""
import numpy as np
import pytest

from lbcase import faces_for, random_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Solver():
    import torch
    assert torch.cuda.is_available()
    from paper_2304_06437_gb300 import build
    build.build()
    from paper_2304_06437_gb300 import Solver as S
    return S


def _run(Solver, lat, dims, faces, wall_u, storage, force, f0, calls):
    with Solver(lat, dims, 0.6, faces=faces, wall_u=wall_u, storage=storage, force=force) as s:
        s.set_populations(np.ascontiguousarray(f0))
        for n in calls:
            s.step(n)
        s.sync()
        f = s.get_populations()
        assert s.info()["steps_done"] == sum(calls)
        return f


@pytest.mark.parametrize("fname", ["periodic", "walls", "lid", "duct"])
@pytest.mark.parametrize("dims", [(37, 21, 13), (65, 17, 9), (64, 32, 5), (31, 49, 2), (1, 1, 1), (3, 20, 40)])
@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("lat", ["D3Q19", "D3Q27"])
def test_runs_equal_single_steps(Solver, lat, storage, dims, fname):
    faces, wall_u = faces_for(lat, fname)
    force = (2e-5, 0, 1e-5) if fname == "duct" else (0, 0, 0)
    f0 = random_state(lat, dims, 91)
    # even and odd run lengths, a recorded run, and single steps after each
    want = _run(Solver, lat, dims, faces, wall_u, storage, force, f0, [1] * 23)
    got = _run(Solver, lat, dims, faces, wall_u, storage, force, f0, [4, 1, 5, 1, 12])
    assert np.array_equal(got, want)
