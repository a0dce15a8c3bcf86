"""Runs of several steps in moment form with 16-bit storage: bit for bit the
populations of single-step launches, every value rounded to the storage at every
step, at the edges of tiles and of the sets' memory, for even and odd lengths."""
import numpy as np
import pytest

from lbcase import faces_for, random_state

pytestmark = pytest.mark.gpu


def _run(lat, dims, faces, wall_u, storage, force, f0, calls):
    from paper_2304_06437_gb300 import Solver
    with Solver(lat, dims, 0.6, faces=faces, wall_u=wall_u, storage=storage, force=force) as s:
        s.set_populations(np.ascontiguousarray(f0))
        for n in calls:
            s.step(n)
        s.sync()
        assert s.info()["steps_done"] == sum(calls)
        return s.get_populations()


@pytest.mark.parametrize("fname", ["periodic", "lid", "duct"])
@pytest.mark.parametrize("dims", [(37, 21, 13), (64, 16, 5), (31, 25, 2), (1, 1, 1), (3, 20, 40), (70, 30, 33)])
@pytest.mark.parametrize("storage", ["f16s", "bf16s"])
@pytest.mark.parametrize("lat", ["D3Q19", "D3Q27"])
def test_runs_equal_single_steps(lat, storage, dims, fname):
    from paper_2304_06437_gb300 import build
    build.build()
    faces, wall_u = faces_for(lat, fname)
    force = (2e-5, 0, 1e-5) if fname == "duct" else (0, 0, 0)
    f0 = random_state(lat, dims, 17)
    want = _run(lat, dims, faces, wall_u, storage, force, f0, [1] * 27)
    got = _run(lat, dims, faces, wall_u, storage, force, f0, [4, 1, 5, 1, 16])
    assert np.array_equal(got, want)
