"""Runs of several steps of 3D domains with walls, still and moving, on every
choice of axes: bit for bit single steps, at partial tiles and one-node extents."""
import numpy as np
import pytest

from lbcase import random_state

pytestmark = pytest.mark.gpu

P, W, M = 0, 1, 2
FACES = [(W, W, P, P, P, P), (P, P, M, W, P, P), (P, P, P, P, W, M), (M, W, W, M, P, P), (W, M, P, P, M, W),
         (P, P, M, M, M, M), (M, M, M, M, M, M)]
# tangential velocities, another on each face
WALL_U = [[0, 0.03, 0.01], [0, -0.02, 0.02], [0.04, 0, 0.01], [0.02, 0, -0.03], [0.03, 0.02, 0], [-0.02, 0.01, 0]]


@pytest.mark.parametrize("faces", FACES)
@pytest.mark.parametrize("dims", [(37, 21, 13), (66, 33, 5), (1, 20, 9), (33, 1, 7)])
@pytest.mark.parametrize("lat,storage", [("D3Q19", "f32"), ("D3Q19", "f16s"), ("D3Q27", "f32"), ("D3Q27", "f64"),
                                         ("D3Q27", "bf16s")])
def test_runs_equal_single_steps(lat, storage, dims, faces):
    from paper_2304_06437_gb300 import Solver, build
    build.build()
    f0 = random_state(lat, dims, 19)
    outs = []
    for calls in ([5, 1, 10], [1] * 16):
        with Solver(lat, dims, 0.6, faces=list(faces), wall_u=WALL_U, storage=storage) as s:
            s.set_populations(np.ascontiguousarray(f0))
            for n in calls:
                s.step(n)
            outs.append(s.get_populations())
    assert np.isfinite(outs[0]).all()
    assert np.array_equal(outs[0], outs[1])
