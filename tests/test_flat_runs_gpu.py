"""lb_step(n) of a 2D domain takes several steps per launch on tiles with a
ring: its populations are bit for bit those of n calls of one step, at the
edges of tiles and rings, for walls and periodic sides on either axis."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

P, W, M = 0, 1, 2  # periodic, wall, moving wall


@pytest.fixture(scope="module")
def lb():
    import torch
    assert torch.cuda.is_available()
    from paper_2304_06437_gb300 import build
    build.build()
    import paper_2304_06437_gb300 as pkg
    return pkg


@pytest.mark.parametrize("dims", [(1, 1), (1, 21), (5, 3), (48, 8), (50, 9), (63, 40), (65, 41), (113, 57), (300, 17)])
@pytest.mark.parametrize("faces", [[P] * 6, [W, W, W, M, P, P], [P, P, M, W, P, P], [W, M, P, P, P, P]])
@pytest.mark.parametrize("storage,forced", [("f32", False), ("f32", True), ("f64", True)])
def test_runs_equal_single_steps(lb, dims, faces, storage, forced):
    full = (dims[0], dims[1], 1)
    rho, u, pi = synth.smooth_random_state(full, 2, seed=11, du=0.03)
    wall_u = [[0.0, 0.03, 0.0], [0.0, 0.02, 0.0], [0.04, 0.0, 0.0], [0.05, 0.0, 0.0], [0.0] * 3, [0.0] * 3]
    force = (1e-4, -2e-4, 0.0) if forced else (0.0, 0.0, 0.0)
    outs = []
    # whole runs of few and many launches against single steps
    for calls in ([4, 17, 7, 32], [1] * 60):
        with lb.Solver("D2Q9", full, 0.57, faces=faces, wall_u=wall_u, storage=storage, force=force) as s:
            s.init_moments(rho, np.ascontiguousarray(u), pi)
            for k in calls:
                s.step(k)
            s.step(1)  # the shell is rebuilt
            outs.append(s.get_populations())
    assert np.isfinite(outs[0]).all()
    assert np.array_equal(outs[0], outs[1])
