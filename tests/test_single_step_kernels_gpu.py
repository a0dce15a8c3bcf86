"""Steps taken one per call go through the context's own brick kernel, whatever
runs of several steps do: every compiled 3D and 2D brick alternative (export warps
decoupled or inside the barrier, TMA stores, paired nodes, other ring depths)
gives the bits of the paper's two-pass schedule, on grids of many ragged bricks."""
import numpy as np
import pytest

from lbcase import faces_for, random_state

pytestmark = pytest.mark.gpu

# lattice, storage, brick (bx, by, bz), pipeline request, (slots, export warps, nodes per thread)
KERNELS = [
    ("D3Q19", "f32", (64, 8, 5), "2,0,-1,0,1", (2, 0, 1)),    # planes stored by TMA
    ("D3Q19", "f32", (64, 8, 5), "3,0,0,1,0", (3, 0, 1)),
    ("D3Q19", "f32", (64, 8, 5), "3,0,-1,2", (3, 0, 2)),      # two nodes a thread
    ("D3Q19", "f32", (32, 16, 5), "3,2,0", (3, 0, 1)),
    ("D3Q19", "f32", (64, 7, 5), "3,2,2", (3, 2, 1)),         # decoupled export warps
    ("D3Q19", "f32", (64, 6, 5), "3,2,4", (3, 4, 1)),
    ("D3Q19", "f32", (32, 14, 5), "3,2,-2", (3, -2, 1)),      # export warps in the barrier
    ("D3Q19", "f32", (32, 8, 5), "2,2,0,1,0,2", (2, 0, 1)),   # two CTAs an SM
    ("D3Q19", "f64", (32, 8, 5), "2,2,0", (2, 0, 1)),
    ("D3Q19", "f16s", (64, 8, 5), "4,2,0,1", (4, 0, 1)),
    ("D3Q19", "f16s", (64, 7, 5), "4,2,2", (4, 2, 1)),
    ("D3Q19", "f16s", (64, 7, 5), "4,2,-2", (4, -2, 1)),
    ("D3Q19", "bf16s", (64, 8, 5), "4,0,-1,2", (4, 0, 2)),
    ("D3Q27", "f32", (32, 14, 4), "2,2,-2", (2, -2, 1)),
    ("D3Q27", "f32", (32, 14, 4), "2,2,0", (2, 0, 1)),
    ("D3Q27", "f32", (32, 10, 4), "2,2,2", (2, 2, 1)),
    ("D3Q27", "f32", (64, 6, 4), "2,0,-1,2", (2, 0, 2)),
    ("D3Q27", "f64", (32, 4, 4), "2,2,0", (2, 0, 1)),
    ("D3Q27", "f16s", (32, 16, 4), "3,2,0", (3, 0, 1)),
    ("D3Q27", "f16s", (32, 10, 4), "3,2,2", (3, 2, 1)),
    ("D2Q9", "f32", (256, 1, 9), "4,0,-1,2", (4, 0, 2)),
    ("D2Q9", "f32", (64, 1, 9), "4,2,0,1", (4, 0, 1)),
    ("D2Q9", "f64", (256, 1, 9), "3,2,0,1", (3, 0, 1)),
]


@pytest.mark.parametrize("lat,storage,tile,pipeline,want", KERNELS)
@pytest.mark.parametrize("fname", ["lid", "periodic", "duct"])
def test_single_steps_equal_two_pass(lat, storage, tile, pipeline, want, fname, monkeypatch):
    from paper_2304_06437_gb300 import Solver, build, fused_plan
    build.build()
    dims = {"D3Q19": (150, 30, 23), "D3Q27": (70, 33, 13), "D2Q9": (300, 37, 1)}[lat]
    faces, wall_u = faces_for(lat, fname)
    force = (2e-5, 0, 1e-5) if fname == "duct" else (0, 0, 0)
    f0 = random_state(lat, dims, 77)
    outs = []
    for scheme, t in (("two_pass", None), ("fused", tile), ("fused", (tile[0], tile[1], 0))):
        if scheme == "fused":
            monkeypatch.setenv("LB_FUSED_PIPELINE", pipeline)
            p = fused_plan(lat, dims, storage, t)
            assert (p["tma_slots"], p["export_warps"], p["nodes_per_thread"]) == want
        with Solver(lat, dims, 0.58, faces=faces, wall_u=wall_u, storage=storage, scheme=scheme, force=force,
                    tile=t) as s:
            monkeypatch.delenv("LB_FUSED_PIPELINE", raising=False)
            if scheme == "fused":
                i = s.info()
                assert i["tile"][:2] == tile[:2] and (i["tma_slots"], i["nodes_per_thread"]) == (want[0], want[2])
            s.set_populations(np.ascontiguousarray(f0))
            for _ in range(9):
                s.step(1)
            outs.append(s.get_populations())
    assert np.array_equal(outs[0], outs[1])
    assert np.array_equal(outs[0], outs[2])


@pytest.mark.parametrize("lat", ["D3Q19", "D3Q27"])
def test_single_steps_at_any_sweep_length(lat):
    from paper_2304_06437_gb300 import Solver, build
    build.build()
    dims = (40, 19, 23)
    faces, wall_u = faces_for(lat, "lid_periodic_z")
    f0 = random_state(lat, dims, 17)
    outs = []
    for bz in (0, 3, 8, 11, 23):
        with Solver(lat, dims, 0.55, faces=faces, wall_u=wall_u, storage="f32", tile=(0, 0, bz)) as s:
            s.set_populations(np.ascontiguousarray(f0))
            for _ in range(9):
                s.step(1)
            outs.append(s.get_populations())
    for o in outs[1:]:
        assert np.array_equal(outs[0], o)
