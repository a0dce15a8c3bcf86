"""The autotuner times single steps of every brick shape, however many steps it
is asked for and whatever lb_step() would do with that many: the context's own
shape is listed with the time of its single steps, not of a run (which takes a
fifth of it at this size)."""
import pytest

from lbcase import faces_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,storage,dims", [("D3Q19", "f32", (48, 40, 44)), ("D3Q27", "f32", (48, 40, 44)),
                                              ("D3Q19", "f64", (48, 40, 44)), ("D3Q27", "f16s", (48, 40, 44)),
                                              ("D2Q9", "f32", (304, 260, 1))])
def test_table_holds_single_steps(lat, storage, dims):
    import torch
    from paper_2304_06437_gb300 import Solver, build, fused_plan
    build.build()
    faces, wall_u = faces_for(lat, "lid")
    st = torch.cuda.Stream()
    with Solver(lat, dims, 0.6, faces=faces, wall_u=wall_u, storage=storage, stream=st) as s:
        best = 1e9
        for _ in range(5):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            with torch.cuda.stream(st):
                e[0].record()
                for _ in range(60):
                    s.step(1)
                e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]) * 1e6 / (60 * s.n))
        own = fused_plan(lat, dims, storage)
        table = s.autotune(steps=60)
    assert table and all(e["status"] == 0 for e in table)
    mine = [e["ns_per_update"] for e in table if (e["bx"], e["by"], e["bz"], e["slots"], e["nodes_per_thread"],
                                                  e["export_warps"]) == (own["bx"], own["by"], own["bz"],
                                                                         own["tma_slots"], own["nodes_per_thread"],
                                                                         own["export_warps"])]
    assert mine and min(mine) > 0.6 * best, (mine, best)
