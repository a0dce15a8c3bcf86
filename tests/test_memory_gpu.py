"""What lb_info reports is what a context takes of the device: its populations,
its shells and the memory of its runs of several steps, before and after a batch
has re-planned it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20
SLACK = 6 * MB  # allocation granules, and what the driver keeps for launches


@pytest.fixture(scope="module")
def lb():
    import torch
    assert torch.cuda.is_available()
    from paper_2304_06437_gb300 import build
    build.build()
    import paper_2304_06437_gb300 as P
    return P


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _held(s):
    i = s.info()
    return i["population_bytes"] + i["aux_bytes"]


FORMS = [("D3Q19", "f16s", (128, 128, 128)), ("D3Q27", "bf16s", (128, 128, 96)), ("D3Q19", "f32", (160, 128, 128)),
         ("D3Q27", "f32", (128, 128, 96)), ("D3Q19", "f64", (128, 128, 96)), ("D2Q9", "f32", (2048, 1024, 1)),
         ("D2Q9", "f16s", (4096, 1024, 1)), ("D3Q19", "two_pass", (128, 128, 96))]


@pytest.mark.parametrize("lat,storage,dims", FORMS)
def test_info_reports_what_is_allocated(lb, lat, storage, dims):
    kw = dict(storage="f32", scheme="two_pass") if storage == "two_pass" else dict(storage=storage)

    def use(s):
        s.step(9)
        s.step(1)
        s.sync()

    with lb.Solver(lat, dims, 0.7, **kw) as s:  # modules and streams come with first use
        use(s)
    before = _free()
    with lb.Solver(lat, dims, 0.7, **kw) as s:
        use(s)
        assert abs(before - _free() - _held(s)) <= SLACK
    assert abs(before - _free()) <= SLACK


@pytest.mark.parametrize("lat,storage,dims", [f for f in FORMS if f[1] != "two_pass"])
def test_info_after_a_batch(lb, lat, storage, dims):
    def use(s):
        with lb.Batch([s]) as b:
            b.step(6)
            b.step(1)
            b.sync()
        s.step(5)
        s.sync()

    with lb.Solver(lat, dims, 0.7, storage=storage) as s:
        use(s)
    before = _free()
    with lb.Solver(lat, dims, 0.7, storage=storage) as s:
        first = _held(s)
        use(s)
        assert abs(before - _free() - _held(s)) <= SLACK
        assert _held(s) >= first
    assert abs(before - _free()) <= SLACK


@pytest.mark.parametrize("lat,storage,dims", [("D3Q19", "f16s", (128, 128, 128)), ("D3Q27", "bf16s", (128, 128, 96)),
                                              ("D3Q19", "bf16s", (96, 128, 112))])
def test_shells_of_a_batch_take_the_room_there_is(lb, lat, storage, dims):
    """The runs' memory lies idle where shells are read: a re-plan allocates
    nothing beside it."""
    with lb.Solver(lat, dims, 0.7, storage=storage) as s:
        first, tile = _held(s), s.info()["tile"]
        with lb.Batch([s]) as b:
            b.step(1)
            b.sync()
            assert s.info()["tile"] != tile
            assert _held(s) == first


@pytest.mark.parametrize("lat,storage,dims", [f for f in FORMS if f[1] != "two_pass"] +
                         [("D3Q19", "f32", (66, 130, 192)), ("D3Q27", "f16s", (100, 100, 100))])
def test_a_served_request_holds_no_more_than_its_footprint(lb, lat, storage, dims):
    from paper_2304_06437_gb300 import serve
    from paper_2304_06437_gb300.solver import context_bytes

    def use(s):
        with lb.Batch([s]) as b:
            b.step(6)
            b.step(1)
            b.sync()
        return _free()

    with lb.Solver(lat, dims, 0.7, storage=storage) as s:
        use(s)
    before = _free()
    # but the snapshot of u, which comes from a pool that contexts share
    foot = serve.footprint_bytes(serve.Request(0, 0.0, lat, dims, 0.7, [0] * 6, storage=storage)) - 12 * np.prod(dims)
    with lb.Solver(lat, dims, 0.7, storage=storage) as s:
        plan = context_bytes(lat, dims, storage)
        assert _held(s) == plan["context_bytes"] + plan["run_bytes"]
        held = before - use(s)
        assert _held(s) <= sum(plan.values()) <= foot
    assert held <= foot + SLACK
    assert foot <= 1.5 * held + SLACK
