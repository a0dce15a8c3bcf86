"""How runs of 2D domains are divided into launches (lb_plan_flat), on the CPU:
the last launch writes the populations and set A of the coefficients lies behind
them, so a run needs an even number of launches, every one of them with at least
one step, and a tile with its ring has to fit shared memory."""
import ctypes

import pytest

MAX_STEPS = 8  # steps of one launch
SIZES = [(n, n) for n in (1, 5, 31, 64, 128, 257, 500, 700, 1024, 2048, 4096, 16384)] + [
    (1, 16384), (16384, 1), (62, 1000000), (1000000, 3), (301, 257), (700, 256), (6000, 5000)]


@pytest.fixture(scope="module")
def plan():
    from paper_2304_06437_gb300 import _binding as B
    from paper_2304_06437_gb300 import build
    build.build()
    lib = B.load()

    def call(storage, dims, n, sms=152):
        p = B.lb_flat_plan_t()
        rc = lib.lb_plan_flat(B.STORAGES[storage], (ctypes.c_int64 * 3)(*dims, 1), n, sms, ctypes.byref(p))
        return rc, p
    return call


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("sms", [152, 148, 1])
def test_every_launch_has_a_step(plan, storage, sms):
    for dims in SIZES:
        for n in list(range(2, 401)) + [999, 1000, 1001, 100001, 2 ** 40 + 1]:
            rc, p = plan(storage, dims, n, sms)
            at = (storage, dims, n, sms, p.launches, p.steps_first, p.steps_last)
            assert rc == 0 and 2 <= p.launches <= n and p.launches % 2 == 0, at
            # the steps are dealt out evenly: the first launch has the most, the last the fewest
            assert 1 <= p.steps_last <= p.steps_first <= min(p.steps_last + 1, MAX_STEPS), at
            assert p.launches * p.steps_last <= n <= p.launches * p.steps_first, at
            assert p.tile_rows >= 1 and p.tile_rows + 2 * p.steps_first <= p.max_rows, at


def test_refusals(plan):
    assert plan("f16s", (64, 64), 8)[0] == -6
    assert plan("f32", (0, 64), 8)[0] == -1
    assert plan("f32", (64, 64), 1)[0] == -1
