"""Batch calls of four or more steps with no, some and all members running on
their own: every member's populations are bit for bit those of single steps, with
calls of one to three steps and steps of members alone in between."""
import numpy as np
import pytest

from lbcase import faces_for, random_state

pytestmark = pytest.mark.gpu

LARGE = [("D3Q19", (61, 56, 50), "f32", "lid"), ("D3Q19", (60, 57, 49), "f16s", "duct"),
         ("D3Q27", (56, 55, 54), "f32", "periodic"), ("D3Q27", (64, 52, 51), "bf16s", "lid"),
         ("D3Q19", (55, 56, 57), "f64", "walls"), ("D2Q9", (301, 257, 1), "f32", "lid"),
         ("D2Q9", (400, 180, 1), "f64", "lid")]
SMALL = [("D3Q19", (12, 9, 7), "f32", "lid"), ("D3Q19", (20, 14, 9), "f16s", "lid"), ("D2Q9", (60, 31, 1), "f32", "lid"),
         ("D2Q9", (77, 31, 1), "bf16s", "lid"), ("D3Q27", (9, 8, 7), "f64", "walls")]
# (members, the number of the first ones that run on their own)
SHARES = {"none": (SMALL, 0), "some": (LARGE + SMALL, len(LARGE)), "all": (LARGE, len(LARGE))}
CALLS = (9, 1, 4, 3, 13, 2, 16)  # the runs' lengths even and odd, the shells at either parity


@pytest.mark.parametrize("share", list(SHARES))
def test_members_equal_single_steps(share):
    import paper_2304_06437_gb300 as lb
    from paper_2304_06437_gb300 import build
    build.build()
    specs, n_alone = SHARES[share]

    def make(i):
        lat, dims, storage, fname = specs[i]
        faces, wall_u = faces_for(lat, fname)
        s = lb.Solver(lat, dims, 0.58 + 0.02 * i, faces=faces, wall_u=wall_u, storage=storage,
                      force=(2e-5, 1e-5, 0.0) if fname == "duct" else (0, 0, 0))
        s.set_populations(np.ascontiguousarray(random_state(lat, dims, 70 + i)))
        return s

    extra = [i % 2 for i in range(len(specs))]  # steps of its own between the batch's
    want = []
    for i in range(len(specs)):
        with make(i) as s:
            for _ in range(sum(CALLS) + extra[i]):
                s.step(1)
            want.append(s.get_populations())
    members = [make(i) for i in range(len(specs))]
    with lb.Batch(members) as b:
        assert sorted(b.alone()) == list(range(n_alone))
        for k, n in enumerate(CALLS):
            b.step(n)
            if k == 1:
                for s, e in zip(members, extra):
                    s.step(e)
        b.sync()
        assert b.info()["steps_done"] == sum(CALLS)
        for s, f, spec, e in zip(members, want, specs, extra):
            assert np.array_equal(s.get_populations(), f), spec
            assert s.info()["steps_done"] == sum(CALLS) + e
    for s in members:
        s.close()
