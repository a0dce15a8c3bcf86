"""Batch calls of several steps run the larger members on streams of the batch
and the others in classes: every member as if stepped alone one step at a time,
with calls of one step and members stepped on their own in between."""
import numpy as np
import pytest

from lbcase import faces_for, random_state

pytestmark = pytest.mark.gpu

SPECS = [  # either side of the sizes from which members run on their own
    ("D3Q19", (49, 41, 37), "f32", "lid"), ("D3Q19", (41, 40, 39), "f32", "duct"), ("D3Q19", (12, 9, 7), "f32", "lid"),
    ("D3Q19", (50, 44, 31), "f16s", "periodic"), ("D3Q19", (20, 14, 9), "f16s", "lid"),
    ("D3Q27", (45, 40, 38), "f32", "walls"), ("D3Q19", (42, 40, 40), "f64", "periodic"),
    ("D2Q9", (150, 133, 1), "f32", "lid"), ("D2Q9", (60, 31, 1), "f32", "periodic"), ("D2Q9", (260, 70, 1), "f64", "lid"),
]


@pytest.mark.parametrize("small_only,large_only", [(False, False), (True, False), (False, True)])
def test_members_as_if_alone(small_only, large_only):
    import paper_2304_06437_gb300 as lb
    from paper_2304_06437_gb300 import build
    build.build()
    large = [int(np.prod(d)) >= (16384 if lat == "D2Q9" else 65536) for lat, d, _, _ in SPECS]
    specs = [s for s, big in zip(SPECS, large) if not (small_only and big) and not (large_only and not big)]

    def make(i):
        lat, dims, storage, fname = specs[i]
        faces, wall_u = faces_for(lat, fname)
        s = lb.Solver(lat, dims, 0.6 + 0.03 * i, faces=faces, wall_u=wall_u, storage=storage,
                      force=(2e-5, 1e-5, 0.0) if fname == "duct" else (0, 0, 0))
        s.set_populations(np.ascontiguousarray(random_state(lat, dims, 70 + i)))
        return s

    want = []
    for i in range(len(specs)):
        with make(i) as s:
            for _ in range(28 + (i % 2)):
                s.step(1)
            want.append(s.get_populations())
    members = [make(i) for i in range(len(specs))]
    with lb.Batch(members) as b:
        b.step(5)
        b.step(1)
        for i, s in enumerate(members):
            if i % 2:
                s.step(1)
        b.step(4)
        b.step(2)
        b.step(16)
        b.sync()
        for i, (s, f) in enumerate(zip(members, want)):
            assert np.array_equal(s.get_populations(), f), specs[i]
            assert s.info()["steps_done"] == 28 + (i % 2)
    for s in members:
        s.close()


def test_small_members_beside_a_large_one_as_if_alone():
    """One large member keeps the mean size up: 2D, 16-bit and one-column members
    of every storage run on their own too; forms without a run stay in classes."""
    import paper_2304_06437_gb300 as lb
    from paper_2304_06437_gb300 import build
    build.build()
    specs = SPECS + [("D3Q19", (110, 101, 97), "f32", "lid"), ("D2Q9", (31, 1, 1), "f32", "periodic"),
                     ("D2Q9", (77, 31, 1), "bf16s", "lid"), ("D3Q27", (9, 8, 7), "bf16s", "walls")]

    def make(i):
        lat, dims, storage, fname = specs[i]
        faces, wall_u = faces_for(lat, fname)
        s = lb.Solver(lat, dims, 0.58 + 0.02 * i, faces=faces, wall_u=wall_u, storage=storage,
                      force=(2e-5, 1e-5, 0.0) if fname == "duct" else (0, 0, 0))
        s.set_populations(np.ascontiguousarray(random_state(lat, dims, 40 + i)))
        return s

    want = []
    for i in range(len(specs)):
        with make(i) as s:
            for _ in range(17):
                s.step(1)
            want.append(s.get_populations())
    members = [make(i) for i in range(len(specs))]
    with lb.Batch(members) as b:
        for n in (6, 1, 10):
            b.step(n)
        b.sync()
        for s, f, spec in zip(members, want, specs):
            assert np.array_equal(s.get_populations(), f), spec
    for s in members:
        s.close()
