"""Population readout of FP32 data adds t_a rho0 in FP64: every bit of the sum,
for zeros, subnormals, values below the sum's last place, ties, values that
leave the binade of t_a rho0, and common magnitudes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,weights", [("D2Q9", [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4),
                                         ("D3Q19", [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)])
@pytest.mark.parametrize("rho0", [1.0, 2.25, 3e-21])
@pytest.mark.parametrize("storage", ["f32", "f16s", "f64"])
def test_population_readout_is_the_fp64_sum(lat, weights, rho0, storage):
    from paper_2304_06437_gb300 import Solver, build
    build.build()
    q = len(weights)
    dims = (67, 5, 1) if lat == "D2Q9" else (67, 5, 3)
    n = int(np.prod(dims))
    rng = np.random.default_rng(3)
    v = np.ldexp(1 + rng.integers(0, 8, (q, n)) / 8, rng.integers(-130, 3, (q, n))) * rng.choice([-1.0, 1.0], (q, n))
    v[:, ::7] = 0
    v[:, 1::7] = rng.standard_normal((q, n))[:, 1::7] * 1e-3
    c = (np.array(weights) * rho0)[:, None]
    # half and three halves of the last place of t_a rho0, and what ends its binade
    ulp = np.spacing(c)
    v[:, 2::14], v[:, 3::14], v[:, 4::14] = ulp / 2, -1.5 * ulp, -c / 2
    stored = (c + v) - c  # what FP64 input can say of the shifted value
    st = {"f32": np.float32, "f16s": np.float16, "f64": np.float64}[storage]
    with np.errstate(over="ignore"):
        want = stored.astype(np.float32).astype(st) if storage == "f16s" else stored.astype(st)
    with Solver(lat, dims, 0.8, storage=storage, rho0=rho0) as s:
        s.set_populations(np.ascontiguousarray(c + v))
        got = s.get_populations()
    assert np.array_equal(got, want.astype(np.float64) + c)
