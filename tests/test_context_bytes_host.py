"""lb_plan_memory on the CPU: populations with their padded rows, two parities of
shells, and what two sets of coefficients in the arithmetic type need beyond them."""
import ctypes

import pytest

Q = {"D2Q9": 9, "D3Q19": 19, "D3Q27": 27}
ES = {"f64": 8, "f32": 4, "f16s": 2, "bf16s": 2}


@pytest.fixture(scope="module")
def S():
    from paper_2304_06437_gb300 import build
    build.build()
    from paper_2304_06437_gb300 import solver
    return solver


@pytest.mark.parametrize("lat", list(Q))
@pytest.mark.parametrize("storage", list(ES))
def test_bytes_of_a_context(S, lat, storage):
    for side in ((1, 1, 1), (17, 5, 3), (33, 33, 33), (128, 128, 128), (300, 37, 12), (64, 8, 700)):
        dims = side[:2] + (1,) if lat == "D2Q9" else side
        b = S.context_bytes(lat, dims, storage)
        vol = -(-dims[0] // 32) * 32 * dims[1] * dims[2]
        pop = Q[lat] * vol * ES[storage]
        rs = 8 if storage == "f64" else 4
        shell = S.fused_plan(lat, dims, storage)["shell_elems_per_parity"]
        # allocations are laid out in pieces of 256 bytes
        assert 0 <= b["context_bytes"] - pop - 2 * shell * rs <= 256 + 2 * 32 * rs
        nc = 6 if lat == "D2Q9" else 10
        both = b["context_bytes"] + b["run_bytes"]
        if lat == "D2Q9":
            # set A behind the populations, set B in their place; no runs in 16 bits
            assert both == max(b["context_bytes"], pop + nc * vol * rs) if ES[storage] > 2 else b["run_bytes"] == 0
        else:
            assert both >= 2 * nc * vol * rs
        assert b["batch_bytes"] <= 4 * pop + (1 << 16)


def test_refusals(S):
    from paper_2304_06437_gb300 import _binding as B
    lib = B.load()
    out = B.lb_context_bytes_t()

    def call(lat, st, dims):
        return lib.lb_plan_memory(lat, st, (ctypes.c_int64 * 3)(*dims), ctypes.byref(out))
    assert call(7, B.LB_F32, (8, 8, 8)) == B.LB_E_INVAL
    assert call(B.LB_D3Q19, 9, (8, 8, 8)) == B.LB_E_INVAL
    assert call(B.LB_D3Q19, B.LB_F32, (0, 8, 8)) == B.LB_E_INVAL
    assert call(B.LB_D2Q9, B.LB_F32, (8, 8, 2)) == B.LB_E_INVAL
