"""Little free device memory: where the matrix product's operands do not fit, the recurrence kernels,
which need less, value the book as they do when asked for."""
import numpy as np
import pytest
import torch

import synth
from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu
F64, COMP, DEFL = rsv.RSV_FORM_F64, rsv.RSV_FORM_F32_COMP, rsv.RSV_FORM_F32_DEFLATED
OUT = rsv.RSV_OUT_V0 | rsv.RSV_OUT_SCEN_TOTAL
N, S = 60_000, 40   # digits of 1,200 steps: 0.6 (deflated) to 1.0 GB
LEFT = 256 << 20


@pytest.fixture
def ctx():
    h = rsv.rsv_create(0, torch.cuda.current_stream())
    rsv.rsv_load_decrements(h, 0, synth.gm_monthly_survival())
    rsv.rsv_load_scenarios(h, synth.vasicek_paths(S, 1200, seed=1))
    yield h
    rsv.rsv_destroy(h)


class Occupied:
    """All but LEFT bytes of the device's memory."""

    def __enter__(self):
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        self.block = torch.empty(free - LEFT, dtype=torch.uint8, device="cuda")

    def __exit__(self, *a):
        del self.block
        torch.cuda.empty_cache()


@pytest.mark.parametrize("form", [F64, COMP, DEFL])
def test_reserves(ctx, form):
    rsv.rsv_load_portfolio(ctx, synth.portfolio_mix(N, seed=2))
    V, tot = torch.zeros(N, S, device="cuda", dtype=torch.float64), torch.zeros(S, device="cuda", dtype=torch.float64)

    def call(variant):
        V.zero_(), tot.zero_()
        rsv.rsv_compute_reserves(ctx, form, OUT, on_device=True, variant=variant, V0d=V, scen_total=tot)
        rsv.rsv_synchronize(ctx)
        return V.cpu().numpy(), tot.cpu().numpy()

    want = call(0)
    with Occupied():
        for _ in range(2):
            got = call(-1)
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    got = call(-1)   # with room again
    assert np.allclose(got[0], want[0], rtol=2e-6, atol=1e-6) and not np.array_equal(got[0], want[0])


def test_lives(ctx):
    rng = np.random.default_rng(1)
    rec = np.zeros(N, rsv.MLIFE_DTYPE)
    rec["m"], rec["k"], rec["amount"] = 2, 1, 100.0
    rec["age_m"] = rng.integers(300, 600, (N, 4))
    V = torch.zeros(N, S, device="cuda", dtype=torch.float64)

    def call(h):
        V.zero_()
        rsv.rsv_compute_mlife(h, rec, COMP, rsv.RSV_OUT_V0, on_device=True, V0d=V)
        rsv.rsv_synchronize(h)
        return V.cpu().numpy()

    with Occupied():
        got = call(ctx)
    assert np.allclose(call(ctx), got, rtol=1e-6)
