"""A call that runs out of device memory leaves the context usable: the next smaller one gives what
it gave before."""
import numpy as np
import pytest
import torch

import synth
from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu
LEFT = 300 << 20


@pytest.fixture
def ctx():
    h = rsv.rsv_create(0, torch.cuda.current_stream())
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


def test_scenarios_too_large_for_their_planes(ctx):
    """Staged (192 MB) but not kept in three formats."""
    rsv.rsv_load_decrements(ctx, 0, synth.gm_monthly_survival())
    rsv.rsv_load_portfolio(ctx, synth.portfolio_mix(50, seed=1))
    v = synth.vasicek_paths(33, 1200, seed=1)
    rsv.rsv_load_scenarios(ctx, v)
    V, W = np.zeros((50, 33)), np.zeros((50, 33))
    rsv.rsv_compute_reserves(ctx, V0d=V)
    with Occupied():
        with pytest.raises(rsv.RsvError, match="RSV_E_NOMEM"):
            rsv.rsv_load_scenarios(ctx, np.full((20_000, 1200), 0.997))
        with pytest.raises(rsv.RsvError, match="RSV_E_STATE"):
            rsv.rsv_compute_reserves(ctx, V0d=W)
    rsv.rsv_load_scenarios(ctx, v)
    rsv.rsv_compute_reserves(ctx, V0d=W)
    assert np.array_equal(V, W)


def test_gradient_of_too_many_rows(ctx):
    rng = np.random.default_rng(1)
    rsv.rsv_mlp_set_params(ctx, rng.normal(0, 0.05, rsv.rsv_mlp_param_count()).astype(np.float32))
    X, t = rng.normal(0, 0.5, (1 << 18, 32)).astype(np.float32), rng.normal(0, 1, 1 << 18).astype(np.float32)
    g, loss = rsv.rsv_mlp_gradient(ctx, X[:64], t[:64])
    with Occupied():
        with pytest.raises(rsv.RsvError, match="RSV_E_NOMEM"):
            rsv.rsv_mlp_gradient(ctx, X, t)
        for _ in range(2):
            h, other = rsv.rsv_mlp_gradient(ctx, X[:64], t[:64])
            assert np.array_equal(g, h) and loss == other
