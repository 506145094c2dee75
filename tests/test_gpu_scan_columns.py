"""The time scan with its scenario columns in shared memory (up to 32 KB) and in global memory,
more chains than warps, and the totals' one and two levels, against the FP64 recurrence.
Tolerances: both are FP64 with a few thousand roundings a chain, all terms of one sign: 1e-12;
totals add n more roundings."""
import numpy as np
import pytest
import torch

from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    h = rsv.rsv_create(0, torch.cuda.current_stream())
    rsv.rsv_load_decrements(h, 0, np.append(np.linspace(0.99999, 0.97, 1430), 0.0))
    yield h
    rsv.rsv_destroy(h)


@pytest.mark.parametrize("n_scen", [1, 2, 3, 4, 33])   # 1,200 months: 28.1 KB at 3, 37.5 KB at 4
@pytest.mark.parametrize("n", [1, 256, 257, 1025, 4000])
def test_scan(ctx, n, n_scen):
    rng = np.random.default_rng(n)
    pol = np.zeros(n, rsv.POLICY_DTYPE)
    pol["product"] = rng.integers(0, 10, n)
    pol["age1_m"], pol["age2_m"] = rng.integers(300, 1000, n), rng.integers(300, 1000, n)
    pol["term_m"] = rng.integers(1, 400, n)
    pol["reversion"] = rng.uniform(0, 1, n)
    pol["amount"] = rng.uniform(1, 2, n)
    rsv.rsv_load_portfolio(ctx, pol)
    rsv.rsv_load_scenarios(ctx, 1.0 - rng.uniform(0.001, 0.006, (n_scen, 1200)))
    V, W, t = np.zeros((n, n_scen)), np.zeros((n, n_scen)), np.zeros(n_scen)
    rsv.rsv_compute_reserves(ctx, rsv.RSV_FORM_F64, rsv.RSV_OUT_V0 | rsv.RSV_OUT_SCEN_TOTAL,
                             variant=rsv.RSV_VARIANT_TIME_SCAN, V0d=V, scen_total=t)
    rsv.rsv_compute_reserves(ctx, rsv.RSV_FORM_F64, rsv.RSV_OUT_V0, variant=0, V0d=W)
    assert np.allclose(V, W, rtol=1e-12, atol=0.0)
    assert np.allclose(t, V.sum(0), rtol=1e-12 + n * 2.0 ** -53, atol=0.0)
