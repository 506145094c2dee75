"""Scenarios of more steps than one launch of the matrix valuation's scenario kernels covers
(64 x 65,535): valued, like shorter ones, by the kernels that take them."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", [rsv.RSV_FORM_F64, rsv.RSV_FORM_F32_COMP])
def test_more_steps_than_a_grid(form):
    n_steps = 64 * 65535 + 1
    pol = synth.portfolio_mix(20, seed=1)
    v = np.ones((1, n_steps))
    v[:, :1200] = synth.vasicek_paths(1, 1200, seed=1)
    ctx = rsv.rsv_create(0, torch.cuda.current_stream())
    try:
        rsv.rsv_load_decrements(ctx, 0, synth.gm_monthly_survival())
        rsv.rsv_load_portfolio(ctx, pol)
        rsv.rsv_load_scenarios(ctx, v)
        V = np.zeros((20, 1))
        rsv.rsv_compute_reserves(ctx, form, V0d=V)
    finally:
        rsv.rsv_destroy(ctx)
    ref, _ = oracle.reserves_batch(pol, synth.gm_monthly_survival(), v[:, :1200])
    assert np.all(np.abs(V - ref) <= (1e-12 if form == rsv.RSV_FORM_F64 else 1e-6) * ref)
