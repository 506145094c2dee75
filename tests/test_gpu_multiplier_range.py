"""Cash-flow multipliers of every size that is accepted, against the recurrence kernels
(variant 0) and, in FP64, the oracle.

Tolerances, relative to each reserve.  FP64: the form's 1e-12.  Compensated: the recurrence reads the
multipliers rounded to FP32, so 2^-24 and its own 1e-8; 1e-6 covers both."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu
COMP, F64 = rsv.RSV_FORM_F32_COMP, rsv.RSV_FORM_F64
TOL = {COMP: 1e-6, F64: 1e-12}
STEPS = 400


@pytest.fixture
def ctx():
    h = rsv.rsv_create(0, torch.cuda.current_stream())
    yield h
    rsv.rsv_destroy(h)


def book():
    pol = synth.portfolio_mix(40, seed=5)
    pol["product"][:] = np.arange(40) % 4
    pol["age2_m"][:] = np.where(pol["product"] == 1, 400 + pol["age1_m"] // 2, 0)
    pol["reversion"][:] = np.where(pol["product"] == 1, 0.6, 0.0)
    pol["term_m"][:] = 1 + np.arange(40) * 10   # annuities too: at most 391 steps
    return pol


def value(ctx, form, variant):
    n, S = 40, 33
    V, tot = np.zeros((n, S)), np.zeros(S)
    rsv.rsv_compute_reserves(ctx, form, rsv.RSV_OUT_V0 | rsv.RSV_OUT_SCEN_TOTAL, variant=variant, V0d=V, scen_total=tot)
    return V, tot


def load(ctx, pol, v):
    rsv.rsv_load_decrements(ctx, 0, synth.gm_monthly_survival())
    rsv.rsv_load_portfolio(ctx, pol)
    rsv.rsv_load_scenarios(ctx, v)


def close(a, b, tol):
    with np.errstate(invalid="ignore"):
        return np.all((a == b) | (np.isnan(a) & np.isnan(b)) | (np.abs(a - b) <= tol * np.abs(b)))


@pytest.mark.parametrize("form", [F64, COMP])
@pytest.mark.parametrize("amount", [1.0, 2.0 ** 80, 2.0 ** -50])
@pytest.mark.parametrize("size", [1e-300, 1e-50, 1e-30, 1e-20, 1e-6, 1e6, 2.0 ** 60, 1e30, 1e45, 1e200])
def test_multipliers_of_one_size(ctx, form, amount, size):
    pol = book()
    pol["amount"][:] = amount
    rng = np.random.default_rng(3)
    cf = size * rng.uniform(0.5, 2.0, (40, STEPS)) * (rng.uniform(size=(40, STEPS)) < 0.5)
    cf[::5] = 1.0
    v = synth.vasicek_paths(33, STEPS, seed=1)
    load(ctx, pol, v)
    rsv.rsv_load_cashflows(ctx, cf)
    V, tot = value(ctx, form, -1)
    W, wtot = value(ctx, form, 0)
    assert close(V, W, TOL[form]) and close(tot, wtot, TOL[form])
    if form == F64 and amount * size > 1e-290:   # below, the oracle's sums of amounts are not normal numbers
        ref, _ = oracle.reserves_batch(pol, synth.gm_monthly_survival(), v, cf=cf)
        assert close(V, ref, TOL[form])


@pytest.mark.parametrize("form", [F64, COMP])
@pytest.mark.parametrize("escalation", [1.0, -0.5, 0.5])
def test_schedules_that_grow_every_step(ctx, form, escalation):
    sch = np.zeros(40, rsv.SCHEDULE_DTYPE)
    sch["every"], sch["steps_per_year"], sch["escalation"] = 1, 1, escalation
    sch["escalation"][::3] = 0.0
    pol = book()
    v = synth.vasicek_paths(33, STEPS, seed=2)
    load(ctx, pol, v)
    rsv.rsv_load_schedules(ctx, sch, STEPS)
    V, tot = value(ctx, form, -1)
    W, wtot = value(ctx, form, 0)
    assert close(V, W, TOL[form]) and close(tot, wtot, TOL[form])
