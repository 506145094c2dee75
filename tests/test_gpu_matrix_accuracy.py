"""The matrix valuation's accuracy at ordinary spreads (rms limits close to what is stated), books of
several panels of digits, and discount products that grow.

rms limits, relative, against extended precision: FP64 5e-15 (up to 600 running products of 2^-53 each
and the sum's rounding), compensated 5e-14 (operands and left-out products 2^-46, 1.4e-14, for the
shortest contracts on their scenario's spread), deflated 2e-8."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu
COMP, DEFL, F64 = rsv.RSV_FORM_F32_COMP, rsv.RSV_FORM_F32_DEFLATED, rsv.RSV_FORM_F64
RMS = {COMP: 5e-14, DEFL: 2e-8, F64: 5e-15}
V0T = rsv.RSV_OUT_V0 | rsv.RSV_OUT_SCEN_TOTAL


@pytest.fixture
def ctx():
    h = rsv.rsv_create(0, torch.cuda.current_stream())
    rsv.rsv_load_decrements(h, 0, synth.gm_monthly_survival())
    yield h
    rsv.rsv_destroy(h)


@pytest.mark.parametrize("form", [F64, COMP, DEFL])
@pytest.mark.parametrize("steps,sigma", [(360, 0.01), (600, 0.01), (1200, 0.004), (1200, 0.01)])
def test_rms_error_of_annuities(ctx, form, steps, sigma):
    tab = synth.gm_monthly_survival().astype(np.longdouble)
    v = synth.vasicek_paths(200, steps, seed=4, sigma=sigma)
    D = np.cumprod(v.astype(np.longdouble), axis=1)
    pol = synth.portfolio_single_life(130, seed=2)
    pol["age1_m"][:] = np.linspace(1440 - min(steps, 1200), 1400, 130).astype(int)
    rsv.rsv_load_portfolio(ctx, pol)
    rsv.rsv_load_scenarios(ctx, v)
    V, tot = np.zeros((130, 200)), np.zeros(200)
    rsv.rsv_compute_reserves(ctx, form, V0T, V0d=V, scen_total=tot)
    ref = np.stack([a * (D[:, :1440 - x] @ np.cumprod(tab[x:])) for x, a in zip(pol["age1_m"], pol["amount"])])
    rel = ((V - ref) / ref).astype(np.float64)
    assert np.sqrt(np.mean(rel ** 2)) <= RMS[form]
    assert np.max(np.abs(tot - ref.sum(0)) / ref.sum(0)) <= RMS[form]


@pytest.mark.parametrize("form", [F64, COMP])
@pytest.mark.parametrize("rate", [-0.05, -0.2])
def test_negative_rates(ctx, form, rate):
    """The largest tilt lies at the end, so that it bounds the level annuities' rows."""
    pol = synth.portfolio_mix(100, seed=3)
    v = np.full((5, 1200), (1.0 + rate) ** (-1.0 / 12.0)) * (1.0 - np.linspace(0, 1e-4, 5))[:, None]
    rsv.rsv_load_portfolio(ctx, pol)
    rsv.rsv_load_scenarios(ctx, v)
    V, tot = np.zeros((100, 5)), np.zeros(5)
    rsv.rsv_compute_reserves(ctx, form, V0T, V0d=V, scen_total=tot)
    ref, ref_tot = oracle.reserves_batch(pol, synth.gm_monthly_survival(), v)
    tol = {F64: 1e-12, COMP: 5e-10}[form]
    assert np.all(np.abs(V - ref) <= tol * np.maximum(ref, 1e-9 * pol["amount"][:, None]))
    assert np.all(np.abs(tot - ref_tot) <= tol * ref_tot)


@pytest.mark.parametrize("form", [F64, COMP])
def test_several_panels(ctx, form):
    """Schedules (level and varying rows) and a pageable host result, which is computed in column blocks:
    more digits than are held at a time (1 GiB) against the same records in books of one panel, bit
    for bit, since a row's digits and sums depend on the row alone."""
    n = 100_000 if form == COMP else 60_000
    pol = synth.portfolio_mix(n, seed=7)
    sch = np.zeros(n, rsv.SCHEDULE_DTYPE)
    sch["every"], sch["steps_per_year"] = 1, 12
    sch["escalation"][::3] = 0.03
    rsv.rsv_load_scenarios(ctx, synth.vasicek_paths(260, 1200, seed=1))

    def value(i):
        part = synth.take(pol, i)
        rsv.rsv_load_portfolio(ctx, part)
        rsv.rsv_load_schedules(ctx, sch[i], 1200)
        V = np.zeros((len(part["product"]), 260))
        rsv.rsv_compute_reserves(ctx, form, V0d=V)
        return V

    V = value(slice(0, n))
    for lo in range(0, n, 25_000):
        assert np.array_equal(V[lo:lo + 25_000], value(slice(lo, min(n, lo + 25_000))))
