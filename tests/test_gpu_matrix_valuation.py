"""The valuation as a matrix product of split operands (the default path of the
compensated and deflated forms): edges of its tiles, every reduced model and state, long
projections, varying cash flows, and the data that keeps the recurrence kernels.

Tolerances.  Compensated: operands to 2^-48 of a row's largest entry, discount products
within 2^11 of a column's largest, so 2^-34 an entry at the worst place, and FP32 truncations of an
accumulator 2^-24 below the result, at most 15 a block of 16 steps: 4,096 steps stay below
2^-33; 5e-10 covers both.  Deflated: its stated bound 15 x 2^-24.  FP64: the form's 1e-12 (the
same estimate with 2^-63, 2^-32 and 36 gives 2^-48).
Error metric: rel = |V_gpu - V_ref| / max(|V_ref|, 1e-9 * amount)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu
COMP, DEFL, F64 = rsv.RSV_FORM_F32_COMP, rsv.RSV_FORM_F32_DEFLATED, rsv.RSV_FORM_F64
TOL = {COMP: 5e-10, DEFL: 15 * 2.0 ** -24, F64: 1e-12}
V0T = rsv.RSV_OUT_V0 | rsv.RSV_OUT_SCEN_TOTAL


@pytest.fixture
def ctx():
    h = rsv.rsv_create(0, torch.cuda.current_stream())
    yield h
    rsv.rsv_destroy(h)


def value(ctx, form, pol, tabs, v, variant=-1, horizon=0):
    for i, t in enumerate(tabs):
        rsv.rsv_load_decrements(ctx, i, t)
    rsv.rsv_load_portfolio(ctx, pol)
    rsv.rsv_load_scenarios(ctx, v)
    V, tot = np.zeros((len(pol["product"]), v.shape[0])), np.zeros(v.shape[0])
    rsv.rsv_compute_reserves(ctx, form, V0T, horizon=horizon, variant=variant, V0d=V, scen_total=tot)
    return V, tot


def check(form, pol, V, tot, ref, ref_tot):
    scale = np.maximum(np.abs(ref), 1e-9 * np.abs(pol["amount"])[:, None])
    scale[scale == 0] = 1.0
    assert np.max(np.abs(V - ref) / scale) <= TOL[form]
    assert np.all(np.abs(tot - ref_tot) <= TOL[form] * np.maximum(np.abs(ref).sum(0), 1e-300))


def every_product(n, seed, form, **ages):
    pol = synth.portfolio_mix(n, seed=seed, **ages)
    two = synth.portfolio_two_life(n, seed=seed, products=(4, 5) if form == DEFL else (4, 5, 6, 7, 8, 9), **ages)
    pol = {k: np.concatenate([pol[k], two[k]]) for k in pol}
    multi = np.where((pol["product"] == 1) | (pol["product"] == 5) | (pol["product"] >= 8))[0]
    pol["state0"][multi[::3]] = 1
    pol["state0"][multi[1::3]] = 2
    return pol


@pytest.mark.parametrize("form", [COMP, DEFL, F64])
@pytest.mark.parametrize("n_pol,n_scen", [(1, 1), (2, 31), (63, 33), (64, 127), (65, 128), (129, 129), (257, 300)])
def test_tile_edges(ctx, form, n_pol, n_scen):
    tabs = [synth.gm_monthly_survival(), synth.gm_monthly_survival(A=0.0003, B=0.00002)]
    pol = every_product(n_pol, n_pol + n_scen, form)
    pol["table2"][pol["product"] >= 4] = 1
    pol["amount"][::7] *= -1.0
    pol["amount"][3::11] = 0.0
    v = synth.vasicek_paths(n_scen, 1200, seed=n_scen)
    ref, ref_tot = oracle.reserves_batch(pol, np.stack(tabs), v)
    check(form, pol, *value(ctx, form, pol, tabs, v), ref, ref_tot)


@pytest.mark.parametrize("form", [COMP, DEFL, F64])
@pytest.mark.parametrize("horizon", [1, 31, 32, 33, 64, 65, 0])
def test_projection_lengths(ctx, form, horizon):
    """Around the 32-step blocks; without a horizon also policies at maturity and lives at
    and past the limiting age."""
    tab = synth.gm_monthly_survival()
    pol = every_product(40, 3, form)
    spec = [(3, 900, 0), (2, 1440, 24), (3, 1439, 1), (0, 1440, 0), (0, 1439, 0), (2, 1450, 12), (3, 1408, 64)]
    for i, (p, age, term) in enumerate(spec):
        pol["product"][i], pol["age1_m"][i], pol["term_m"][i], pol["state0"][i] = p, age, term, 0
        pol["age2_m"][i], pol["reversion"][i] = 0, 0.0
    v = synth.vasicek_paths(40, 1200, seed=2)
    ref, ref_tot = oracle.reserves_batch(pol, tab, v, horizon=horizon)
    V, tot = value(ctx, form, pol, [tab], v, horizon=horizon)
    check(form, pol, V, tot, ref, ref_tot)
    if horizon == 0:
        assert np.all(V[0] == pol["amount"][0])


@pytest.mark.parametrize("form", [COMP, DEFL, F64])
@pytest.mark.parametrize("steps", [1000, 1001, 2001, 4001])
def test_long_level_projections(ctx, form, steps):
    """No mortality and no interest to speak of: every entry near the row's largest, the sums
    that the leading digits must hold exactly."""
    tab = np.full(4090, 1.0 - 1e-7)
    pol = synth.portfolio_single_life(5, seed=1)
    pol["age1_m"][:], pol["term_m"][:] = np.arange(5), steps
    v = np.full((3, steps), 1.0 - np.array([[1e-9], [1e-7], [1e-6]]))
    ref, ref_tot = oracle.reserves_batch(pol, tab, v)
    check(form, pol, *value(ctx, form, pol, [tab], v), ref, ref_tot)


@pytest.mark.parametrize("form", [COMP, DEFL, F64])
@pytest.mark.parametrize("bits", [3, 4, 5, 7, 8, 9, 10])
def test_scenarios_far_from_their_mean(ctx, form, bits):
    """Flat rates whose discount products end 2^bits apart from their mean's, single payments
    where the discount product is smallest against its scenario's largest."""
    tab = synth.gm_monthly_survival()
    pol = every_product(60, bits, form)
    pol["product"][:12], pol["term_m"][:12], pol["state0"][:12] = 2, 1, 0
    pol["age1_m"][:12] = np.arange(240, 1440, 100)
    pol["age1_m"][12:15], pol["product"][12:15], pol["state0"][12:15] = 1439, 0, 0
    slope = np.linspace(-1, 1, 41)[:, None] * (bits - 0.01) * np.log(2.0) / 1200
    v = np.exp(-0.0033 - slope + np.zeros((41, 1200)))
    ref, ref_tot = oracle.reserves_batch(pol, tab, v)
    check(form, pol, *value(ctx, form, pol, [tab], v), ref, ref_tot)


@pytest.mark.parametrize("form", [COMP, F64])
def test_varying_cash_flows(ctx, form):
    """Rows that are level and rows that are not, deferred and annual payments."""
    tab = synth.gm_monthly_survival()
    pol = every_product(90, 8, COMP)
    n = len(pol["product"])
    rng = np.random.default_rng(4)
    cf = rng.uniform(0.0, 2.0, (n, 1200)) * (rng.uniform(size=(n, 1200)) < 0.3)
    cf[::2] = 1.0
    cf[1::10, :400] = 0.0
    v = synth.vasicek_paths(70, 1200, seed=9)
    rsv.rsv_load_decrements(ctx, 0, tab)
    rsv.rsv_load_portfolio(ctx, pol)
    rsv.rsv_load_cashflows(ctx, cf)
    V, tot = value(ctx, form, pol, [tab], v)
    ref, ref_tot = oracle.reserves_batch(pol, tab, v, cf=cf)
    check(form, pol, V, tot, ref, ref_tot)


@pytest.mark.parametrize("form", [COMP, DEFL, F64])
@pytest.mark.parametrize("what", ["spread", "discount", "large", "small", "table"])
def test_data_out_of_range_keeps_the_recurrence(ctx, form, what):
    tab, v = synth.gm_monthly_survival(), synth.vasicek_paths(33, 1200, seed=1)
    pol = synth.portfolio_mix(50, seed=5)
    if what == "spread":
        v[3] = 1.01
    if what == "discount":
        v[:] = 0.95
    if what == "large":
        pol["amount"][7] = 1e30
    if what == "small":
        pol["amount"][7] = 1e-25
    if what == "table":
        tab = synth.constant_force_table(0.8)
    a, b = value(ctx, form, pol, [tab], v), value(ctx, form, pol, [tab], v, variant=0)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("n,n_scen", [(1, 1), (127, 31), (128, 128), (130, 129)])
def test_lives_against_the_fp64_form(ctx, n, n_scen):
    """Contracts on one to four lives with every k, both families, dead lives at valuation,
    lives at and past the limiting age: the FP64 kernel applies the lives' transitions to
    every chain."""
    rng = np.random.default_rng(n)
    rec = np.zeros(n, rsv.MLIFE_DTYPE)
    rec["m"] = 1 + np.arange(n) % 4
    rec["kind"] = (np.arange(n) // 4) % 2
    rec["k"] = 1 + rng.integers(0, 100, n) % rec["m"]
    rec["age_m"] = rng.integers(200, 1300, (n, 4))
    rec["age_m"][::9, 0] = 1440
    rec["age_m"][4::9, 0] = 1450
    rec["table"] = rng.integers(0, 2, (n, 4))
    rec["term_m"] = np.where(rec["kind"] == 1, rng.integers(1, 480, n), np.where(np.arange(n) % 3, 0, 200))
    spare = np.where(rec["kind"] == 1, rec["k"] - 1, rec["m"] - rec["k"])   # lives that may be dead already
    rec["dead0"] = np.where(spare > 0, rng.integers(0, 2, n), 0)
    rec["amount"] = rng.lognormal(5.0, 2.0, n)
    for i, t in enumerate([synth.gm_monthly_survival(), synth.gm_monthly_survival(A=0.0003, B=0.00002)]):
        rsv.rsv_load_decrements(ctx, i, t)
    rsv.rsv_load_scenarios(ctx, synth.vasicek_paths(n_scen, 1240, seed=n))
    res = {}
    for form in (rsv.RSV_FORM_F64, COMP):
        V, tot = np.zeros((n, n_scen)), np.zeros(n_scen)
        rsv.rsv_compute_mlife(ctx, rec, form, V0T, V0d=V, scen_total=tot)
        res[form] = V, tot
    V, tot = res[rsv.RSV_FORM_F64]
    scale = np.maximum(np.abs(V), 1e-9 * rec["amount"][:, None])
    assert np.max(np.abs(res[COMP][0] - V) / scale) <= TOL[COMP]
    assert np.all(np.abs(res[COMP][1] - tot) <= TOL[COMP] * tot)
