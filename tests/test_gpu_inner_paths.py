"""The nested run's inner paths, valued while they are generated on the portfolio's
expected cash flows: the double-float generator of the deflated form against the FP64
one, and tables at the edges of the survivor columns against the FP64 oracle.

Tolerance of the two generators: a month's random walk and discount product are
carried to about 2^-46, and a rate error lives on for some 120 months of a twelfth each, so a
month adds at most about 2^-42 to the discount product; 1,440 months stay below 4e-10."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu
F64, DEFL, COMP = rsv.RSV_FORM_F64, rsv.RSV_FORM_F32_DEFLATED, rsv.RSV_FORM_F32_COMP


@pytest.fixture
def ctx():
    h = rsv.rsv_create(0, torch.cuda.current_stream())
    yield h
    rsv.rsv_destroy(h)


def liabilities(ctx, form, pol, tab, **spec):
    rsv.rsv_load_decrements(ctx, 0, tab)
    rsv.rsv_load_portfolio(ctx, pol)
    on = (spec["n_outer"], spec["n_nodes"])
    L, m, q = np.zeros(on + (spec["n_inner"],)), np.zeros(on), np.zeros(on)
    rsv.rsv_compute_nested(ctx, form, **spec, L_mean=m, L_q995=q, L_all=L)
    return L


@pytest.mark.parametrize("n_outer,n_nodes,step,n_inner", [(1, 1, 1, 1), (3, 5, 7, 43), (2, 3, 12, 64), (1, 2, 12, 129),
                                                          (5, 122, 12, 11), (1, 4, 399, 257)])
def test_double_float_generator_matches_fp64(ctx, n_outer, n_nodes, step, n_inner):
    tab = synth.gm_monthly_survival()
    pol = synth.portfolio_mix(37, seed=n_inner, age_lo_y=0, age_hi_y=119)
    spec = dict(n_outer=n_outer, n_nodes=n_nodes, node_step_m=step, n_inner=n_inner, seed=(1 << 40) + n_inner)
    a, b = (liabilities(ctx, f, pol, tab, **spec) for f in (F64, DEFL))
    assert np.all(np.abs(b - a) <= 4e-10 * np.abs(a))


def test_models_outside_the_double_float_range_run_in_fp64(ctx):
    tab = synth.gm_monthly_survival()
    pol = synth.portfolio_mix(20, seed=3)
    for model in (dict(b=0.3, r0=0.3), dict(r0=0.4), dict(sigma=0.1)):
        spec = dict(n_outer=2, n_nodes=3, node_step_m=12, n_inner=50, seed=1, **model)
        assert np.array_equal(liabilities(ctx, F64, pol, tab, **spec), liabilities(ctx, DEFL, pol, tab, **spec))


@pytest.mark.parametrize("table", ["below 2^-512", "zero inside", "all die"])
def test_survivor_columns_at_their_edges(ctx, table):
    tab = synth.constant_force_table(4.0)
    if table == "zero inside":
        tab = synth.gm_monthly_survival()
        tab[900] = 0.0
    if table == "all die":
        tab = np.zeros(40)
    pol = synth.portfolio_mix(24, seed=9, age_lo_y=0, age_hi_y=118)
    two = synth.portfolio_two_life(24, seed=9, age_lo_y=0, age_hi_y=118, products=(4, 5, 6, 7, 8, 9))
    pol = {k: np.concatenate([pol[k], two[k]]) for k in pol}
    jl = np.where((pol["product"] == 1) | (pol["product"] >= 8))[0]
    pol["state0"][jl[::3]] = 1
    pol["state0"][jl[1::3]] = 2
    spec = dict(n_outer=1, n_nodes=3, node_step_m=60, n_inner=9, seed=5)
    for form in (F64, COMP):
        L = liabilities(ctx, form, pol, tab, **spec)
        for n in range(3):
            ref, _, _ = oracle.nested_node(pol, tab, 5, 0, n, np.arange(9), node_step=60)
            assert np.all(np.abs(L[0, n] - ref) <= 1e-11 * np.abs(ref)), (form, n)
