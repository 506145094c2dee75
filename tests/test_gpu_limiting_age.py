"""A contract that matures now on a life at the limiting age, the book's oldest record: due in full
in reserves and at the first node of a nested run, whatever the layout's padding of the tables.

Tolerances: the sum due is the amount itself; in the nested runs it is a difference of two
liabilities, 1e-12 of them in FP64 walks and the stated 4e-10 in the deflated form."""
import numpy as np
import pytest
import torch

import synth
from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu
F64, COMP, DEFL = rsv.RSV_FORM_F64, rsv.RSV_FORM_F32_COMP, rsv.RSV_FORM_F32_DEFLATED
CASES = [(f, t, p) for f in (F64, COMP, DEFL) for t in (1, 2) for p in (3, 7, 9) if f != DEFL or p == 3]


def book(n_tables, product, matured):
    pol = np.zeros(1 + matured, rsv.POLICY_DTYPE)
    pol["age1_m"], pol["amount"] = 720, 100.0
    if matured:
        pol["product"][1], pol["age1_m"][1], pol["amount"][1] = product, 1440, 1000.0
        pol["age2_m"][1] = 1440 if product > 3 else 0
        pol["table1"][1] = n_tables - 1
        pol["table2"][1] = n_tables - 1 if product > 3 else 0
    return pol


@pytest.fixture
def ctx():
    h = rsv.rsv_create(0, torch.cuda.current_stream())
    yield h
    rsv.rsv_destroy(h)


def tables(ctx, n):
    rsv.rsv_load_decrements(ctx, 0, synth.gm_monthly_survival())
    if n > 1:
        rsv.rsv_load_decrements(ctx, 1, synth.gm_monthly_survival(A=0.0003, B=0.00002))


@pytest.mark.parametrize("form,n_tables,product", CASES)
def test_reserve(ctx, form, n_tables, product):
    tables(ctx, n_tables)
    rsv.rsv_load_scenarios(ctx, synth.vasicek_paths(33, 720, seed=1))
    rsv.rsv_load_portfolio(ctx, book(n_tables, product, 1))
    for variant in (-1, 0):
        V = np.zeros((2, 33))
        rsv.rsv_compute_reserves(ctx, form, variant=variant, V0d=V)
        assert np.all(V[1] == 1000.0) and np.all(V[0] > 1000.0)


@pytest.mark.parametrize("form,n_tables,product", CASES)
def test_nested(ctx, form, n_tables, product):
    tables(ctx, n_tables)
    L = []
    for matured in (0, 1):
        rsv.rsv_load_portfolio(ctx, book(n_tables, product, matured))
        mean, q = np.zeros((2, 3)), np.zeros((2, 3))
        rsv.rsv_compute_nested(ctx, form, n_outer=2, n_nodes=3, n_inner=64, seed=3, L_mean=mean, L_q995=q)
        L.append(mean)
    due = np.array([1000.0, 0.0, 0.0])
    assert np.all(np.abs(L[1] - L[0] - due) <= (4e-10 if form == DEFL else 1e-12) * L[1])
