"""Matrix valuation: projections whose operands stay near one value, so that the products of a
digit level add up with one sign over the whole projection, the largest sums that an accumulator
meets.

Reference: sum of D(t) E(t) in extended precision.  Tolerances, relative.  FP64: the running
products of 4,000 factors, at most 2^-53 a factor and two of them, 9e-13, and the form's 63-bit
operands; 1e-12 in all.  Compensated: the same and operands and left-out digit products of
2^-45 (3e-14); 1e-12.  Deflated: the stated 15 x 2^-24."""
import numpy as np
import pytest
import torch

import synth
from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu
COMP, DEFL, F64 = rsv.RSV_FORM_F32_COMP, rsv.RSV_FORM_F32_DEFLATED, rsv.RSV_FORM_F64
TOL = {COMP: 1e-12, DEFL: 15 * 2.0 ** -24, F64: 1e-12}


@pytest.fixture
def ctx():
    h = rsv.rsv_create(0, torch.cuda.current_stream())
    yield h
    rsv.rsv_destroy(h)


@pytest.mark.parametrize("form", [COMP, DEFL, F64])
@pytest.mark.parametrize("steps", [250, 256, 257, 512, 1000, 1001, 1025, 2001, 4000])
def test_digits_of_one_sign(ctx, form, steps):
    """First factors from 0.992 to 0.9999, then a drift of 0 to about 1e-6 a step."""
    drift = np.array([0.0, 1e-9, 1.1e-7, 1.2e-6])
    first = np.array([0.9960, 0.99305, 0.9999, 0.9961])
    v = np.tile(1.0 - drift[:, None], (1, steps))
    v[:, 0] = first
    pol = synth.portfolio_single_life(1, seed=1)
    pol["age1_m"][:], pol["term_m"][:] = 0, steps
    rsv.rsv_load_portfolio(ctx, pol)
    rsv.rsv_load_scenarios(ctx, v)
    D = np.cumprod(v.astype(np.longdouble), axis=1)
    for f, d in zip(first[::-1], drift):
        tab = np.full(4090, 1.0 - d)
        tab[0] = f
        rsv.rsv_load_decrements(ctx, 0, tab)
        V, tot = np.zeros((1, len(v))), np.zeros(len(v))
        rsv.rsv_compute_reserves(ctx, form, rsv.RSV_OUT_V0 | rsv.RSV_OUT_SCEN_TOTAL, V0d=V, scen_total=tot)
        ref = D @ np.cumprod(tab[:steps].astype(np.longdouble)) * pol["amount"][0]
        assert np.max(np.abs(V[0] - ref) / ref) <= TOL[form]
        assert np.max(np.abs(tot - ref) / ref) <= TOL[form]
