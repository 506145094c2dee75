"""Loading: the device's check of the discount factors, and books at the edges of the parts
that the host lays them out in (8,192 records)."""
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


def book(n):
    rng = np.random.default_rng(n)
    pol = np.zeros(n, rsv.POLICY_DTYPE)
    pol["product"] = rng.integers(0, 3, n)
    pol["age1_m"], pol["age2_m"] = rng.integers(300, 1000, n), rng.integers(300, 1000, n)
    pol["term_m"] = rng.integers(1, 400, n)
    pol["reversion"] = rng.uniform(0, 1, n)
    pol["amount"] = rng.uniform(1, 2, n)
    return pol


@pytest.mark.parametrize("bad", [0.0, -1.0, np.inf, np.nan])
@pytest.mark.parametrize("at", [(0,), (1199,), (37 * 1200 - 1,), (20000, 20001, 44000)])
def test_bad_factor(ctx, bad, at):
    pol = book(5)
    good = np.full((37, 1200), 0.997)
    V, W = np.zeros((5, 37)), np.zeros((5, 37))
    rsv.rsv_load_portfolio(ctx, pol)
    rsv.rsv_load_scenarios(ctx, good)
    rsv.rsv_compute_reserves(ctx, V0d=V)
    v = np.full((37, 1200), 0.9)
    v.ravel()[list(at)] = bad
    with pytest.raises(rsv.RsvError, match=f"discount factor {at[0]} "):
        rsv.rsv_load_scenarios(ctx, v)
    rsv.rsv_compute_reserves(ctx, V0d=W)   # the loaded set stands
    assert np.array_equal(V, W)


@pytest.mark.parametrize("n", [8191, 8192, 16384, 40001])
def test_book_in_parts(ctx, n):
    """A book laid out in one or several parts against its pieces of 4,000 records, one part
    each: the same reserves up to the FP32-digit product's 1e-12."""
    pol = book(n)
    rsv.rsv_load_scenarios(ctx, np.full((3, 1200), [[0.995], [0.997], [0.999]]))
    V = np.zeros((n, 3))
    rsv.rsv_load_portfolio(ctx, pol)
    rsv.rsv_compute_reserves(ctx, V0d=V)
    for lo in range(0, n, 4000):
        part = pol[lo:lo + 4000]
        W = np.zeros((len(part), 3))
        rsv.rsv_load_portfolio(ctx, part)
        rsv.rsv_compute_reserves(ctx, V0d=W)
        assert np.allclose(V[lo:lo + 4000], W, rtol=1e-12, atol=0.0)
