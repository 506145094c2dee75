"""Time scans of two threads, each on a context and stream of its own, whose launches need different
amounts of shared memory (tables 23 KB and columns of 16 or 32 KB)."""
import threading

import numpy as np
import pytest
import torch

import synth
from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu


def test_scans_in_two_threads():
    pol = synth.portfolio_single_life(40, seed=1)
    errors = []

    def work(n_scen):
        try:
            h = rsv.rsv_create(0, torch.cuda.Stream())
            rsv.rsv_load_decrements(h, 0, synth.gm_monthly_survival())
            rsv.rsv_load_portfolio(h, pol)
            rsv.rsv_load_scenarios(h, np.full((n_scen, 2000), 0.997))
            V, W = np.zeros((40, n_scen)), np.zeros((40, n_scen))
            for i in range(20000):
                rsv.rsv_compute_reserves(h, rsv.RSV_FORM_F64, variant=rsv.RSV_VARIANT_TIME_SCAN, V0d=W if i else V)
                assert i == 0 or np.array_equal(V, W)
            rsv.rsv_destroy(h)
        except Exception as e:   # handed to the test's thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(n,)) for n in (1, 2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
