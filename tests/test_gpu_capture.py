"""On-device valuations captured into a CUDA graph after the scenarios or the book were loaded anew
(same sizes, one valuation before): the replay, and the calls before and after it, give what a
context of its own gives, bit for bit."""
import numpy as np
import pytest
import torch

import synth
from paper_1401_1757_gb300 import rsv

pytestmark = pytest.mark.gpu
F64, COMP, DEFL = rsv.RSV_FORM_F64, rsv.RSV_FORM_F32_COMP, rsv.RSV_FORM_F32_DEFLATED
OUT = rsv.RSV_OUT_V0 | rsv.RSV_OUT_SCEN_TOTAL


class Context:
    def __init__(self, form):
        self.form, self.stream = form, torch.cuda.Stream()
        self.h = rsv.rsv_create(0, self.stream)
        self.V = torch.zeros(300, 100, device="cuda", dtype=torch.float64)
        self.tot = torch.zeros(100, device="cuda", dtype=torch.float64)
        rsv.rsv_load_decrements(self.h, 0, synth.gm_monthly_survival())

    def scenarios(self, seed):   # a higher volatility spreads the set, so that the digits change
        rsv.rsv_load_scenarios(self.h, synth.vasicek_paths(100, 1200, seed=seed, sigma=0.004 if seed % 2 else 0.01))

    def book(self, seed):
        rsv.rsv_load_portfolio(self.h, synth.portfolio_mix(300, seed=seed))

    def call(self):
        rsv.rsv_compute_reserves(self.h, self.form, OUT, on_device=True, V0d=self.V, scen_total=self.tot)

    def result(self):
        self.stream.synchronize()
        return self.V.clone(), self.tot.clone()

    def close(self):
        rsv.rsv_destroy(self.h)


def same(a, b):
    return torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("form", [F64, COMP, DEFL])
@pytest.mark.parametrize("replay_first", [True, False])
def test_capture_after_reload(form, replay_first):
    c = Context(form)
    with torch.cuda.stream(c.stream):
        c.scenarios(1), c.book(1), c.call()
        for what, seed in [("scenarios", 2), ("scenarios", 3)] + ([("book", 4), ("scenarios", 6)] if form != DEFL else []):
            getattr(c, what)(seed)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=c.stream):
                c.call()
            ref = Context(form)
            with torch.cuda.stream(ref.stream):
                ref.scenarios(3 if what == "book" else seed), ref.book(4 if seed >= 4 else 1), ref.call()
            want = ref.result()
            ref.close()
            got = []
            for step in (["replay", "call"] if replay_first else ["call", "replay"]) + ["call", "replay"]:
                c.V.zero_(), c.tot.zero_()
                if step == "replay":
                    graph.replay()
                elif what == "book" and not replay_first and not got:
                    graph.replay()   # the book's records travel with the graph
                else:
                    c.call()
                got.append(c.result())
            assert all(same(g, want) for g in got), (what, seed, [same(g, want) for g in got])
    c.close()
