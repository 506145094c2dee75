"""What the library is measured on: one call each through its public entry points
(paper_1401_1757_gb300.rsv, the binding of include/rsv.h).

A case names a family and its sizes:

* ``reserves``  rsv_compute_reserves of a loaded book under a loaded scenario set;
* ``mlife``     rsv_compute_mlife of a book of contracts on one to four lives;
* ``nested``    rsv_compute_nested, the brute-force Solvency II run;
* ``network``   rsv_mlp_gradient, one training step's gradient of the surrogate.

Books, scenarios and schedules follow the distributions of this repository's
configurations; every array is drawn from the seed.  Discount factors are
Vasicek paths (a 0.1, b 0.04, sigma 0.01, r0 0.03), mortality is
Gompertz-Makeham to age 120, ages and terms are whole months.
"""
import math

import numpy as np
import torch

from paper_1401_1757_gb300 import rsv

A, B, SIGMA, R0, DT = 0.1, 0.04, 0.01, 0.03, 1.0 / 12.0
LIMIT = 1440                       # age 120 in months
FORMS = {"f64": rsv.RSV_FORM_F64, "comp": rsv.RSV_FORM_F32_COMP, "deflated": rsv.RSV_FORM_F32_DEFLATED}
V0, TOTALS = rsv.RSV_OUT_V0, rsv.RSV_OUT_SCEN_TOTAL


def reserves(name, book, form, n_pol, n_scen, n_steps=1200, horizon=0, out="f32", place="device", flat=False,
             schedules=False):
    return dict(name=name, family="reserves", book=book, form=form, n_pol=n_pol, n_scen=n_scen, n_steps=n_steps,
                horizon=horizon, out=out, place=place, flat=flat, schedules=schedules)


def listed():
    return [
        # The smallest call: a book of pensions in payment at one flat rate, exact; what a pricing
        # or a reporting program asks for many times over (configuration 1).
        reserves("flat rate exact", "annuities", "f64", 1000, 1, n_steps=720, out="f64", flat=True),
        # A small book with an odd number of scenarios, results to ordinary host arrays: the
        # interactive call in the default form.
        reserves("small mixed book host", "mix", "comp", 1537, 157, out="f64", place="host"),
        # A whole office's in-force book under the 1,000 scenarios of Solvency II, default form
        # (configuration 2).
        reserves("mixed book", "mix", "comp", 100_000, 1000),
        # The same in the form that is fastest within 1e-6.
        reserves("mixed book deflated", "mix", "deflated", 100_000, 1000),
        # The largest: a million annuities, 50 years (configuration 5, the benchmark's headline).
        reserves("million annuities deflated", "annuities", "deflated", 1_000_000, 1000, n_steps=600, horizon=600),
        # End to end: records and scenarios reloaded from host memory in the call, reserves
        # delivered into page-locked host memory.
        reserves("book reloaded deflated", "annuities", "deflated", 100_000, 1000, n_steps=600, horizon=600,
                 place="reload"),
        # Escalating and annual payments (the paper's cohort, Section 5) as cash-flow schedules.
        reserves("scheduled payments", "mix", "comp", 20_000, 1000, schedules=True),
        # Two-life products in full precision: the run that others are checked against.
        reserves("two lives exact", "two_life", "f64", 3000, 333, out="f64"),
        # Contracts on up to four lives (Section 4.3).
        dict(name="up to four lives", family="mlife", form="comp", n_pol=5000, n_scen=1000, n_steps=1200),
        # Nested valuation by brute force, at full size (configuration 3).
        dict(name="nested deflated", family="nested", book="annuities", form="deflated", n_pol=2000, n_outer=100,
             n_nodes=40, n_inner=1000),
        # A few outer paths of a mixed book in the default form: what an outer path costs.
        dict(name="nested mixed book", family="nested", book="mix", form="comp", n_pol=331, n_outer=8, n_nodes=25,
             n_inner=1000),
        # One training step of the surrogate: forward and backward at the batch that it trains with.
        dict(name="surrogate gradient", family="network", rows=8192),
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["scan", "comp", "comp", "deflated", "deflated", "deflated", "reload", "schedules", "f64",
                       "mlife", "nested", "nested", "nested_comp", "network"])
    if kind == "scan":
        return _unnamed(reserves("", "annuities", "f64", log_int(rng, 200, 20_000), 1, n_steps=720, out="f64", flat=True))
    if kind == "comp":
        place = rng.choice(["device", "device", "host"])
        n = log_int(rng, 100, 5000) if place == "host" else log_int(rng, 300, 60_000)
        return _unnamed(reserves("", rng.choice(["mix", "mix", "two_life", "annuities"]), "comp", n,
                                 log_int(rng, 33, 1000), out=rng.choice(["f32", "f64"]) if n < 5000 else "f32",
                                 place=place))
    if kind == "deflated":
        T = rng.choice([360, 600, 1200])
        return _unnamed(reserves("", rng.choice(["mix", "annuities"]), "deflated", log_int(rng, 500, 300_000),
                                 log_int(rng, 50, 1000), n_steps=T, horizon=T if T < 1200 else 0))
    if kind == "reload":
        return _unnamed(reserves("", rng.choice(["mix", "annuities"]), "deflated", log_int(rng, 1000, 100_000),
                                 log_int(rng, 50, 1000), n_steps=600, horizon=600, place="reload"))
    if kind == "schedules":
        return _unnamed(reserves("", "mix", "comp", log_int(rng, 500, 20_000), log_int(rng, 50, 1000), schedules=True))
    if kind == "f64":
        return _unnamed(reserves("", rng.choice(["mix", "two_life"]), "f64", log_int(rng, 100, 3000),
                                 log_int(rng, 30, 333), out="f64"))
    if kind == "mlife":
        return dict(family="mlife", form="comp", n_pol=log_int(rng, 100, 5000), n_scen=log_int(rng, 50, 1000),
                    n_steps=1200)
    if kind in ("nested", "nested_comp"):
        small = kind == "nested_comp"
        return dict(family="nested", book=rng.choice(["annuities", "mix"]), form="comp" if small else "deflated",
                    n_pol=log_int(rng, 50, 331 if small else 2000), n_outer=log_int(rng, 2, 8 if small else 60),
                    n_nodes=log_int(rng, 3, 25 if small else 40), n_inner=log_int(rng, 100, 1000))
    return dict(family="network", rows=64 * log_int(rng, 4, 128))


def _unnamed(case):
    del case["name"]
    return case


# ---- inputs -----------------------------------------------------------------
def mortality():
    k, lnc = np.arange(LIMIT, dtype=np.float64), math.log(1.1)
    return np.exp(-(0.0005 / 12 + 0.00003 * np.exp(lnc * k / 12) * math.expm1(lnc / 12) / lnc))


def step_moments():
    e, g, h = math.exp(-A * DT), -math.expm1(-A * DT), -math.expm1(-2 * A * DT)
    var_r, cov = SIGMA ** 2 * h / (2 * A), SIGMA ** 2 / (2 * A * A) * g * g
    var_i = (SIGMA / A) ** 2 * (DT - 2 * g / A + h / (2 * A))
    l11 = math.sqrt(var_r)
    l21 = cov / l11
    return e, g / A, l11, l21, math.sqrt(max(var_i - l21 * l21, 0.0))


def scenarios(case, seed):
    """Monthly discount factors [n_scen, n_steps]."""
    S, T = case["n_scen"], case["n_steps"]
    if case.get("flat"):
        return np.full((S, T), (1.04 + 1e-4 * (seed % 97)) ** -DT)
    e, k1, l11, l21, l22 = step_moments()
    z = np.random.default_rng([seed, 2]).standard_normal((T, 2, S))
    r, v = np.full(S, R0), np.empty((T, S))
    for t in range(T):
        v[t] = np.exp(-(B * DT + (r - B) * k1 + l21 * z[t, 0] + l22 * z[t, 1]))
        r = B + (r - B) * e + l11 * z[t, 0]
    return np.ascontiguousarray(v.T)


def book(case, seed):
    """Policy records: annuities in payment (ages 60-90), the 40/20/20/20 mix of annuities,
    reversionary annuities, term assurances and endowments (ages 20-85), or the six two-life
    products."""
    n, kind = case["n_pol"], case["book"]
    rng = np.random.default_rng([seed, 1])
    pol = np.zeros(n, rsv.POLICY_DTYPE)
    lo, hi = (720, 1080) if kind == "annuities" else (240, 1020)
    pol["age1_m"] = rng.integers(lo, hi + 1, n)
    other = rng.integers(lo, hi + 1, n)
    if kind == "annuities":
        prod = np.zeros(n, np.int64)
    elif kind == "mix":
        prod = rng.choice(4, n, p=[0.4, 0.2, 0.2, 0.2])
    else:
        prod = rng.integers(4, 10, n)
    pol["product"] = prod
    two = (prod == 1) | (prod >= 4)
    pol["age2_m"] = np.where(two, other, 0)
    term = np.isin(prod, (2, 6, 8))
    endow = np.isin(prod, (3, 7, 9))
    pol["term_m"] = 12 * np.where(term, rng.integers(5, 41, n), np.where(endow, rng.integers(10, 31, n), 0))
    pol["amount"] = np.where(term | endow, rng.lognormal(math.log(1e5), 0.5, n), rng.lognormal(math.log(1e4), 0.5, n) / 12)
    pol["reversion"] = np.where(prod == 1, rng.uniform(0.5, 1.0, n), 0.0)
    return pol


def schedules(case, seed):
    """About 80% paid monthly, 20% annually on the anniversary; 5% escalating."""
    n = case["n_pol"]
    rng = np.random.default_rng([seed, 3])
    sch = np.zeros(n, rsv.SCHEDULE_DTYPE)
    sch["since"] = rng.integers(0, 12, n)
    annual = rng.uniform(size=n) < 0.2
    sch["every"] = np.where(annual, 12, 1)
    sch["first"] = np.where(annual, 11 - sch["since"], 0)
    sch["steps_per_year"] = 12
    sch["escalation"] = np.where(rng.uniform(size=n) < 0.05, rng.choice([0.03, 0.0425, 0.05], n), 0.0)
    return sch


def lives(case, seed):
    """Two to four lives, k-of-m annuities and k-th death assurances in equal parts."""
    n = case["n_pol"]
    rng = np.random.default_rng([seed, 4])
    pol = np.zeros(n, rsv.MLIFE_DTYPE)
    pol["m"] = rng.integers(2, 5, n)
    pol["kind"] = np.arange(n) % 2
    pol["k"] = 1 + rng.integers(0, 1 << 20, n) % pol["m"]
    pol["age_m"] = rng.integers(360, 961, (n, 4))
    assurance = pol["kind"] == 1
    pol["term_m"] = np.where(assurance, 12 * rng.integers(5, 41, n), 0)
    pol["amount"] = np.where(assurance, rng.lognormal(math.log(1e5), 0.5, n), rng.lognormal(math.log(1e4), 0.5, n) / 12)
    return pol


def network_batch(case, seed):
    """Feature rows as the surrogate forms them (one-hot product and state, scaled ages, term,
    rate and their products) and normalised targets."""
    n, rng = case["rows"], np.random.default_rng([seed, 5])
    X = np.zeros((n, 32), np.float32)
    X[np.arange(n), rng.integers(0, 4, n)] = 1
    X[np.arange(n), 4 + rng.integers(0, 3, n)] = 1
    X[:, 7:19] = rng.normal(0.0, 0.6, (n, 12))
    return X, rng.standard_normal(n).astype(np.float32)


def network_params(seed):
    """He-normal weights, no biases, in the flat layout of the interface."""
    rng = np.random.default_rng([seed, 6])
    sizes = [(32, 256), (256, 256), (256, 256), (256, 256)]
    parts = [np.concatenate([rng.normal(0.0, math.sqrt(2 / i), i * o), np.zeros(o)]) for i, o in sizes]
    return np.concatenate(parts + [rng.normal(0.0, 1 / 16, 256), np.zeros(1)]).astype(np.float32)


class State:
    """A context with its data loaded, the output buffers, and what a call passes."""

    def __init__(self, case):
        self.case, self.ctx = case, rsv.rsv_create(0, torch.cuda.current_stream())

    def __del__(self):
        rsv.rsv_destroy(self.ctx)


def prepare(case, seed):
    s = State(case)
    if case["family"] == "network":
        rsv.rsv_mlp_set_params(s.ctx, network_params(seed))
        s.X, s.target = network_batch(case, seed)
        return s
    rsv.rsv_load_decrements(s.ctx, 0, mortality())
    if case["family"] == "nested":
        rsv.rsv_load_portfolio(s.ctx, book(case, seed))
        on = (case["n_outer"], case["n_nodes"])
        s.out = {k: torch.empty(on, dtype=torch.float64, device="cuda") for k in ("L_mean", "L_q995", "r_node", "D0")}
        s.seed = seed
        return s
    n, S = case["n_pol"], case["n_scen"]
    v = scenarios(case, seed)
    rsv.rsv_load_scenarios(s.ctx, v)
    if case["family"] == "mlife":
        s.pol = lives(case, seed)
        s.V0 = torch.empty((n, S), dtype=torch.float64, device="cuda")
        s.total = torch.empty(S, dtype=torch.float64, device="cuda")
        return s
    s.pol = book(case, seed)
    rsv.rsv_load_portfolio(s.ctx, s.pol)
    if case["schedules"]:
        rsv.rsv_load_schedules(s.ctx, schedules(case, seed), case["n_steps"])
    wide = torch.float64 if case["out"] == "f64" else torch.float32
    if case["place"] == "device":
        s.V0 = torch.empty((n, S), dtype=wide, device="cuda")
        s.total = torch.empty(S, dtype=torch.float64, device="cuda")
    elif case["place"] == "reload":
        s.V0 = torch.empty((n, S), dtype=wide, pin_memory=True)
        s.total = torch.empty(S, dtype=torch.float64, pin_memory=True)
        s.v = torch.from_numpy(v).pin_memory()
    else:
        s.V0 = np.empty((n, S), np.float64 if case["out"] == "f64" else np.float32)
        s.total = np.empty(S)
    return s


def run(s):
    case = s.case
    if case["family"] == "network":
        return rsv.rsv_mlp_gradient(s.ctx, s.X, s.target)
    form = FORMS[case["form"]]
    if case["family"] == "mlife":
        rsv.rsv_compute_mlife(s.ctx, s.pol, form, V0 | TOTALS, on_device=True, V0d=s.V0, scen_total=s.total)
        return {"V0": s.V0, "total": s.total}
    if case["family"] == "nested":
        rsv.rsv_compute_nested(s.ctx, form, n_outer=case["n_outer"], n_nodes=case["n_nodes"], n_inner=case["n_inner"],
                               seed=s.seed, a=A, b=B, sigma=SIGMA, r0=R0, on_device=True, **s.out)
        return {k: narrow(case, x) if k[0] == "L" else x for k, x in s.out.items()}
    if case["place"] == "reload":
        rsv.rsv_load_portfolio(s.ctx, s.pol)
        rsv.rsv_load_scenarios(s.ctx, s.v)
    rsv.rsv_compute_reserves(s.ctx, form, V0 | TOTALS, horizon=case["horizon"], on_device=case["place"] == "device",
                             variant=rsv.RSV_VARIANT_TIME_SCAN if case["flat"] else -1, scen_total=s.total,
                             **{"V0d" if case["out"] == "f64" else "V0": s.V0})
    return {"V0": s.V0, "total": narrow(case, s.total)}


def narrow(case, x):
    """The deflated form is an FP32 form (its bound is 15 x 2^-24): a program that takes it keeps
    its sums as FP32 too."""
    return x.float() if case["form"] == "deflated" else x


# ---- what a pass cannot do without --------------------------------------------
def steps(pol, horizon=0):
    """Projection steps of each policy record."""
    x, y = LIMIT - pol["age1_m"].astype(np.int64), LIMIT - pol["age2_m"].astype(np.int64)
    prod, S = pol["product"], pol["term_m"].astype(np.int64)
    S = np.where(prod == 0, x, np.where((prod == 1) | (prod == 5), np.maximum(x, y), np.where(prod == 4, np.minimum(x, y), S)))
    return np.minimum(S, horizon) if horizon else S


def work(case):
    """Inputs read once and outputs written once; one multiply and one add for each expected cash
    flow and scenario (nested: 40 operations for each month of an inner path, whose cash flows are
    the book's sums)."""
    if case["family"] == "network":
        n, p = case["rows"], 32 * 256 + 3 * 256 * 256 + 256
        return {"bytes": n * 33 * 4 + 8 * p, "flops": 6 * n * p}
    if case["family"] == "mlife":
        pol, n, S = lives(case, 0), case["n_pol"], case["n_scen"]
        left = np.sort(LIMIT - pol["age_m"].astype(np.int64) * (np.arange(4) < pol["m"][:, None]) -
                       LIMIT * (np.arange(4) >= pol["m"][:, None]), axis=1)
        T = np.where(pol["kind"] == 1, pol["term_m"], left[np.arange(n), 4 - pol["k"]])
        return {"bytes": 8 * (n * S + S + S * case["n_steps"]) + 64 * n, "flops": 2 * S * int(T.sum())}
    T = steps(book(case, 0), case.get("horizon", 0))
    if case["family"] == "nested":
        left = sum(max(0, int(T.max()) - 12 * k) for k in range(case["n_nodes"]))
        return {"bytes": 48 * case["n_pol"] + 32 * case["n_outer"] * case["n_nodes"],
                "flops": 42 * case["n_outer"] * case["n_inner"] * left + 2 * int(T.sum())}
    n, S = case["n_pol"], case["n_scen"]
    each = 8 if case["out"] == "f64" else 4
    return {"bytes": each * n * S + 8 * S + 8 * S * case["n_steps"] + 48 * n, "flops": 2 * S * int(T.sum())}


# ---- the same in plain 64 bits -----------------------------------------------
def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def cash_flows(pol, T, cf=None, horizon=0):
    """Expected cash flow of every record in each month, unit amounts, [n, T] (the maturity sum in
    the month it falls at the end of); every table entry past age 120 is death."""
    p_month = dev(np.concatenate([mortality(), np.zeros(LIMIT + 64)]))
    t = torch.arange(T, device="cuda")
    S = dev(steps(pol, horizon))[:, None]
    live = t[None, :] < S
    prod, rho = dev(pol["product"])[:, None], dev(pol["reversion"])[:, None]
    rho = torch.where(prod == 5, 1.0, rho)

    def path(age):   # alive at the start of each month, and through it
        p = p_month[(dev(age).long()[:, None] + t[None, :]).clamp(max=LIMIT + 32)]
        end = torch.cumprod(p, 1)
        start = torch.cat([torch.ones_like(end[:, :1]), end[:, :-1]], 1)
        return start, end

    x0, x1 = path(pol["age1_m"])
    two = (pol["product"] == 1) | (pol["product"] >= 4)
    y0, y1 = path(pol["age2_m"]) if two.any() else (x0, x1)
    flow = torch.where(prod == 0, x1, x0 - x1)
    if two.any():
        flow = torch.where((prod == 1) | (prod == 5), x1 + rho * (y1 - x1 * y1), flow)
        flow = torch.where(prod == 4, x1 * y1, flow)
        flow = torch.where((prod == 6) | (prod == 7), x0 * y0 - x1 * y1, flow)
        flow = torch.where(prod >= 8, (1 - x1) * (1 - y1) - (1 - x0) * (1 - y0), flow)
    if cf is not None:   # payments and death benefits, not the maturity sum
        flow = flow * cf
    flow = torch.where(live, flow, 0.0)
    if two.any() or (pol["product"] == 3).any():
        full = dev(steps(pol))[:, None]
        held = torch.where(prod == 3, x1, torch.where(prod == 7, x1 * y1, x1 + y1 - x1 * y1))
        flow = flow + torch.where(((prod == 3) | (prod == 7) | (prod == 9)) & (t[None, :] == S - 1) & (S == full),
                                  held, 0.0)
    return flow


def multipliers(sch, T):
    t = torch.arange(T, device="cuda")[None, :]
    every, first, since = (dev(sch[k]).long()[:, None] for k in ("every", "first", "since"))
    n = (t + since) // 12
    paid = (t >= first) & ((t - first) % every == 0)
    return torch.where(paid, (1 + dev(sch["escalation"])[:, None]) ** n.double(), 0.0)


def lives_flows(pol, T):
    """Expected cash flows of the m-life records: the number alive at the end of each month is a
    sum of independent indicators."""
    p_month = dev(np.concatenate([mortality(), np.zeros(LIMIT + 64)]))
    n, t = len(pol), torch.arange(T, device="cuda")
    m, k, kind = (dev(pol[c]).long()[:, None] for c in ("m", "k", "kind"))
    alive = [torch.ones((n, T + 1), dtype=torch.float64, device="cuda")]   # Pr[j alive], j = 0 ..
    for i in range(4):
        end = torch.cumprod(p_month[(dev(pol["age_m"][:, i]).long()[:, None] + t[None, :]).clamp(max=LIMIT + 32)], 1)
        p = torch.where(i < m, torch.cat([torch.ones_like(end[:, :1]), end], 1), 0.0)
        pad = [torch.zeros_like(alive[0])] + alive + [torch.zeros_like(alive[0])]
        alive = [pad[j + 1] * (1 - p) + pad[j] * p for j in range(i + 2)]
    at_least = sum(torch.where(k <= j, alive[j], 0.0) for j in range(5))
    dead = sum(torch.where(m - k >= j, alive[j], 0.0) for j in range(5))      # k or more dead
    flow = torch.where(kind == 0, at_least[:, 1:], dead[:, 1:] - dead[:, :-1])
    return torch.where((kind == 0) | (t[None, :] < dev(pol["term_m"]).long()[:, None]), flow, 0.0)


def philox(k, c1, c2, c3, seed):
    M0, M1, W = 0xD2511F53, 0xCD9E8D57, 0xFFFFFFFF
    k0, k1 = seed & W, seed >> 32
    c = [torch.full_like(c1, k), c1, c2, c3]
    for _ in range(10):
        a, b = M0 * c[0], M1 * c[2]
        c = [((b >> 32) & W) ^ c[1] ^ k0, b & W, ((a >> 32) & W) ^ c[3] ^ k1, a & W]
        k0, k1 = (k0 + 0x9E3779B9) & W, (k1 + 0xBB67AE85) & W
    return c


def gaussians(w, h):
    u1, u2 = (w[2 * h].double() + 0.5) / 2 ** 32, (w[2 * h + 1].double() + 0.5) / 2 ** 32
    R, x = torch.sqrt(-2 * torch.log(u1)), 2 * math.pi * u2
    return R * torch.cos(x), R * torch.sin(x)


def exact_nested(case, seed):
    pol, NO, NN, NI = book(case, seed), case["n_outer"], case["n_nodes"], case["n_inner"]
    e, k1, l11, l21, l22 = step_moments()
    S = steps(pol)
    T = int(S.max())
    flow = dev(pol["amount"]) @ cash_flows(pol, T)
    o = torch.arange(NO, device="cuda")
    r, D = torch.full((NO,), R0, dtype=torch.float64, device="cuda"), torch.ones(NO, dtype=torch.float64, device="cuda")
    rates, discounts = [r], [D]
    zero = torch.zeros_like(o)
    for t in range(12 * (NN - 1)):
        w = philox(t >> 1, o, zero, zero + (2 << 24), seed) if t % 2 == 0 else w
        z1, z2 = gaussians(w, t & 1)
        D = D * torch.exp(-(B * DT + (r - B) * k1 + l21 * z1 + l22 * z2))
        r = B + (r - B) * e + l11 * z1
        if (t + 1) % 12 == 0:
            rates.append(r)
            discounts.append(D)
    shape = (NN, NO, NI)
    i = torch.arange(NI, device="cuda").expand(shape).contiguous()
    node = torch.arange(NN, device="cuda")[:, None, None].expand(shape).contiguous()
    key = ((3 << 24) | o)[None, :, None].expand(shape).contiguous()
    r, D = torch.stack(rates)[:, :, None].expand(shape), torch.ones(shape, dtype=torch.float64, device="cuda")
    due = [pol["amount"] * (S == 12 * n) * (pol["product"] == 3) for n in range(NN)]   # matures at the node
    l = np.concatenate([[1.0], np.cumprod(mortality()), np.zeros(LIMIT)])
    due = [float(np.sum(d * l[pol["age1_m"] + 12 * n] / l[pol["age1_m"]])) if d.any() else 0.0 for n, d in enumerate(due)]
    L = D * torch.tensor(due, dtype=torch.float64, device="cuda")[:, None, None]
    flow = torch.cat([flow, torch.zeros(12 * NN, dtype=torch.float64, device="cuda")])
    months = 12 * torch.arange(NN, device="cuda")
    for t in range(T):
        w = philox(t >> 1, i, node, key, seed) if t % 2 == 0 else w
        z1, z2 = gaussians(w, t & 1)
        D = D * torch.exp(-(B * DT + (r - B) * k1 + l21 * z1 + l22 * z2))
        r = B + (r - B) * e + l11 * z1
        L = torch.addcmul(L, D, flow[months + t][:, None, None])
    kth = torch.topk(L, max(1, math.ceil(0.005 * NI - 1e-9)), dim=2).values[:, :, -1]
    return {"L_mean": L.mean(2).T, "L_q995": kth.T, "r_node": torch.stack(rates, 1), "D0": torch.stack(discounts, 1)}


def exact_network(case, seed):
    X, target = network_batch(case, seed)
    p = dev(network_params(seed)).double().requires_grad_()
    a, at = dev(X).double(), 0
    for width in (32, 256, 256, 256):
        W, b = p[at:at + width * 256].view(width, 256), p[at + width * 256:at + width * 256 + 256]
        a, at = torch.nn.functional.gelu(a @ W + b, approximate="tanh"), at + width * 256 + 256
    loss = ((a @ p[at:at + 256] + p[at + 256] - dev(target).double()) ** 2).mean()
    loss.backward()
    return p.grad, float(loss)


def exact(case, seed):
    if case["family"] == "network":
        return exact_network(case, seed)
    if case["family"] == "nested":
        return exact_nested(case, seed)
    D = torch.cumprod(dev(scenarios(case, seed)), 1)
    n, S, T = case["n_pol"], case["n_scen"], case["n_steps"]
    if case["family"] == "mlife":
        pol = lives(case, seed)
        flow = lives_flows(pol, T) * dev(pol["amount"])[:, None]
        return {"V0": flow @ D.T, "total": D @ flow.sum(0)}
    pol = book(case, seed)
    if case["book"] == "annuities":   # one reserve per age
        ages, at = np.unique(pol["age1_m"], return_inverse=True)
        one = np.zeros(len(ages), rsv.POLICY_DTYPE)
        one["age1_m"] = ages
        V, w = cash_flows(one, T, horizon=case["horizon"]) @ D.T, dev(pol["amount"])
        weights = torch.zeros(len(ages), dtype=torch.float64, device="cuda").index_add_(0, dev(at), w)
        return {"V0": V[dev(at)] * w[:, None], "total": weights @ V}
    whole = n * S <= 10_000_000   # the matrix product in 64 bits takes too long beyond
    sch = schedules(case, seed) if case["schedules"] else None
    V, total = [], torch.zeros(T, dtype=torch.float64, device="cuda")
    for lo in range(0, n, 10_000):
        part = pol[lo:lo + 10_000]
        flow = cash_flows(part, T, multipliers(sch[lo:lo + 10_000], T) if case["schedules"] else None, case["horizon"])
        flow = flow * dev(part["amount"])[:, None]
        total += flow.sum(0)
        if whole:
            V.append(flow @ D.T)
    return {"V0": torch.cat(V) if whole else None, "total": D @ total}

