"""Performance cases of the library: the calls its users make, at the sizes they make them.

A case names one kind of call and its sizes.  prepare() builds what a program has in hand before
the call (a context, requests, given paths), run() makes the call once through the public entry
points (api.Context and the stage calls of lsmc), exact() restates the method in 64 bits with
torch alone: Philox4x32-10 counters, the Andersen QE or full-truncation Euler step,
Longstaff-Schwartz regression on the centred basis, central bumps.
"""
import math

import numpy as np
import torch

from paper_2206_03719_gb300 import api, workloads
from paper_2206_03719_gb300 import lsmc as L

PREC = {"fp64": L.LSMC_FP64, "mixed": L.LSMC_MIXED, "df": L.LSMC_DF}
ALL = ",".join(workloads.ALL_GREEKS)


# ---- the cases --------------------------------------------------------------------------------

def listed():
    five = "80,90,100,110,120"
    return [
        # a desk's single quote: 4096 x 32, basis {1,S,S^2}, price + delta, gamma, vega (the
        # repository's small workload); latency and launches
        dict(name="quote_small_fp64", kind="price", precision="fp64", scheme="qe", basis="s2",
             option="put", paths=4096, steps=32, strikes="100", greeks="delta,gamma,vega",
             oos=False, regen=False, store="native"),
        # the repository's headline: five strikes, all five Greeks, 131,072 x 252, basis with v
        dict(name="paper_fp64", kind="price", precision="fp64", scheme="qe", basis="sv2",
             option="put", paths=131072, steps=252, strikes=five, greeks=ALL,
             oos=False, regen=False, store="native"),
        # the same request in the float-pair precision that serves it faster
        dict(name="paper_df", kind="price", precision="df", scheme="qe", basis="sv2",
             option="put", paths=131072, steps=252, strikes=five, greeks=ALL,
             oos=False, regen=False, store="native"),
        # the large single-precision run: 1,048,576 paths
        dict(name="large_mixed", kind="price", precision="mixed", scheme="qe", basis="sv2",
             option="put", paths=1048576, steps=252, strikes=five, greeks=ALL,
             oos=False, regen=False, store="native"),
        # the memory-saving and low-bias options together: full-truncation Euler, ragged path
        # count, 16-bit path store, out-of-sample pricing of calls on a dividend payer
        dict(name="oos_store16_df", kind="price", precision="df", scheme="ft_euler", basis="sv2",
             option="call", paths=50003, steps=126, strikes="95,105", greeks=ALL,
             oos=True, regen=False, store="fp16"),
        # an uneven book revalued in one call (512-contract book's distributions), double precision
        dict(name="book_fp64", kind="book", precision="fp64", contracts=12, paths_hi=262144),
        # the same kind of book, larger, in float pairs
        dict(name="book_df", kind="book", precision="df", contracts=24, paths_hi=262144),
        # a burst of requests through the serving loop
        dict(name="serve_mixed", kind="serve", precision="mixed", contracts=48, paths_hi=262144),
        # path generation alone, for a caller that prices something else on the paths; odd sizes
        dict(name="paths_fp64", kind="paths", precision="fp64", scheme="qe", paths=65537, steps=100),
        # the regression pass alone on paths that the caller has (put, quadratic fit), ragged
        dict(name="backward_fp64", kind="backward", precision="fp64", basis="s2", option="put",
             paths=100001, steps=50, strike=105.0),
        # the paper's multi-asset path reduction, its "small" size
        dict(name="stac_small_fp64", kind="multi", precision="fp64", scheme="qe", assets=10,
             steps=126, paths=25000, corr=0.0),
        # lower and dual upper bounds of an American put
        dict(name="bounds_df", kind="bounds", precision="df", scheme="qe", basis="sv2",
             paths=32768, steps=100, strikes="90,100,110", outer=256, inner=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["price"] * 4 + ["book", "book", "serve", "paths", "backward", "multi",
                                       "bounds"])
    prec = rng.choice(["fp64", "fp64", "df", "df", "mixed"])
    scheme = rng.choice(["qe", "qe", "qe", "ft_euler"])
    basis = rng.choice(["s2", "sv2"])
    steps = _log_int(rng, 12, 500)
    if kind == "price":
        # at most about the headline's path steps x strikes
        n_strikes = rng.choice([1, 1, 2, 3, 5])
        most = {"fp64": 1.4e8, "df": 1.7e8, "mixed": 1.0e9}[prec] / (steps * n_strikes)
        paths = _log_int(rng, 2000, max(4000, min(most, 1000000)))
        strikes = sorted(rng.sample([80.0, 85.0, 90.0, 95.0, 100.0, 105.0, 110.0, 115.0, 120.0],
                                    n_strikes))
        oos = rng.random() < 0.2
        return dict(kind=kind, precision=prec, scheme=scheme, basis=basis,
                    option=rng.choice(["put", "put", "call"]), paths=paths, steps=steps,
                    strikes=",".join("%g" % k for k in strikes),
                    greeks=rng.choice([ALL, ALL, "delta,gamma,vega", "delta", ""]), oos=oos,
                    regen=(not oos and rng.random() < 0.15),
                    store=rng.choice(["native"] * 5 + ["fp16", "bf16"]))
    if kind == "book":
        n = {"fp64": 8, "df": 24, "mixed": 48}[prec]
        return dict(kind=kind, precision=prec, contracts=rng.randint(2, n),
                    paths_hi=_log_int(rng, 8192, 262144))
    if kind == "serve":
        n = {"fp64": 8, "df": 24, "mixed": 48}[prec]
        return dict(kind=kind, precision=prec, contracts=rng.randint(2, n),
                    paths_hi=_log_int(rng, 8192, 262144))
    if kind == "paths":
        return dict(kind=kind, precision=prec, scheme=scheme, steps=steps,
                    paths=_log_int(rng, 1000, 3.0e7 / steps))
    if kind == "backward":
        return dict(kind=kind, precision=prec, basis=basis, option=rng.choice(["put", "call"]),
                    paths=_log_int(rng, 1000, 3.0e7 / steps), steps=steps,
                    strike=rng.choice([90.0, 97.5, 100.0, 105.0, 112.0]))
    if kind == "multi":
        assets = rng.randint(2, 30)
        return dict(kind=kind, precision=prec, scheme=scheme, assets=assets, steps=steps,
                    paths=_log_int(rng, 1000, min(50000, 1.2e8 / (steps * assets))),
                    corr=rng.choice([0.0, 0.0, 0.3]))
    steps = _log_int(rng, 12, 126)
    strikes = sorted(rng.sample([90.0, 95.0, 100.0, 105.0, 110.0], rng.choice([1, 2, 3])))
    cells = {"fp64": 4e7, "df": 2e8, "mixed": 4e8}[prec] / (steps * steps / 2)
    inner = _log_int(rng, 32, 256)
    return dict(kind="bounds", precision=prec, scheme=scheme, basis=basis,
                paths=_log_int(rng, 4096, 65536), steps=steps,
                strikes=",".join("%g" % k for k in strikes),
                outer=_log_int(rng, 32, max(33, min(1024, cells / inner))), inner=inner)


# ---- what a program has in hand ---------------------------------------------------------------

def _model(rng, option="put"):
    """The headline workload's model with the day's market data: spot, variance, rate."""
    m = dict(workloads.HESTON_BASE)
    m["S0"] = float(np.round(rng.uniform(99.0, 101.0), 2))
    m["v0"] = float(np.round(rng.uniform(0.035, 0.045), 4))
    m["r"] = float(np.round(rng.uniform(0.015, 0.03), 4))
    if option == "call":
        m["q"] = 0.03  # an American call is worth exercising early on a dividend payer
    return m


def _request(case, seed):
    rng = np.random.default_rng([seed, 1])
    option = case.get("option", "put")
    return workloads.Workload(
        name=case["kind"], model=_model(rng, option),
        strikes=[float(k) for k in case["strikes"].split(",")], T=1.0, n_paths=case["paths"],
        n_steps=case["steps"], option=option, basis=case["basis"], scheme=case["scheme"],
        precision=case["precision"],
        greeks=tuple(g for g in case.get("greeks", "").split(",") if g),
        rel_dS=0.01, rel_dS_gamma=0.02, seed=int(rng.integers(1, 2**62)),
        stream=int(rng.integers(0, 2**16)), regenerate=case.get("regen", False),
        out_of_sample=case.get("oos", False), store=case.get("store", "native"))


def _book(case, seed):
    """Contracts of the uneven book: their sizes belong to the case, so that every seed is the
    same amount of work; models, maturities, strikes and random streams to the seed."""
    sizes = workloads.book(case["contracts"], seed=220603719 + case["contracts"],
                           paths_hi=case["paths_hi"], precision=case["precision"])
    other = workloads.book(case["contracts"], seed=int(seed) + 17, precision=case["precision"])
    key = int(np.random.default_rng([seed, 2]).integers(1, 2**62))
    return [o.replace(n_paths=s.n_paths, n_steps=s.n_steps, seed=key)
            for o, s in zip(other, sizes)]


def _heston(m):
    return L.lsmc_heston(**m)


def _path_tensor(case):
    shape = (case["steps"] + 1, case["paths"])
    if case["precision"] == "df":
        return torch.empty(shape + (2,), dtype=torch.float32, device="cuda")
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    return torch.empty(shape, dtype=dt, device="cuda")


def prepare(case, seed):
    L.load()
    kind = case["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind in ("price", "bounds"):
        # device memory from PyTorch's allocator, as the README's example has it
        return dict(case=case, ctx=api.Context(torch_allocator=True), wl=_request(case, seed))
    if kind == "book":
        return dict(case=case, ctx=api.Context(torch_allocator=True), wls=_book(case, seed))
    if kind == "serve":
        ctx = api.Context(workspace_bytes=16 << 30, max_inflight=4)
        return dict(case=case, ctx=ctx, wls=_book(case, seed))
    rng = np.random.default_rng([seed, 3])
    key, strm = int(rng.integers(1, 2**62)), int(rng.integers(0, 2**16))
    if kind == "multi":
        models = workloads.stac_models(case["assets"], seed=int(seed))
        M = _path_tensor(case)
        return dict(case=case, models=[_heston(m) for m in models], M=M, key=key, stream_id=strm,
                    stream=stream)
    model = _model(rng, case.get("option", "put"))
    S, V = _path_tensor(case), _path_tensor(case)
    st = dict(case=case, model=_heston(model), S=S, V=V, key=key, stream_id=strm, stream=stream)
    if kind == "backward":
        # paths that came from elsewhere
        P, N = case["paths"], case["steps"]
        S64 = torch.full((N + 1, P), model["S0"], dtype=torch.float64, device="cuda")
        V64 = torch.full((N + 1, P), model["v0"], dtype=torch.float64, device="cuda")
        sim = _Sim([model], [1.0], N, "qe", P)
        for n in range(N):
            sim.step(*_draws(P, n, strm, 0, key, False))
            S64[n + 1], V64[n + 1] = model["S0"] * torch.exp(sim.x[0]), sim.v[0]
        for src, dst in ((S64, S), (V64, V)):
            if case["precision"] == "df":
                hi = src.float()
                dst[..., 0], dst[..., 1] = hi, (src - hi.double()).float()
            else:
                dst.copy_(src)
        st["contract"] = L.lsmc_contract(
            L.LSMC_PUT if case["option"] == "put" else L.LSMC_CALL, L.LSMC_AMERICAN,
            case["strike"], 1.0)
        st["out"] = torch.zeros(5, dtype=torch.float64, device="cuda")
        st["ns"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    return st


# ---- one pass -----------------------------------------------------------------------------------

# (n_near_ties, the number of decisions within rounding reach of their threshold, is a diagnostic
# of rounding itself and not a price)
_COUNTS = ("n_singular_solves", "n_revaluations", "status")


def _columns(rows, greeks):
    keys = ("price", "price_se", "european_price") + tuple(greeks)
    out = {k: np.array([r[k] for r in rows]) for k in keys}
    out.update({k: np.array([r[k] for r in rows], dtype=np.int64) for k in _COUNTS})
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "price":
        return _columns(state["ctx"].price(state["wl"]), state["wl"].greeks)
    if kind == "book":
        return _columns(state["ctx"].price_book(state["wls"]), workloads.ALL_GREEKS)
    if kind == "serve":
        ctx = state["ctx"]
        tickets = [ctx.submit(w) for w in state["wls"]]
        rows = []
        for w, t in zip(state["wls"], tickets):
            status, res = ctx.wait(t, len(w.strikes))
            if status != L.LSMC_OK:
                raise L.LsmcError(status, "serving")
            rows += [r.as_dict() for r in res]
        return _columns(rows, workloads.ALL_GREEKS)
    if kind == "bounds":
        rows = state["ctx"].price_bounds(state["wl"], case["outer"], case["inner"])
        return {k: np.array([r[k] for r in rows])
                for k in ("lower", "lower_se", "upper", "upper_se", "martingale_end",
                          "martingale_end_se")}
    scheme = L.LSMC_SCHEME_FT_EULER if case.get("scheme") == "ft_euler" else L.LSMC_SCHEME_QE
    prec = PREC[case["precision"]]
    if kind == "paths":
        L.lsmc_paths(state["model"], 1.0, scheme, prec, case["paths"], case["steps"],
                     state["key"], state["stream_id"], state["S"].data_ptr(),
                     state["V"].data_ptr(), state["stream"])
        return {"S": state["S"], "V": state["V"]}
    if kind == "multi":
        L.lsmc_multi_asset_max(state["models"], case["steps"] / 252.0, scheme, prec, case["corr"],
                               case["paths"], case["steps"], state["key"], state["stream_id"],
                               state["M"].data_ptr(), state["stream"])
        return {"M": state["M"]}
    basis = L.LSMC_BASIS_SV2 if case["basis"] == "sv2" else L.LSMC_BASIS_S2
    L.lsmc_backward(state["S"].data_ptr(), state["V"].data_ptr(), case["paths"], case["steps"],
                    prec, state["model"], state["contract"], basis, state["out"].data_ptr(), None,
                    state["ns"].data_ptr(), state["stream"])
    return {"price_se_european_continuation": state["out"][:4], "n_singular": state["ns"]}


# ---- what a pass cannot do without ----------------------------------------------------------------

# flops of the method, a fused multiply-add as 2, a division, square root, exponential, logarithm
# or normal quantile as one: a draw of (path, date); a step of one simulation; a regression path
# step (the product S, the payoff, the comparison, and for half of the paths the moment sums and
# the exercise test).  Bytes: what is given and what is returned.
_STEP = 32.0


def _price_work(P, N, n_strikes, n_greek_sc, groups, basis, style_oos=False):
    reg = 3.0 + 0.5 * (55.0 if basis == "sv2" else 24.0)
    fwd = P * N * (2.0 + groups * _STEP)
    bwd = P * N * n_strikes * n_greek_sc * reg
    if style_oos:
        fwd *= 2.0
        bwd += P * N * n_strikes * n_greek_sc * 10.0
    return fwd + bwd


def work(case):
    kind, prec = case["kind"], case["precision"]
    size = 4 if prec == "mixed" else 8
    if kind in ("price", "bounds"):
        P, N = case["paths"], case["steps"]
        strikes = len(case["strikes"].split(","))
        g = set(x for x in case.get("greeks", "").split(",") if x)
        groups = 1 + 2 * ("vega" in g) + 2 * ("theta" in g)
        sc = 1 + 2 * ("delta" in g) + 2 * ("gamma" in g) + 2 * len(g & {"vega", "rho", "theta"})
        fl = _price_work(P, N, strikes, sc, groups, case["basis"],
                         case.get("oos", False) or kind == "bounds")
        if kind == "bounds":
            fl += case["outer"] * case["inner"] * N * (N + 1) / 2.0 * (2.0 + _STEP + 4.0 * strikes)
        return {"bytes": 200.0 + 96.0 * strikes, "flops": fl}
    if kind in ("book", "serve"):
        fl = sum(_price_work(w.n_paths, w.n_steps, 1, 11, 5, "s2") for w in _book(case, 0))
        return {"bytes": 300.0 * case["contracts"], "flops": fl}
    cells = float(case["paths"]) * (case["steps"] + 1)
    if kind == "paths":
        return {"bytes": 2.0 * cells * size, "flops": cells * (2.0 + _STEP)}
    if kind == "multi":
        return {"bytes": cells * size, "flops": cells * case["assets"] * (4.0 + _STEP)}
    rows = 2.0 if case["basis"] == "sv2" else 1.0
    return {"bytes": rows * cells * size,
            "flops": cells * (3.0 + 0.5 * (55.0 if case["basis"] == "sv2" else 24.0))}


# ---- the method in 64 bits ------------------------------------------------------------------------

_DEV = "cuda" if torch.cuda.is_available() else "cpu"
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 on int64 tensors (or ints) of counter words; four int64 words."""
    k0, k1 = key & _M32, (key >> 32) & _M32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32,
                          ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32)
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _quantile(u, omu):
    z = torch.special.ndtri(torch.minimum(u, omu))
    return torch.where(u < omu, z, -z)


def _grid(hi, lo, single):
    if single:
        u = ((hi >> 9).double() + 0.5) * 2.0**-23
    else:
        u = (((hi << 20) | (lo >> 12)).double() + 0.5) * 2.0**-52
    return u, 1.0 - u


def _draws(P, n, stream, word3, key, single):
    p = torch.arange(P, dtype=torch.int64, device=_DEV)
    full = lambda v: torch.full_like(p, v)  # noqa: E731
    w = _philox(p, full(n), full(stream), full(word3), key)
    u, omu = _grid(w[0], w[1], single)
    uX, omuX = _grid(w[2], w[3], single)
    return omu, _quantile(u, omu), _quantile(uX, omuX)


class _Sim:
    """Paths of simulations that share their draws: rows of x = ln(S / S0) and v, one simulation
    per entry of models / Ts."""

    def __init__(self, models, Ts, N, scheme, P):
        col = lambda f: torch.tensor([[f(m, T / N)] for m, T in zip(models, Ts)],  # noqa: E731
                                     dtype=torch.float64, device=_DEV)
        self.qe = scheme == "qe"
        self.x = torch.zeros((len(models), P), dtype=torch.float64, device=_DEV)
        self.v = col(lambda m, dt: m["v0"]).expand(-1, P).clone()
        self.theta, self.xi = col(lambda m, dt: m["theta"]), col(lambda m, dt: m["xi"])
        self.rho, self.dt = col(lambda m, dt: m["rho"]), col(lambda m, dt: dt)
        self.kdt = col(lambda m, dt: m["kappa"] * dt)
        self.mu = col(lambda m, dt: (m["r"] - m["q"]) * dt)
        if self.qe:
            E = lambda m, dt: math.exp(-m["kappa"] * dt)  # noqa: E731
            omE = lambda m, dt: -math.expm1(-m["kappa"] * dt)  # noqa: E731
            self.mA, self.mB = col(lambda m, dt: m["theta"] * omE(m, dt)), col(E)
            self.sB = col(lambda m, dt: m["xi"]**2 * E(m, dt) * omE(m, dt) / m["kappa"])
            self.sA = col(lambda m, dt: m["theta"] * m["xi"]**2 * omE(m, dt)**2 / (2 * m["kappa"]))
            h = lambda m, dt: 0.5 * dt * (m["kappa"] * m["rho"] / m["xi"] - 0.5)  # noqa: E731
            self.K0 = col(lambda m, dt: -m["rho"] * m["kappa"] * m["theta"] * dt / m["xi"])
            self.K1 = col(lambda m, dt: h(m, dt) - m["rho"] / m["xi"])
            self.K2 = col(lambda m, dt: h(m, dt) + m["rho"] / m["xi"])
            self.K3 = col(lambda m, dt: 0.5 * dt * (1 - m["rho"]**2))

    def step(self, omu, zV, zX):
        x, v = self.x, self.v
        if self.qe:
            m, s2 = self.mA + self.mB * v, self.sA + self.sB * v
            psi = s2 / (m * m)
            inv = 2.0 / psi
            b2 = inv - 1.0 + torch.sqrt((inv * (inv - 1.0)).clamp(min=0.0))
            vq = m / (1.0 + b2) * (torch.sqrt(b2.clamp(min=0.0)) + zV)**2
            omp = 2.0 / (psi + 1.0)  # 1 - p
            ve = torch.where(omu >= omp, torch.zeros_like(v), m / omp * torch.log(omp / omu))
            v1 = torch.where(psi <= 1.5, vq, ve)
            self.x = x + self.mu + self.K0 + self.K1 * v + self.K2 * v1 + \
                torch.sqrt(self.K3 * (v + v1)) * zX
            self.v = v1
            return
        vp = v.clamp(min=0.0)
        sq = torch.sqrt(vp * self.dt)
        self.v = v + self.kdt * (self.theta - vp) + self.xi * sq * zV
        self.x = x + (self.mu - 0.5 * vp * self.dt) + \
            sq * (self.rho * zV + torch.sqrt(1 - self.rho**2) * zX)

    def variance(self):
        return self.v if self.qe else self.v.clamp(min=0.0)


def _round16(a, store):
    """a rounded to binary16 / bfloat16, nearest even, exactly once."""
    if store == "native":
        return a
    m, e = torch.frexp(a)
    if store == "fp16":
        bits = 11 - (-13 - e).clamp(min=0)  # fewer in the subnormal range
    else:
        bits = torch.full_like(e, 8)
    return torch.ldexp(torch.round(torch.ldexp(m, bits)), e - bits)


def _solve(A, R, count):
    """Batched normal equations by Cholesky; (coefficients, solved): unsolved below the basis's
    count of paths or where a pivot is not above 1e-13 of the largest diagonal entry."""
    B = A.shape[-1]
    tol = 1e-13 * torch.diagonal(A, dim1=-2, dim2=-1).amax(-1)
    ok = count >= B
    Lc = torch.zeros_like(A)
    for j in range(B):
        d = A[:, j, j] - (Lc[:, j, :j]**2).sum(-1)
        ok = ok & (d > tol)
        Lc[:, j, j] = torch.sqrt(torch.where(ok, d, torch.ones_like(d)))
        for i in range(j + 1, B):
            Lc[:, i, j] = (A[:, i, j] - (Lc[:, i, :j] * Lc[:, j, :j]).sum(-1)) / Lc[:, j, j]
    beta = torch.cholesky_solve(R[..., None], Lc)[..., 0]
    return torch.where(ok[:, None], beta, torch.zeros_like(beta)), ok


def _basis(S, V, K, theta, sv2):
    x = S / K - 1.0
    one = torch.ones_like(x)
    if not sv2:
        return torch.stack([one, x, x * x], 1)
    w = V / theta - 1.0
    return torch.stack([one, x, x * x, w, x * w, w * w], 1)


def _lsmc(row, N, P, K, r, dt, theta, put, sv2, h0, price_row=None):
    """Longstaff-Schwartz of instances (rows of tensors): row(n) -> (S, V) of date n, each
    (instances, P).  price_row: independent paths that the policy is applied to.  Columns: price,
    standard error, European price, continuation value; count of unsolved dates."""
    pay = (lambda S: (K - S).clamp(min=0.0)) if put else (lambda S: (S - K).clamp(min=0.0))
    disc = torch.exp(-r * dt)
    S, _ = row(N)
    Y = pay(S)
    euro = (Y * torch.exp(-r * dt * N)).mean(1)
    unsolved = torch.zeros(K.shape[0], dtype=torch.int64, device=_DEV)
    betas = {}
    for n in range(N - 1, 0, -1):
        Y = Y * disc
        S, V = row(n)
        h = pay(S)
        itm = h > 0.0
        X = _basis(S, V, K, theta, sv2)
        Xm = X * itm[:, None, :]
        A = Xm @ Xm.transpose(1, 2)
        R = (Xm @ Y[..., None])[..., 0]
        beta, ok = _solve(A, R, itm.sum(1))
        unsolved += ~ok
        cont = (beta[:, None, :] @ X)[:, 0]
        go = itm & ok[:, None] & (h > cont)
        Y = torch.where(go, h, Y)
        betas[n] = (beta, ok)
        del X, Xm
    Z = Y * disc
    if price_row is not None:
        S, _ = price_row(N)
        Z = pay(S) * torch.exp(-r * dt * N)
        euro = Z.mean(1)
        for n in range(N - 1, 0, -1):  # the first exercise date wins: later ones overwritten
            S, V = price_row(n)
            h = pay(S)
            beta, ok = betas[n]
            cont = (beta[:, None, :] @ _basis(S, V, K, theta, sv2))[:, 0]
            Z = torch.where((h > 0.0) & ok[:, None] & (h > cont), h * torch.exp(-r * dt * n), Z)
    mean = Z.mean(1)
    se = torch.sqrt(((Z - mean[:, None])**2).sum(1) / max(1, P - 1) / P)
    return torch.stack([torch.maximum(h0, mean), se, euro, mean], 1), unsolved


def _scenarios(wl):
    """(kind, model, T, simulation): bumps of S0 and r reuse the base simulation's x and v (x is
    ln(S/S0), and a rate bump moves it by n dr dt)."""
    m, g = wl.model, set(wl.greeks)
    sc = [("base", m, wl.T, 0)]
    sims = [(m, wl.T)]

    def own(kind, mm, T):
        sims.append((mm, T))
        sc.append((kind, mm, T, len(sims) - 1))

    if "delta" in g:
        sc += [("s+", dict(m, S0=m["S0"] * (1 + wl.rel_dS)), wl.T, 0),
               ("s-", dict(m, S0=m["S0"] * (1 - wl.rel_dS)), wl.T, 0)]
    if "gamma" in g:
        sc += [("g+", dict(m, S0=m["S0"] * (1 + wl.rel_dS_gamma)), wl.T, 0),
               ("g-", dict(m, S0=m["S0"] * (1 - wl.rel_dS_gamma)), wl.T, 0)]
    if "vega" in g:
        own("v+", dict(m, v0=m["v0"] * (1 + wl.rel_dv0)), wl.T)
        own("v-", dict(m, v0=m["v0"] * (1 - wl.rel_dv0)), wl.T)
    if "rho" in g:
        sc += [("r+", dict(m, r=m["r"] + wl.abs_dr), wl.T, 0),
               ("r-", dict(m, r=m["r"] - wl.abs_dr), wl.T, 0)]
    if "theta" in g:
        own("t-", m, wl.T - wl.abs_dT)
        own("t+", m, wl.T + wl.abs_dT)
    return sc, sims


def _simulate(wl, sims, stream):
    P, N = wl.n_paths, wl.n_steps
    sim = _Sim([m for m, _ in sims], [T for _, T in sims], N, wl.scheme, P)
    E = torch.empty((N + 1, len(sims), P), dtype=torch.float64, device=_DEV)
    V = torch.empty_like(E)
    for n in range(N):
        sim.step(*_draws(P, n, stream, 0, wl.seed, wl.precision == "mixed"))
        E[n + 1] = _round16(torch.exp(sim.x), wl.store)
        V[n + 1] = _round16(sim.variance(), wl.store)
    return E, V


def _price_exact(wl):
    sc, sims = _scenarios(wl)
    N, P, m0 = wl.n_steps, wl.n_paths, wl.model
    E, V = _simulate(wl, sims, wl.stream)
    if wl.out_of_sample:
        E2, V2 = _simulate(wl, sims, wl.stream ^ 0x80000000)
    col = lambda f: torch.tensor([[f(*s)] for s in sc], dtype=torch.float64, device=_DEV)  # noqa: E731
    dt = col(lambda k, m, T, g: T / N)
    r, theta = col(lambda k, m, T, g: m["r"]), col(lambda k, m, T, g: m["theta"])
    S0 = col(lambda k, m, T, g: m["S0"])
    dr = r - m0["r"]
    g = torch.tensor([s[3] for s in sc], device=_DEV)
    put = wl.option == "put"

    def rows(E, V):
        return lambda n: (E[n][g] * S0 * torch.exp(dr * dt * n), V[n][g])

    table = []
    for K in wl.strikes:
        Kt = torch.full_like(S0, K)
        h0 = (Kt - S0 if put else S0 - Kt).clamp(min=0.0)[:, 0]
        cols, bad = _lsmc(rows(E, V), N, P, Kt, r, dt, theta, put, wl.basis == "sv2", h0,
                          rows(E2, V2) if wl.out_of_sample else None)
        cols = cols.cpu().numpy()
        p = {s[0]: cols[i, 0] for i, s in enumerate(sc)}
        row = dict(price=p["base"], price_se=cols[0, 1], european_price=cols[0, 2],
                   n_singular_solves=int(bad.sum()), n_revaluations=len(sc),
                   status=int(bad.sum() > 0))
        if "s+" in p:
            row["delta"] = (p["s+"] - p["s-"]) / (2 * wl.rel_dS * m0["S0"])
        if "g+" in p:
            row["gamma"] = (p["g+"] - 2 * p["base"] + p["g-"]) / (wl.rel_dS_gamma * m0["S0"])**2
        if "v+" in p:
            row["vega"] = (p["v+"] - p["v-"]) / (2 * wl.rel_dv0 * m0["v0"])
        if "r+" in p:
            row["rho"] = (p["r+"] - p["r-"]) / (2 * wl.abs_dr)
        if "t+" in p:
            row["theta"] = (p["t-"] - p["t+"]) / (2 * wl.abs_dT)
        table.append(row)
    return table


def exact(case, seed):
    kind, prec = case["kind"], case["precision"]
    if kind in ("price", "book", "serve"):
        wls = [_request(case, seed)] if kind == "price" else _book(case, seed)
        # past about a minute's worth of path steps x regressions: no value
        if sum(w.n_paths * w.n_steps * len(w.strikes) for w in wls) > 6e8:
            return None
        out = _columns([r for w in wls for r in _price_exact(w)], wls[0].greeks)
        # single-precision and 16-bit paths move decisions next to the boundary: their Greeks,
        # differences of such prices, have no value to be held to
        if prec == "mixed" or wls[0].store != "native":
            out.update({k: None for k in wls[0].greeks})
        out.update({k: None for k in _COUNTS})
        return out
    if kind == "bounds":
        wl = _request(dict(case, oos=True), seed).replace(greeks=())
        rows = _price_exact(wl)
        return {"lower": np.array([r["price"] for r in rows]),
                "lower_se": np.array([r["price_se"] for r in rows]), "upper": None,
                "upper_se": None, "martingale_end": None, "martingale_end_se": None}
    rng = np.random.default_rng([seed, 3])
    key, strm = int(rng.integers(1, 2**62)), int(rng.integers(0, 2**16))
    P, N, single = case["paths"], case["steps"], prec == "mixed"
    pairs = lambda a: a if prec != "df" else torch.stack(  # noqa: E731
        [a.float().double(), a - a.float().double()], -1)
    if kind == "multi":
        models, T = workloads.stac_models(case["assets"], seed=int(seed)), case["steps"] / 252.0
        M = torch.full((N + 1, P), max(m["S0"] for m in models), dtype=torch.float64, device=_DEV)
        M[1:] = 0.0
        for a, m in enumerate(models):
            sim = _Sim([m], [T], N, case["scheme"], P)
            for n in range(N):
                omu, zV, zX = _draws(P, n, strm, a, key, single)
                if case["corr"] > 0.0:
                    zc = _draws(P, n, strm, 0xFFFFFFFF, key, single)[2]
                    zX = math.sqrt(case["corr"]) * zc + math.sqrt(1 - case["corr"]) * zX
                sim.step(omu, zV, zX)
                M[n + 1] = torch.maximum(M[n + 1], m["S0"] * torch.exp(sim.x[0]))
        return {"M": pairs(M)}
    model = _model(rng, case.get("option", "put"))
    if kind == "paths":
        sim = _Sim([model], [1.0], N, case["scheme"], P)
        S = torch.full((N + 1, P), model["S0"], dtype=torch.float64, device=_DEV)
        V = torch.full((N + 1, P), model["v0"], dtype=torch.float64, device=_DEV)
        for n in range(N):
            sim.step(*_draws(P, n, strm, 0, key, single))
            S[n + 1], V[n + 1] = model["S0"] * torch.exp(sim.x[0]), sim.variance()[0]
        return {"S": pairs(S), "V": pairs(V)}
    st = prepare(case, seed)  # the given paths
    wide = lambda t: t.double().sum(-1) if prec == "df" else t.double()  # noqa: E731
    S, V = wide(st["S"]).to(_DEV), wide(st["V"]).to(_DEV)
    one = lambda v: torch.tensor([[v]], dtype=torch.float64, device=_DEV)  # noqa: E731
    put = case["option"] == "put"
    h0 = max(0.0, case["strike"] - model["S0"] if put else model["S0"] - case["strike"])
    cols, bad = _lsmc(lambda n: (S[n][None], V[n][None]), N, P, one(case["strike"]),
                      one(model["r"]), one(1.0 / N), one(model["theta"]), put,
                      case["basis"] == "sv2", one(h0)[0])
    return {"price_se_european_continuation": cols[0], "n_singular": None}
