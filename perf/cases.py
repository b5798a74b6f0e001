"""Work that users of the payoff-expression engine have it do, through its
public Python entry points: quoting one contract (from a single-date call to
a daily barrier), per-path payoffs, sensitivities, a portfolio, the network
of the learned control variate, and control-variate pricing.

A case names a contract template and its sizes; the seed gives the market
(spots, volatilities, correlation, rate) and the path seed, so one contract
is priced on changing markets as a pricing service does.  One context per
setting (interpreting, or with run-time specialised kernels) lives as long
as the program.  ``exact`` restates the method in 64 bits with torch.
"""
import math
import random

import numpy as np
import torch

import paper_2108_03076_gb300 as pc

# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------


def _price(name, contract, d, n, paths, jit, out="price"):
    return dict(name=name, kind="price", contract=contract, d=d, n=n, paths=paths, jit=jit, out=out)


def listed():
    return [
        # a quote of a vanilla call, instrument loaded for the request and
        # dropped after it: the smallest call, latency counts
        _price("quote_european", "european", 1, 1, 1 << 16, False, "quote"),
        # the worst-of autocallable note, compiled once and repriced
        _price("autocall_compiled", "autocall", 3, 5, 1 << 20, True),
        # the same note under the context's default (interpreting) setting,
        # every path's payoff kept (a risk report), a ragged path count
        _price("autocall_paths", "autocall", 3, 5, 300007, False, "paths"),
        # the daily down-and-out barrier: the headline run, the largest
        _price("barrier_compiled", "barrier", 3, 365, 1 << 22, True, "sums"),
        # a one-year business-daily barrier on two assets, never compiled
        _price("barrier_interpreted", "barrier", 2, 252, 100003, False, "sums"),
        # an average summed newest fixing first: the whole path is looked
        # back at, the window of dates does not fit on chip
        _price("asian_newest_first", "asian_newest", 2, 300, 1 << 18, False, "sums"),
        # price, delta and vega of a basket call, compiled
        dict(name="greeks_basket", kind="greeks", contract="basket", d=3, n=5, paths=1 << 20, jit=True, mode="adjoint"),
        # the same of the daily barrier on four underlyings
        dict(name="greeks_barrier", kind="greeks", contract="barrier", d=4, n=365, paths=1 << 17, jit=True, mode="adjoint"),
        # a book of templated contracts, planned once and replayed as the market data stands
        dict(name="portfolio", kind="portfolio", contracts=192, book=4, jit=True, oneshot=False),
        # gradients of the hedge network on a full training set
        dict(name="mlp_gradients", kind="mlp", op="gradients", rows=65536, width=256),
        # a short refit of the network: Adam steps on minibatches
        dict(name="mlp_train", kind="mlp", op="train", rows=8192, width=256, batch=1024, steps=50),
        # the autocallable by its learned control variate: hedge tables from
        # the network, then the paths
        dict(name="control_variate", kind="cv", grid=12, paths=1 << 20, jit=True, gamma=True),
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(["price", "greeks", "portfolio", "mlp", "cv"], [10, 4, 2, 4, 2])[0]
    if kind == "price":
        c = rng.choice(["european", "basket", "autocall", "autocall", "barrier", "barrier", "barrier", "asian", "asian_newest"])
        d = {"european": 1, "asian": 1, "asian_newest": 2}.get(c) or rng.randint(1, 4)
        n = {"european": 1, "basket": rng.randint(1, 12), "autocall": rng.randint(2, 12), "barrier": _log_int(rng, 20, 365),
             "asian": _log_int(rng, 10, 200), "asian_newest": _log_int(rng, 20, 300)}[c]
        # long averages are past the specialising limit or slow to specialise
        jit = rng.random() < 0.5 and not (c.startswith("asian") and n > 40)
        most = min(1 << 22, (1 << 22) * 365 * 3 // (n * d * (1 if jit else 6)))
        return dict(kind=kind, contract=c, d=d, n=n, paths=_log_int(rng, 1 << 11, most), jit=jit,
                    out=rng.choice(["price", "price", "sums", "paths", "quote"]))
    if kind == "greeks":
        c, d = rng.choice(["basket", "barrier"]), rng.randint(1, 4)
        n = rng.randint(1, 12) if c == "basket" else _log_int(rng, 20, 365)
        mode = rng.choice(["adjoint", "adjoint", "tangent"])
        most = min(1 << 20, (1 << 18) * 365 * 4 // (n * d * (8 if mode == "tangent" else 2)))
        return dict(kind=kind, contract=c, d=d, n=n, paths=_log_int(rng, 1 << 11, most), jit=rng.random() < 0.5, mode=mode)
    if kind == "portfolio":
        jit = rng.random() < 0.4
        return dict(kind=kind, contracts=_log_int(rng, 12, 64 if jit else 128), book=rng.randint(0, 1 << 20), jit=jit,
                    oneshot=rng.random() < 0.5)
    if kind == "mlp":
        op = rng.choice(["forward", "gradients", "train"])
        if op == "train":
            return dict(kind=kind, op=op, rows=_log_int(rng, 2048, 32768), width=rng.choice([64, 128, 256]),
                        batch=_log_int(rng, 256, 4096), steps=rng.randint(10, 40))
        return dict(kind=kind, op=op, rows=_log_int(rng, 500, 65536), width=rng.choice([64, 128, 256, 384]))
    return dict(kind=kind, grid=rng.randint(5, 16), paths=_log_int(rng, 1 << 13, 1 << 21), jit=rng.random() < 0.6,
                gamma=rng.random() < 0.7)


# ---------------------------------------------------------------------------
# Contracts (payoff intermediate language) and markets
# ---------------------------------------------------------------------------


def _chain(op, xs):
    out = xs[0]
    for x in xs[1:]:
        out = f"({op} {out} {x})"
    return out


def _worst(d, t):
    return _chain("min", [f"(div (model {i} {t}) 1.0)" for i in range(d)])


def _basket(d):
    return f"(div {_chain('add', [f'(model {i} $0)' for i in range(d)])} {float(d)})"


def contract_text(contract, d, n, strike=1.0, barrier=0.7, spreads=13):
    """(program text, template parameters)."""
    if contract == "european":  # struck at 100, as its market's spot
        return f"(mult (max (sub (model 0 $0) {100.0 * strike}) 0.0) (payoff $0 0 1))", [n]
    if contract == "basket":
        return f"(mult (max (sub {_basket(d)} {strike}) 0.0) (payoff $0 0 1))", [n]
    if contract == "digital":
        return f"(mult (if (lt {strike} {_basket(d)}) 1.0 0.0) (payoff $0 0 1))", [n]
    if contract == "call_spread":
        return (f"(mult (sub (max (sub {_basket(d)} {strike}) 0.0) (max (sub {_basket(d)} {strike + 0.2}) 0.0)) "
                f"(payoff $0 0 1))"), [n]
    if contract == "autocall":
        kis = [f"(le {_worst(d, n - j)} 0.6)" for j in range(n)]
        ki = kis[-1]
        for x in reversed(kis[:-1]):
            ki = f"(or {x} {ki})"
        body = f"(mult (if {ki} {_worst(d, n)} 1.0) (payoff {n} 0 1))"
        for k in range(n, 0, -1):
            body = f"(loopif (le 1.0 {_worst(d, k)}) (mult {1.0 + 0.05 * k!r} (payoff {k} 0 1)) {body} 0)"
        return body, []
    if contract == "barrier":  # knocked out at any date, else a ladder of call spreads on the worst-of
        hit = _chain("or", [f"(le (div (model {i} 0) 1.0) {barrier})" for i in range(d)])
        a = [k * 1.95 / spreads for k in range(spreads + 1)]
        W = _worst(d, 0)
        ladder = _chain("add", [f"(sub (max (sub {W} {a[k]!r}) 0.0) (max (sub {W} {a[k + 1]!r}) 0.0))" for k in range(spreads)])
        return f"(loopif {hit} 0.0 (mult {ladder} (payoff 0 0 1)) $0)", [n]
    if contract == "asian":  # oldest fixing first
        s = _chain("add", [f"(model 0 (tplus $0 {-j}))" for j in reversed(range(n))])
        return f"(mult (max (sub (div {s} {float(n)}) {strike}) 0.0) (payoff $0 0 1))", [n]
    if contract == "asian_newest":
        s = _chain("add", [f"(add (model 0 (tplus $0 {-j})) (model 1 (tplus $0 {-j})))" for j in range(n)])
        return f"(mult (max (sub (div {s} {float(2 * n)}) {strike}) 0.0) (payoff $0 0 1))", [n]
    raise ValueError(contract)


def _market(contract, d, n, seed, days=None):
    """Spots, volatilities, correlation, rate, days; seed of the paths."""
    g = np.random.Generator(np.random.MT19937(seed))
    level = 100.0 if contract == "european" else 1.0
    rho = float(g.uniform(0.4, 0.6))
    if days is None:
        days = [365 * (k + 1) for k in range(n)] if contract in ("european", "basket", "autocall") else list(range(1, n + 1))
    return dict(S0=[float(level * v) for v in g.uniform(0.97, 1.03, d)], sigma=[float(v) for v in g.uniform(0.15, 0.35, d)],
                corr=[[1.0 if i == j else rho for j in range(d)] for i in range(d)], r=float(g.uniform(0.02, 0.04)),
                days=days), int(g.integers(1 << 62))


def _book(case):
    """The contracts of a portfolio: templates, maturities, date counts,
    strikes and path budgets as a book of OTC contracts mixes them."""
    g, items = random.Random(case["book"]), []
    for i in range(case["contracts"]):
        c = g.choice(["basket", "digital", "call_spread", "autocall", "barrier", "asian"])
        d, years = g.randint(1, 4), g.uniform(0.5, 10.0)
        n = min(_log_int(g, 1, 365), {"autocall": 12, "asian": 200}.get(c, 365))
        last = max(round(years * 365), n)
        days = sorted({max(1, round(last * (k + 1) / n)) for k in range(n)})
        strike = g.uniform(0.8, 1.2)
        text, tp = contract_text(c, d, len(days), strike, 0.6 + 0.1 * strike, 1 + i % 13)
        items.append(dict(contract=c, d=d, days=days, text=text, tparams=tp,
                          paths=int(min(1 << 18, max(1 << 12, math.exp(g.gauss(math.log(2 ** 15), 1.0)))))))
    return items


# ---------------------------------------------------------------------------
# States
# ---------------------------------------------------------------------------

_contexts = {}


def _context(jit):
    if jit not in _contexts:
        stream = torch.cuda.Stream()
        ctx = pc.pc_create(0, stream.cuda_stream)
        pc.pc_set_jit(ctx, jit)
        _contexts[jit] = (ctx, stream)  # the stream lives as long as its context
    return _contexts[jit][0]


class State:
    """Handles and buffers of one case; freed with it."""

    def __init__(self, case):
        self.case, self.ctx = case, _context(bool(case.get("jit")))
        self.models, self.contracts, self.plan, self.net = [], [], None, None

    def model(self, mk):
        self.models.append(pc.pc_model_create(self.ctx, **mk))
        return self.models[-1]

    def contract(self, text, tparams):
        words, consts = pc.pc_assemble(text)
        self.contracts.append(pc.pc_load_payoff(self.ctx, words, consts, tparams))
        return self.contracts[-1]

    def __del__(self):
        if self.plan:
            pc.pc_batch_destroy(self.plan)
        if self.net:
            pc.pc_mlp_destroy(self.net)
        for k in self.contracts:
            pc.pc_contract_destroy(k)
        for m in self.models:
            pc.pc_model_destroy(m)


def _widths(case):
    return [16, case["width"], case["width"], case["width"], 5]


def _network(widths, seed):
    """Parameters as a fresh network's, and features, targets and loss weights."""
    g = np.random.Generator(np.random.MT19937(seed))
    parts = []
    for fin, fout in zip(widths[:-1], widths[1:]):
        parts += [g.uniform(-1, 1, fin * fout) / math.sqrt(fin), g.uniform(-1, 1, fout) / math.sqrt(fin)]
    return np.concatenate(parts).astype(np.float32), g


def _samples(g, rows):
    """Rows like the hedge network's: log-moneyness, volatilities, ..., 1."""
    x = np.zeros((rows, 16), np.float32)
    x[:, :3] = g.normal(0, 0.4, (rows, 3))
    x[:, 3:6] = g.uniform(0.15, 0.35, (rows, 3))
    x[:, 6], x[:, 7], x[:, 8] = g.uniform(0.3, 0.7, rows), g.uniform(0.01, 0.05, rows), 1.0
    k = g.integers(0, 5, rows)
    x[:, 9], x[:, 10], x[:, 11] = (5 - k) / 5.0, k / 5.0, g.uniform(size=rows) < 0.25
    x[:, 12], x[:, 13], x[:, 14], x[:, 15] = g.uniform(0.03, 0.07, rows), g.uniform(0.95, 1.05, rows), g.uniform(0.5, 0.7, rows), 1.0
    w = x[:, :3].min(axis=1)
    y = np.stack([np.minimum(np.exp(w), 1.0 + x[:, 12])] + [np.where(x[:, i] == w, 0.5, 0.1) for i in range(3)] + [0 * w], 1)
    return x, (y + 0.05 * g.normal(size=y.shape)).astype(np.float32)


_LOSS_W = np.array([1.0, 0.1, 0.1, 0.1, 0.0], np.float32)


def prepare(case, seed):
    s = State(case)
    kind = case["kind"]
    if kind in ("price", "greeks"):
        mk, s.seed = _market(case["contract"], case["d"], case["n"], seed)
        s.m = s.model(mk)
        text, s.tparams = contract_text(case["contract"], case["d"], case["n"])
        s.words, s.consts = pc.pc_assemble(text)
        s.k = s.contract(text, s.tparams)
        if case["jit"] and kind == "price":
            pc.pc_jit_compile(s.m, s.k)
        s.sums = torch.zeros(3, dtype=torch.float64, device="cuda")
        s.paths = torch.zeros(case["paths"] if case.get("out") == "paths" else 0, dtype=torch.float32, device="cuda")
    elif kind == "portfolio":
        s.items = _book(case)
        s.n_paths = [it["paths"] for it in s.items]
        for i, it in enumerate(s.items):
            mk, path_seed = _market(it["contract"], it["d"], 0, seed * 1009 + i, it["days"])
            s.model(mk)
            s.contract(it["text"], it["tparams"])
            s.seed = path_seed if i == 0 else s.seed
        if not case["oneshot"]:
            s.plan = pc.pc_batch_create(s.models, s.contracts, s.n_paths, s.seed)
    elif kind == "mlp":
        params, g = _network(_widths(case), seed)
        x, y = _samples(g, case["rows"])
        s.params = params
        s.net = pc.pc_mlp_create(s.ctx, _widths(case), case.get("batch", case["rows"]), 1)
        pc.pc_mlp_set_params(s.net, params)
        s.x, s.t = torch.tensor(x, device="cuda"), torch.tensor(y, device="cuda")
        s.y = torch.zeros(case["rows"], 5, device="cuda")
        s.g = torch.zeros(params.size, device="cuda")
    else:
        mk, s.seed = _market("autocall", 3, 5, seed)
        s.m = s.model(mk)
        s.k = s.contract(*contract_text("autocall", 3, 5))
        params, _ = _network([16, 256, 256, 256, 5], seed)
        s.net = pc.pc_mlp_create(s.ctx, [16, 256, 256, 256, 5], 16384, 1)
        pc.pc_mlp_set_params(s.net, params)
        s.desc = pc.pc_cv_grid(s.m, case["grid"], 4.5)
        s.desc.use_gamma = int(case["gamma"])
        s.desc.beta, s.desc.beta2 = 0.9, 0.8 if case["gamma"] else 0.0
        s.cap = pc.pc_cv_table_size(s.desc) + 4
        s.tables = torch.zeros(s.cap, device="cuda")
    return s


def run(s):
    c, kind = s.case, s.case["kind"]
    if kind == "price":
        if c["out"] == "price":
            return pc.pc_price(s.m, s.k, c["paths"], s.seed)
        if c["out"] == "quote":
            k = pc.pc_load_payoff(s.ctx, s.words, s.consts, s.tparams)
            quote = pc.pc_price(s.m, k, c["paths"], s.seed)
            pc.pc_contract_destroy(k)
            return quote
        if c["out"] == "paths":
            pc.pc_price_paths(s.m, s.k, c["paths"], 0, s.seed, 0, s.sums.data_ptr(), s.paths.data_ptr())
            return s.sums, s.paths
        pc.pc_price_async(s.m, s.k, c["paths"], 0, s.seed, 0, s.sums.data_ptr())
        return s.sums
    if kind == "greeks":
        return (pc.pc_greeks_adjoint if c["mode"] == "adjoint" else pc.pc_greeks)(s.m, s.k, c["paths"], s.seed, c["d"])
    if kind == "portfolio":
        if c["oneshot"]:
            return pc.pc_price_batch(s.models, s.contracts, s.n_paths, s.seed)
        pc.pc_batch_launch(s.plan)
        return pc.pc_batch_results(s.plan, len(s.contracts))
    if kind == "mlp":
        if c["op"] == "forward":
            pc.pc_mlp_forward(s.net, s.x.data_ptr(), c["rows"], s.y.data_ptr())
            return s.y
        if c["op"] == "gradients":
            loss = pc.pc_mlp_gradients(s.net, s.x.data_ptr(), s.t.data_ptr(), _LOSS_W, c["rows"], s.g.data_ptr())
            return loss, s.g
        pc.pc_mlp_set_params(s.net, s.params)
        loss = pc.pc_mlp_train(s.net, s.x.data_ptr(), s.t.data_ptr(), c["rows"], _LOSS_W, c["batch"], c["steps"], 1e-3, 11)
        return loss, pc.pc_mlp_get_params(s.net)
    pc.pc_cv_tables_async(s.net, s.m, s.desc, s.tables.data_ptr(), s.cap)
    return pc.pc_price_cv(s.m, s.k, s.desc, s.tables.data_ptr(), c["paths"], s.seed)


def _path_ops(n, d, sites=None):
    """Operations of a path: the Philox blocks (60) and Box-Muller pairs (13)
    of its n d normals, the bridge, correlation and GBM; the payoff left out."""
    blocks = -(-n * d // 4)
    return 60 * blocks + 13 * -(-n * d // 2) + 3 * d * n + n * (d * (d + 1) // 2 + 2 * d)


def work(case):
    kind = case["kind"]
    if kind in ("price", "greeks"):
        n, d = case["n"], case["d"]
        out = 4 * case["paths"] if case.get("out") == "paths" else 0
        return {"bytes": out + n * (32 + 12 * d) + 4096, "flops": case["paths"] * _path_ops(n, d)}
    if kind == "portfolio":
        items = _book(case)
        return {"bytes": sum(4096 + len(it["days"]) * (32 + 12 * it["d"]) for it in items),
                "flops": sum(it["paths"] * _path_ops(len(it["days"]), it["d"]) for it in items)}
    if kind == "mlp":
        w = _widths(case)
        mac = sum(a * b for a, b in zip(w[:-1], w[1:]))
        par = mac + sum(w[1:])
        if case["op"] == "forward":
            return {"bytes": case["rows"] * 4 * 21 + 4 * par, "flops": 2 * mac * case["rows"]}
        if case["op"] == "gradients":
            return {"bytes": case["rows"] * 4 * 21 + 8 * par, "flops": (6 * mac - 2 * w[0] * w[1]) * case["rows"]}
        return {"bytes": case["steps"] * (case["batch"] * 84 + 28 * par), "flops": case["steps"] * (6 * mac - 2 * w[0] * w[1]) * case["batch"]}
    rows = 8 * case["grid"] ** 3 + 1
    mac = 16 * 256 + 2 * 256 * 256 + 256 * 5
    return {"bytes": rows * 48 + 4 * mac, "flops": 2 * mac * rows + case["paths"] * _path_ops(5, 3)}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------


def _uniform_blocks(b0, b1, paths, seed, stream):
    """Philox4x32-10 words of counters (b, path), b0 <= b < b1, as uniforms [b1 - b0, 4, N]."""
    low = 0xFFFFFFFF
    b = torch.arange(b0, b1, device="cuda")[:, None]
    x = [b.expand(-1, paths.numel()), paths & low, paths >> 32, torch.full_like(b, stream)]
    k0, k1 = seed & low, (seed >> 32) & low
    for _ in range(10):
        p, q = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57  # 32 x 32 bits, kept modulo 2^64
        x = [((q >> 32) & low) ^ x[1] ^ k0, q & low, ((p >> 32) & low) ^ x[3] ^ k1, p & low]
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return torch.stack([((v >> 8).double() + 0.5) * 2.0 ** -24 for v in x], 1)


def _normals(count, paths, seed, stream):
    """Normals 0 .. count - 1 of each path, a few Philox blocks at a time."""
    for b0 in range(0, -(-count // 4), 16):
        u = _uniform_blocks(b0, min(b0 + 16, -(-count // 4)), paths, seed, stream)
        r, th = torch.sqrt(-2.0 * torch.log(u[:, 0::2])), 2.0 * math.pi * u[:, 1::2]
        z = torch.stack([r * torch.cos(th), r * torch.sin(th)], 2).reshape(-1, paths.numel())
        yield from z


def _correlated(mk, paths, seed, stream):
    """X = L W [n + 1][d] over the dates: Brownian bridge by bisection, its
    nodes in the order that a walk through the dates meets them."""
    n, d = len(mk["days"]), len(mk["S0"])
    tau = [0.0] + [v / 365.0 for v in mk["days"]]
    nodes, queue = [(0, -n, n, None)], [(0, n)]
    for l, r in queue:
        if r - l >= 2:
            mid = (l + r) // 2
            nodes.append((l, -mid, mid, r))
            queue += [(l, mid), (mid, r)]
    z = _normals(n * d, paths, seed, stream)
    W = [None] * (n + 1)
    W[0] = [torch.zeros(paths.numel(), dtype=torch.float64, device="cuda")] * d
    for l, _, mid, r in sorted(nodes, key=lambda v: v[:2]):
        zs = [next(z) for _ in range(d)]
        if r is None:
            W[mid] = [math.sqrt(tau[n]) * v for v in zs]
            continue
        span = tau[r] - tau[l]
        wl, wr = (tau[r] - tau[mid]) / span, (tau[mid] - tau[l]) / span
        sd = math.sqrt((tau[mid] - tau[l]) * (tau[r] - tau[mid]) / span)
        W[mid] = [wl * W[l][i] + wr * W[r][i] + sd * zs[i] for i in range(d)]
    L = np.linalg.cholesky(np.array(mk["corr"]))
    for o in range(n + 1):
        W[o] = [sum(float(L[i, k]) * W[o][k] for k in range(i + 1)) for i in range(d)]
    return W, tau


def _parse(text):
    stack = [[]]
    for t in text.replace("(", " ( ").replace(")", " ) ").split():
        if t == "(":
            stack.append([])
        elif t == ")":
            e = stack.pop()
            stack[-1].append(e)
        else:
            stack[-1].append(t)
    return stack[0][0]


def _time(t, params):
    if isinstance(t, list):
        return _time(t[1], params) + _time(t[2], params)
    return params[int(t[1:])] if t.startswith("$") else int(t)


_BINARY = {"add": torch.add, "sub": torch.sub, "mult": torch.mul, "div": torch.div, "lt": torch.lt, "le": torch.le,
           "and": torch.logical_and, "or": torch.logical_or, "min": torch.minimum, "max": torch.maximum}


def _payoff(e, t0, params, S, disc, one):
    if not isinstance(e, list):
        return float(e) * one
    op = e[0]
    go = lambda x, t=t0: _payoff(x, t, params, S, disc, one)  # noqa: E731
    if op == "model":
        return S(int(e[1]), _time(e[2], params) + t0)
    if op == "payoff":
        return disc(_time(e[1], params) + t0) * one
    if op == "if":
        return torch.where(go(e[1]), go(e[2]), go(e[3]))
    if op == "loopif":
        n = _time(e[4], params)
        done = torch.zeros_like(one, dtype=torch.bool)
        res = torch.zeros_like(one)
        for k in range(n + 1):
            with torch.no_grad():
                new = go(e[1], t0 + k) & ~done
                done = done | new
            if isinstance(e[2], list):
                res = torch.where(new, go(e[2], t0 + k), res)
            else:
                res = torch.where(new, float(e[2]) * one, res)
        return torch.where(done, res, go(e[3], t0 + n))
    return _BINARY[op](go(e[1]), go(e[2]))


def _exact_paths(mk, text, params, n_paths, seed, stream=0, greeks=False):
    """Per chunk of paths: payoffs, and with `greeks` their derivatives by each S0 and sigma [2 d, N]."""
    prog, d, n = _parse(text), len(mk["S0"]), len(mk["days"])
    chunk = max(1 << 12, min(1 << 20, (1 << 28) // ((n + 1) * d)) >> (2 if greeks else 0))
    for first in range(0, n_paths, chunk):
        paths = torch.arange(first, min(first + chunk, n_paths), device="cuda")
        X, tau = _correlated(mk, paths, seed, stream)
        one = torch.ones(paths.numel(), dtype=torch.float64, device="cuda")
        S0 = [(v * one).requires_grad_(greeks) for v in mk["S0"]]
        sig = [(v * one).requires_grad_(greeks) for v in mk["sigma"]]

        def S(i, o):
            return S0[i] * torch.exp((mk["r"] - 0.5 * sig[i] ** 2) * tau[o] + sig[i] * X[o][i])

        v = _payoff(prog, 0, params, S, lambda o: math.exp(-mk["r"] * tau[o]), one)
        if greeks:
            grads = torch.autograd.grad(v.sum(), S0 + sig, allow_unused=True)
            yield v.detach(), torch.stack([torch.zeros_like(one) if x is None else x for x in grads])
        else:
            yield v, None


def _mean_se(s, s2, n):
    mean = s / n
    return mean, math.sqrt(max(0.0, (s2 - n * mean * mean) / (n - 1.0)) / n)


def _exact_sums(*args):
    got = [(v.sum().item(), (v * v).sum().item()) for v, _ in _exact_paths(*args)]
    return sum(a for a, _ in got), sum(b for _, b in got)


def _exact_network(widths, params, x, t=None):
    p, ws, at = torch.tensor(params, device="cuda").double().requires_grad_(), [], 0
    for fin, fout in zip(widths[:-1], widths[1:]):
        ws.append((p[at:at + fin * fout].view(fout, fin), p[at + fin * fout:at + fin * fout + fout]))
        at += fin * fout + fout
    h = torch.tensor(x, device="cuda").double()
    for i, (w, b) in enumerate(ws):
        h = h @ w.T + b
        if i + 1 < len(ws):
            h = torch.nn.functional.softplus(h, threshold=50.0)
    if t is None:
        return h.detach()
    loss = ((h - torch.tensor(t, device="cuda").double()) ** 2 * torch.tensor(_LOSS_W, device="cuda").double()).sum() / len(x)
    return loss.item(), torch.autograd.grad(loss, p)[0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        if case["op"] == "train":  # a trajectory of rounded weights: no such value
            return None
        params, g = _network(_widths(case), seed)
        x, y = _samples(g, case["rows"])
        return _exact_network(_widths(case), params, x, y if case["op"] == "gradients" else None)
    if kind == "portfolio":
        price, se = [], []
        for i, it in enumerate(_book(case)):
            mk, path_seed = _market(it["contract"], it["d"], 0, seed * 1009 + i, it["days"])
            first = path_seed if i == 0 else first
            p, e = _mean_se(*_exact_sums(mk, it["text"], it["tparams"], it["paths"], first, i), it["paths"])
            price.append(p)
            se.append(e)
        return np.array(price), np.array(se)
    c = "autocall" if kind == "cv" else case["contract"]
    d, n = (3, 5) if kind == "cv" else (case["d"], case["n"])
    mk, path_seed = _market(c, d, n, seed)
    text, params = contract_text(c, d, n)
    N = case["paths"]
    if kind == "greeks":
        s, s2 = torch.zeros(1 + 2 * d, dtype=torch.float64), torch.zeros(1 + 2 * d, dtype=torch.float64)
        for v, gr in _exact_paths(mk, text, params, N, path_seed, 0, True):
            q = torch.cat([v[None], gr])
            s, s2 = s + q.sum(1).cpu(), s2 + (q * q).sum(1).cpu()
        m = [_mean_se(float(a), float(b), N) for a, b in zip(s, s2)]
        return m[0][0], np.array([v for v, _ in m[1:1 + d]]), np.array([v for v, _ in m[1 + d:]]), np.array([e for _, e in m])
    if kind == "price" and case["out"] == "paths":
        v = torch.cat([x for x, _ in _exact_paths(mk, text, params, N, path_seed)])
        return torch.tensor([v.sum().item(), (v * v).sum().item(), float(N)], dtype=torch.float64), v
    s, s2 = _exact_sums(mk, text, params, N, path_seed)
    if kind == "cv":  # the control variate's own estimate rests on rounded hedge tables; the plain one is given
        return (None, None), _mean_se(s, s2, N)
    return torch.tensor([s, s2, float(N)], dtype=torch.float64) if case["out"] == "sums" else _mean_se(s, s2, N)
