"""Barriers over a range of dates on the interpreting kernels: a test of plain
leaves (decoded once, on dates just produced, produced before, or history) has
the payoffs, bit for bit, of the same test on leaves scaled by two (the
general form; exact in binary).  And kernels that start at a later date sum
what their per-path form writes."""
import numpy as np
import pytest

from gpu_common import torch
import paper_2108_03076_gb300 as pc

pytestmark = pytest.mark.gpu

N = 5000


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_03076_gb300 import build
    build.build()
    st = torch.cuda.Stream()
    torch.cuda.set_stream(st)
    c = pc.pc_create(0, st.cuda_stream)
    yield c
    pc.pc_destroy(c)


def model(ctx, d, n, now=0):
    corr = [[1.0 if i == j else 0.3 for j in range(d)] for i in range(d)]
    hist = [[1.0 - 0.01 * i + 0.02 * j for j in range(d)] for i in range(now)]
    return pc.pc_model_create(ctx, [1.0 + 0.05 * i for i in range(d)], [0.3] * d, corr, 0.02,
                              [7 * (k + 1) for k in range(n)], now, hist or None, [-7 * (i + 1) for i in range(now)] or None)


def paths(ctx, m, text):
    w, c = pc.pc_assemble(text)
    k = pc.pc_load_payoff(ctx, w, c)
    out = torch.zeros(2, 4, dtype=torch.float64, device="cuda")
    x = torch.full((N,), float("nan"), device="cuda")
    pc.pc_price_paths(m, k, N, 3, 99, 7, out[0].data_ptr(), x.data_ptr())
    pc.pc_price_async(m, k, N, 3, 99, 7, out[1].data_ptr())
    torch.cuda.synchronize()
    pc.pc_contract_destroy(k)
    o = out[:, :3].cpu().numpy()
    np.testing.assert_array_equal(o[0], o[1])
    return x.cpu().numpy()


def sensitivities(ctx, m, d, text):
    """Per-path tangents of every underlying and adjoints, with their sums."""
    w, c = pc.pc_assemble(text)
    k = pc.pc_load_payoff(ctx, w, c)
    res = []
    for l in range(d):
        out = torch.zeros(8, dtype=torch.float64, device="cuda")
        x = torch.full((3 * N,), float("nan"), device="cuda")
        pc.pc_debug_greeks_paths(m, k, N, 3, 99, l, out.data_ptr(), x.data_ptr())
        res += [out, x]
    out = torch.zeros(20, dtype=torch.float64, device="cuda")
    x = torch.full(((1 + 2 * d) * N,), float("nan"), device="cuda")
    pc.pc_debug_adjoint_paths(m, k, N, 3, 99, out.data_ptr(), x.data_ptr())
    torch.cuda.synchronize()
    pc.pc_contract_destroy(k)
    return [r.cpu().numpy() for r in res + [out, x]]


def chain(op, xs):
    s = xs[0]
    for x in xs[1:]:
        s = f"({op} {s} {x})"
    return s


TESTS = {
    "any_below": lambda leaf, d, k: chain("or", [f"(le {leaf(i)} {k(0.8125)})" for i in range(d)]),
    "any_strictly_above": lambda leaf, d, k: chain("or", [f"(lt {k(1.1875)} {leaf(i)})" for i in range(d)]),
    "worst_below": lambda leaf, d, k: f"(lt {chain('min', [leaf(i) for i in range(d)])} {k(0.8125)})",
    "best_above": lambda leaf, d, k: f"(le {k(1.1875)} {chain('max', [leaf(i) for i in range(d)])})",
    "all_below": lambda leaf, d, k: chain("and", [f"(le {leaf(i)} {k(1.0625)})" for i in range(d)]),
    "worst_above": lambda leaf, d, k: f"(le {k(0.9375)} {chain('min', [leaf(i) for i in range(d)])})",
}


@pytest.mark.parametrize("test", list(TESTS))
@pytest.mark.parametrize("d,n,now", [(1, 5, 0), (1, 40, 3), (2, 40, 0), (2, 9, 3), (3, 30, 2), (4, 12, 1)])
def test_plain_tests_equal_scaled_ones(ctx, test, d, n, now):
    m = model(ctx, d, n, now)
    plain = TESTS[test](lambda i: f"(model {i} 0)", d, lambda k: k)
    scaled = TESTS[test](lambda i: f"(mult (model {i} 0) 2.0)", d, lambda k: 2.0 * k)
    top = n + now
    try:
        seen = set()
        for form in ("{}", "(add (mult 0.0 (model 0 %d)) {})" % top, "(add {} (mult 0.0 (model 0 %d)))" % (top // 2),
                     "(add (mult 0.0 (model 0 %d)) {})" % (top // 2)):
            a, b = (paths(ctx, m, form.format(f"(loopif {t} 0.25 (model {d - 1} 0) {top})")) for t in (plain, scaled))
            np.testing.assert_array_equal(a, b)
            seen.add(a.tobytes())
        assert len(seen) == 1  # the forms read the same dates in other orders
    finally:
        pc.pc_model_destroy(m)


@pytest.mark.parametrize("d", [1, 2, 3, 4])
@pytest.mark.parametrize("n,first", [(2, 2), (30, 2), (30, 17), (365, 364)])
def test_sums_of_walks_that_start_later(ctx, d, n, first):
    m = model(ctx, d, n)
    try:
        x = paths(ctx, m, f"(max (sub (model {d - 1} {first}) (model 0 {n})) 0.0)")
        assert np.all(np.isfinite(x)) and (first == n and d == 1 or x.max() > 0)
    finally:
        pc.pc_model_destroy(m)


@pytest.mark.parametrize("test", list(TESTS))
@pytest.mark.parametrize("d,n,now", [(1, 40, 3), (2, 9, 0), (3, 30, 2), (4, 12, 1)])
def test_sensitivities_of_plain_tests_equal_scaled_ones(ctx, test, d, n, now):
    m = model(ctx, d, n, now)
    plain = TESTS[test](lambda i: f"(model {i} 0)", d, lambda k: k)
    scaled = TESTS[test](lambda i: f"(mult (model {i} 0) 2.0)", d, lambda k: 2.0 * k)
    top = n + now
    try:
        for form in ("{}", "(add (mult 0.0 (model 0 %d)) {})" % top):
            a, b = (sensitivities(ctx, m, d, form.format(f"(loopif {t} 0.25 (model {d - 1} 0) {top})"))
                    for t in (plain, scaled))
            for x, y in zip(a, b):
                np.testing.assert_array_equal(x, y)
    finally:
        pc.pc_model_destroy(m)
