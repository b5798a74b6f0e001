"""Walks that leave unread dates out: the interpreting kernels skip to the
date a program needs, a specialised kernel runs a static walk over the dates
it reads.  Every value must be the full walk's bit for bit: a zero-rate
contract paying S_l(o) has the payoffs of pc_debug_paths' S_l(o) (which walks
every date), whatever the set of dates read, on both evaluators."""
import numpy as np
import pytest

from gpu_common import torch
import paper_2108_03076_gb300 as pc

pytestmark = pytest.mark.gpu

N = 203  # paths: several tiles, ragged


@pytest.fixture(scope="module", params=[False, True], ids=["interpreted", "specialised"])
def ctx(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_03076_gb300 import build
    build.build()
    st = torch.cuda.Stream()
    torch.cuda.set_stream(st)
    c = pc.pc_create(0, st.cuda_stream)
    pc.pc_set_jit(c, request.param)
    yield c
    pc.pc_destroy(c)


def model(ctx, d, n):
    corr = [[1.0 if i == j else 0.3 for j in range(d)] for i in range(d)]
    return pc.pc_model_create(ctx, [1.0 + 0.5 * i for i in range(d)], [0.2 + 0.05 * i for i in range(d)], corr, 0.0,
                              [3 * k + 2 for k in range(n)])


def payoffs(ctx, m, text, offset):
    w, k = pc.pc_assemble(text)
    h = pc.pc_load_payoff(ctx, w, k)
    out = torch.zeros(4, dtype=torch.float64, device="cuda")
    x = torch.full((N,), float("nan"), device="cuda")
    pc.pc_price_paths(m, h, N, offset, 99, 7, out.data_ptr(), x.data_ptr())
    torch.cuda.synchronize()
    pc.pc_contract_destroy(h)
    return x.cpu().numpy()


def read(reads, l=0):
    """S_l summed over the dates in the order given (zero rate: discount 1)."""
    s = f"(model {l} {reads[0]})"
    for o in reads[1:]:
        s = f"(add {s} (model {l} {o}))"
    return f"(mult {s} (payoff {max(reads)} 0 1))"


@pytest.mark.parametrize("d", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 16, 17, 100, 365])
def test_unread_dates_change_no_value(ctx, d, n):
    offset = (1 << 32) - 100  # paths cross a multiple of 2^32
    m = model(ctx, d, n)
    try:
        S = torch.zeros((N, d, n + 1), device="cuda")
        pc.pc_debug_paths(m, N, offset, 99, 7, S.data_ptr())
        torch.cuda.synchronize()
        S = S.cpu().numpy()
        picks = sorted({1, 2, n // 3, n // 2, n // 2 + 1, n - 1, n} & set(range(1, n + 1)))
        sets = [[o] for o in picks] + [picks, picks[::-1], [n, 1], [1, n]]
        if n >= 5:
            sets += [[2, n - 1, 3], list(range(1, min(n, 15) + 1)), list(range(n - 3, n + 1))]
        for i, reads in enumerate(sets):
            l = i % d
            want = S[:, l, reads[0]]
            for o in reads[1:]:
                want = want + S[:, l, o]  # float32, in the program's order
            np.testing.assert_array_equal(payoffs(ctx, m, read(reads, l), offset), want, err_msg=f"{reads}")
    finally:
        pc.pc_model_destroy(m)


@pytest.mark.parametrize("d,n", [(1, 12), (3, 16), (2, 90)])
def test_loops_and_skipped_branches_meet_the_frontier(ctx, d, n):
    """A loop that some warps leave early, then reads ahead of and behind its
    last date; an if whose branches read different dates before a common read."""
    m = model(ctx, d, n)
    try:
        S = torch.zeros((N, d, n + 1), device="cuda")
        pc.pc_debug_paths(m, N, 0, 99, 7, S.data_ptr())
        torch.cuda.synchronize()
        S = S.cpu().numpy()
        h, top = n // 2, np.float32(1.04)
        loop = f"(loopif (lt {float(top)} (model 0 0)) 2.0 (model 0 1) {h})"
        hit = (S[:, 0, :h + 1] > top).any(axis=1)
        first = np.where(hit, np.float32(2.0), S[:, 0, h + 1])
        both = f"(mult (add {loop} (model {d - 1} {n})) (payoff {n} 0 1))"
        np.testing.assert_array_equal(payoffs(ctx, m, both, 0), first + S[:, d - 1, n])
        back = f"(mult (add {loop} (model {d - 1} 2)) (payoff {n} 0 1))"
        np.testing.assert_array_equal(payoffs(ctx, m, back, 0), first + S[:, d - 1, 2])
        # one path in a few takes the then-branch: some warps skip it
        c = float(np.sort(S[:, 0, 1])[-3])
        branch = f"(mult (add (if (le {c!r} (model 0 1)) (model 0 {h}) (model 0 {h + 2})) (model 0 {n})) (payoff {n} 0 1))"
        want = np.where(S[:, 0, 1] >= np.float32(c), S[:, 0, h], S[:, 0, h + 2]) + S[:, 0, n]
        np.testing.assert_array_equal(payoffs(ctx, m, branch, 0), want)
    finally:
        pc.pc_model_destroy(m)


def test_a_program_on_many_grids(ctx):
    """One program on more grids than it gets static walks for: the later
    models take the general kernel, with the same values."""
    text = "(mult (add (model 0 1) (model 0 4)) (payoff 4 0 1))"
    for n in range(4, 16):
        m = model(ctx, 1, n)
        try:
            S = torch.zeros((N, 1, n + 1), device="cuda")
            pc.pc_debug_paths(m, N, 0, 99, 7, S.data_ptr())
            torch.cuda.synchronize()
            S = S.cpu().numpy()
            np.testing.assert_array_equal(payoffs(ctx, m, text, 0), S[:, 0, 1] + S[:, 0, 4])
        finally:
            pc.pc_model_destroy(m)
