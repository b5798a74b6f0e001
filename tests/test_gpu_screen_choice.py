"""Which launches are screened, and that the screened ones settle the paths
that the walk would have: barriers whose range misses some of the screened
dates, against the same paths in pieces too small to be screened."""
import numpy as np
import pytest

from gpu_common import torch
import paper_2108_03076_gb300 as pc
from test_gpu_screen import CASES, run

pytestmark = pytest.mark.gpu

PIECE, PIECES, OFFSET = 40000 - 7, 11, 12345


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


def market(ctx, n, now=0, spots=(1.0, 1.02)):
    hist = [[1.01 * spots[0], 0.98 * spots[0]]] * now
    return pc.pc_model_create(ctx, list(spots), [0.28, 0.2], [[1.0, 0.4], [0.4, 1.0]], 0.02, list(range(1, n + 1)), now,
                              hist or None, [-1 - i for i in range(now)] or None)


def kernels(m, k):
    return pc.pc_debug_price_kernels(m, k, PIECE * PIECES), pc.pc_debug_price_kernels(m, k, PIECE)


@pytest.mark.parametrize("case,want", [
    ("knock_out_either", 3), ("rebate_on_the_worst", 3), ("up_and_out_on_the_best", 3), ("above_either", 3),
    ("late_range", 3), ("one_watched_later", 3), ("both", 1), ("inside_a_sum", 1),
    # one screened date in the range and 1 % of the paths below the level there
    ("early_range", 1)])
def test_barriers_that_are_screened(ctx, case, want):
    text, tp, n, now = CASES[case]
    w, c = pc.pc_assemble(text)
    m, k = market(ctx, n, now), pc.pc_load_payoff(ctx, w, c, tp)
    try:
        assert kernels(m, k) == (want, 1)
    finally:
        pc.pc_contract_destroy(k)
        pc.pc_model_destroy(m)


# Of 300 dates the screened ones are 300, 150, 75 and 225.
RANGES = {"to_the_quarter": (1, 75), "before_the_middle": (1, 130), "past_the_middle": (1, 151),
          "from_the_middle": (150, 99), "last_quarter": (225, 30), "between_two": (80, 60)}


@pytest.mark.parametrize("name", list(RANGES))
def test_ranges_that_hold_some_of_the_screened_dates(ctx, name):
    first, length = RANGES[name]
    dates = [d for d in (75, 150, 225, 300) if first <= d <= first + length]
    text = (f"(loopif (le (model 0 {first}) 0.93) 0.25 (mult (model 1 {300 - length}) (payoff {300 - length} 0 1)) "
            f"{length})")
    w, c = pc.pc_assemble(text)
    m, k = market(ctx, 300), pc.pc_load_payoff(ctx, w, c)
    try:
        assert kernels(m, k) == (3 if dates else 1, 1)
        x, sums = run(ctx, m, k, PIECE * PIECES, OFFSET)
        if dates:  # every other path is settled, and has the literal as its payoff
            walked = pc.pc_debug_walked_paths(ctx)
            assert np.count_nonzero(x != np.float32(0.25)) <= walked < 0.98 * x.size
        parts = [run(ctx, m, k, PIECE, OFFSET + i * PIECE)[0] for i in range(PIECES)]
        np.testing.assert_array_equal(x, np.concatenate(parts))
        assert 0.02 < np.mean(x == np.float32(0.25)) < 0.98
        plain = torch.zeros(4, dtype=torch.float64, device="cuda")
        pc.pc_price_noalloc(m, k, PIECE * PIECES, OFFSET, 4711, 3, plain.data_ptr())
        torch.cuda.synchronize()
        np.testing.assert_array_equal(sums[:3], plain.cpu().numpy()[:3])
    finally:
        pc.pc_contract_destroy(k)
        pc.pc_model_destroy(m)
