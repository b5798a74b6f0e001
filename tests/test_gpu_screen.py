"""Screened launches: paths of a barrier decided at the last, middle or
quarter dates leave before the walk.  Payoffs and sums must equal, bit for
bit, those of launches too small to be screened (the same paths in pieces)
and of pc_price_noalloc (never screened), on both evaluators."""
import numpy as np
import pytest

from gpu_common import torch
import paper_2108_03076_gb300 as pc

pytestmark = pytest.mark.gpu

LADDER = "(mult (max (sub (min (model 0 0) (model 1 0)) 0.9) 0.0) (payoff 0 0 1))"
OR = "(or (le (model 0 0) 0.75) (le (model 1 0) 0.75))"
CASES = {
    # name: (program, template parameters, dates, t_now)
    "knock_out_either": (f"(loopif {OR} 0.0 {LADDER} $0)", [240], 240, 0),
    "rebate_on_the_worst": (f"(loopif (lt (min (model 0 0) (model 1 0)) 0.8) 0.25 {LADDER} $0)", [365], 365, 0),
    "up_and_out_on_the_best": (f"(loopif (le 1.2 (max (model 0 0) (model 1 0))) 0.1 {LADDER} $0)", [301], 301, 0),
    "above_either": (f"(loopif (or (lt 1.25 (model 0 0)) (lt 1.25 (model 1 0))) 0.0 {LADDER} $0)", [256], 256, 0),
    # the range ends before the middle; the payoff is read later
    "early_range": (f"(loopif {OR} 0.0 (mult (model 1 150) (payoff 150 0 1)) 130)", [], 300, 0),
    # the range starts late (the condition looks ahead)
    "late_range": ("(loopif (le (model 0 100) 0.8) 0.5 (mult (model 1 199) (payoff 199 0 1)) 100)", [], 200 + 99, 0),
    # one underlying watched of two; a later valuation date
    "one_watched_later": ("(loopif (le (model 0 3) 0.85) 0.0 (mult (model 1 0) (payoff 0 0 1)) 250)", [], 253, 2),
    # and-tests are not screened, nor is a loop inside a sum
    "both": (f"(loopif (and (le (model 0 0) 0.9) (le (model 1 0) 0.9)) 0.0 {LADDER} $0)", [240], 240, 0),
    "inside_a_sum": (f"(add 1.0 (loopif {OR} 0.0 {LADDER} $0))", [240], 240, 0),
}


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


def run(ctx, m, k, n, offset):
    out = torch.zeros(4, dtype=torch.float64, device="cuda")
    x = torch.full((n,), float("nan"), device="cuda")
    pc.pc_price_paths(m, k, n, offset, 4711, 3, out.data_ptr(), x.data_ptr())
    torch.cuda.synchronize()
    return x.cpu().numpy(), out.cpu().numpy()


@pytest.mark.parametrize("case", list(CASES))
def test_screened_equals_unscreened(ctx, case):
    text, tp, n, now = CASES[case]
    piece, pieces, offset = 40000 - 7, 11, 12345  # 440 k paths: screened from 200 dates; a piece is not
    hist = [[1.01, 0.98]] * now
    m = pc.pc_model_create(ctx, [1.0, 1.02], [0.28, 0.2], [[1.0, 0.4], [0.4, 1.0]], 0.02, list(range(1, n + 1)), now,
                           hist or None, [-1 - i for i in range(now)] or None)
    w, c = pc.pc_assemble(text)
    k = pc.pc_load_payoff(ctx, w, c, tp)
    try:
        N = piece * pieces
        x, sums = run(ctx, m, k, N, offset)
        parts = [run(ctx, m, k, piece, offset + i * piece)[0] for i in range(pieces)]
        np.testing.assert_array_equal(x, np.concatenate(parts))
        plain = torch.zeros(4, dtype=torch.float64, device="cuda")
        pc.pc_price_noalloc(m, k, N, offset, 4711, 3, plain.data_ptr())
        torch.cuda.synchronize()
        np.testing.assert_array_equal(sums[:3], plain.cpu().numpy()[:3])
        again = torch.zeros(4, dtype=torch.float64, device="cuda")
        pc.pc_price_async(m, k, N, offset, 4711, 3, again.data_ptr())
        torch.cuda.synchronize()
        np.testing.assert_array_equal(again.cpu().numpy()[:3], sums[:3])
    finally:
        pc.pc_contract_destroy(k)
        pc.pc_model_destroy(m)



def test_captured_launches_keep_their_buffers(ctx):
    """A screened launch captured on the caller's stream replays right after a
    larger call has grown the context's screen buffers; a capture that would
    have to grow them runs unscreened."""
    text, tp, n, _ = CASES["knock_out_either"]
    m = pc.pc_model_create(ctx, [1.0, 1.02], [0.28, 0.2], [[1.0, 0.4], [0.4, 1.0]], 0.02, list(range(1, n + 1)), 0, None, None)
    w, c = pc.pc_assemble(text)
    k = pc.pc_load_payoff(ctx, w, c, tp)
    small, large = 300_000, 600_000  # both screened, the partials of either fit from the start
    try:
        out = torch.zeros(3, 4, dtype=torch.float64, device="cuda")
        ref = torch.zeros(2, 4, dtype=torch.float64, device="cuda")
        for i, paths in enumerate((small, large)):
            pc.pc_price_noalloc(m, k, paths, 0, 99, 0, ref[i].data_ptr())
        pc.pc_price_async(m, k, 100, 0, 99, 0, out[0].data_ptr())     # (the unscreened kernel is loaded)
        pc.pc_price_async(m, k, small, 0, 99, 0, out[0].data_ptr())
        torch.cuda.synchronize()
        graphs = []
        for i, paths in enumerate((small, large)):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=torch.cuda.current_stream()):
                pc.pc_price_async(m, k, paths, 0, 99, 0, out[i].data_ptr())
            graphs.append(g)
        pc.pc_price_async(m, k, large, 0, 99, 0, out[2].data_ptr())   # grows the buffers
        out[:2].zero_()
        for g in graphs:
            g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out[:2, :3].cpu().numpy(), ref[:, :3].cpu().numpy())
        np.testing.assert_array_equal(out[2, :3].cpu().numpy(), ref[1, :3].cpu().numpy())
    finally:
        pc.pc_contract_destroy(k)
        pc.pc_model_destroy(m)
