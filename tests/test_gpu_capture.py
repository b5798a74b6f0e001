"""Calls captured on the caller's stream: a graph's replay equals the same
call made eagerly, bit for bit, whatever the calls between capture and replay
do with the context's scratch; a capture that would need more scratch than
the context holds runs without it or is refused."""
import numpy as np
import pytest

from gpu_common import torch
import paper_2108_03076_gb300 as pc
import workloads as W

pytestmark = pytest.mark.gpu

TILE, WARPS = 64, 4  # paths a tile, warps a block


@pytest.fixture(params=[False, True], ids=["interpreted", "specialised"])
def ctx(request):
    """A context of its own per test: its scratch starts small."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_03076_gb300 import build
    build.build()
    st = torch.cuda.Stream()
    torch.cuda.set_stream(st)
    c = pc.pc_create(0, st.cuda_stream)
    pc.pc_set_jit(c, request.param)
    yield c
    torch.cuda.synchronize()
    pc.pc_destroy(c)


def capture(call):
    """(graph, None) of `call` captured on the current stream, or (None, the
    refusal)."""
    g, refused = torch.cuda.CUDAGraph(), None
    mark = torch.zeros(1, device="cuda")
    with torch.cuda.graph(g, stream=torch.cuda.current_stream()):
        mark.add_(1)
        try:
            call()
        except pc.PcError as e:
            refused = e
    return (None if refused else g), refused


def market(ctx, spec):
    return pc.pc_model_create(ctx, spec.S0, spec.sigma, spec.corr, spec.r, spec.days)


def contract(ctx, text, tp=()):
    w, k = pc.pc_assemble(text)
    return pc.pc_load_payoff(ctx, w, k, tp)


def newest_first(n):
    s = "(add (model 0 $0) (model 1 $0))"
    for j in range(1, n):
        s = f"(add {s} (add (model 0 (tplus $0 {-j})) (model 1 (tplus $0 {-j}))))"
    return f"(max (sub (div {s} {2.0 * n}) 1.1) 0.0)"


def test_hbm_window_never_smaller_than_its_launch(ctx, request):
    """A window buffer of six blocks an SM, then a captured call of one path
    more: the interpreter keeps to six blocks, a specialised launch that holds
    more is refused.  Captured after an eager call of that size, it runs."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    spec = W.MarketSpec([1.0, 1.2], [0.25, 0.3], W.const_corr(2, 0.4), 0.02, list(range(1, 13)))
    m, k = market(ctx, spec), contract(ctx, newest_first(12), [12])
    pc.pc_set_window_mode(ctx, pc.WINDOW_HBM)
    n = 6 * sms * WARPS * TILE
    out = torch.zeros(5, 4, dtype=torch.float64, device="cuda")

    def price(paths, row):
        return lambda: pc.pc_price_async(m, k, paths, 0, 7, 0, out[row].data_ptr())
    try:
        price(n, 0)()
        small, refused = capture(price(n, 1))
        assert refused is None
        first, refused = capture(price(n + 1, 2))
        assert first is not None or refused.name == "PC_ECUDA"
        if first is not None:
            first.replay()
            torch.cuda.synchronize()
        price(n + 1, 3)()  # grows the buffer; the captured one is kept
        second, again = capture(price(n + 1, 4))
        assert again is None
        small.replay()
        second.replay()
        torch.cuda.synchronize()
        o = out[:, :3].cpu().numpy()
        np.testing.assert_array_equal(o[1], o[0])
        np.testing.assert_array_equal(o[4], o[3])
        if first is not None:
            np.testing.assert_array_equal(o[2], o[3])
        pc.pc_set_window_mode(ctx, pc.WINDOW_SHARED)
        price(n + 1, 0)()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out[0, :3].cpu().numpy(), o[3])
    finally:
        pc.pc_contract_destroy(k)
        pc.pc_model_destroy(m)


def test_captured_scratch_is_kept(ctx):
    """Pricing and sensitivity graphs replayed after calls that outgrow the
    tile partials and the tapes they hold."""
    spec = W.MarketSpec([1.0, 1.2], [0.25, 0.3], W.const_corr(2, 0.4), 0.02, list(range(1, 31)))
    m = market(ctx, spec)
    k = contract(ctx, "(mult (max (sub (max (model 0 15) (model 1 30)) 1.1) 0.0) (payoff 30 0 1))")
    small, large = 20_000, 2_400_000
    out = torch.zeros(2, 16, dtype=torch.float64, device="cuda")
    sens = torch.zeros(2, 16, dtype=torch.float64, device="cuda")
    big = torch.zeros(16, dtype=torch.float64, device="cuda")
    try:
        pc.pc_price_async(m, k, small, 0, 7, 0, out[0].data_ptr())
        pc.pc_greeks_adjoint_async(m, k, small, 0, 7, 0, sens[0].data_ptr())
        price, refused = capture(lambda: pc.pc_price_async(m, k, small, 0, 7, 0, out[1].data_ptr()))
        assert refused is None
        greeks, refused = capture(lambda: pc.pc_greeks_adjoint_async(m, k, small, 0, 7, 0, sens[1].data_ptr()))
        assert refused is None
        # a capture that would have to grow them is refused
        for call in (pc.pc_price_async, pc.pc_greeks_adjoint_async):
            _, refused = capture(lambda: call(m, k, large, 0, 7, 0, big.data_ptr()))
            assert refused is not None and refused.name == "PC_ECUDA"
        pc.pc_price_async(m, k, large, 0, 7, 0, big.data_ptr())
        pc.pc_greeks_adjoint_async(m, k, large, 0, 7, 0, big.data_ptr())
        for g in (price, greeks):
            g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out[1].cpu().numpy(), out[0].cpu().numpy())
        np.testing.assert_array_equal(sens[1].cpu().numpy(), sens[0].cpu().numpy())
        assert out[0, 2].item() == small and out[0, 0].item() > 0
    finally:
        pc.pc_contract_destroy(k)
        pc.pc_model_destroy(m)


BARRIER = ("(loopif (or (le (model 0 0) 0.75) (le (model 1 0) 0.75)) 0.0 "
           "(mult (max (sub (min (model 0 0) (model 1 0)) {K}) 0.0) (payoff 0 0 1)) 240)")


def daily(ctx):
    return pc.pc_model_create(ctx, [1.0, 1.02], [0.28, 0.2], [[1.0, 0.4], [0.4, 1.0]], 0.02, list(range(1, 241)))


def test_a_failed_screened_call_writes_no_payoffs(ctx):
    """A call that finds no memory for the window of dates leaves the payoffs
    as they were, the screened paths' too."""
    m, k = daily(ctx), contract(ctx, BARRIER.format(K=0.9))
    n = 300_000
    out = torch.zeros(4, dtype=torch.float64, device="cuda")
    x = torch.full((n,), float("nan"), device="cuda")
    try:
        pc.pc_price_paths(m, k, n, 0, 99, 0, out.data_ptr(), x.data_ptr())  # (the screen's buffers are there)
        torch.cuda.synchronize()
        assert not torch.isnan(x).any()
        x.fill_(float("nan"))
        pc.pc_set_window_mode(ctx, pc.WINDOW_HBM)
        pc.pc_debug_fail_allocations(ctx, 1)
        with pytest.raises(pc.PcError) as e:
            pc.pc_price_paths(m, k, n, 0, 99, 0, out.data_ptr(), x.data_ptr())
        assert e.value.name == "PC_ENOMEM"
        torch.cuda.synchronize()
        assert torch.isnan(x).all()
    finally:
        pc.pc_debug_fail_allocations(ctx, 0)
        pc.pc_contract_destroy(k)
        pc.pc_model_destroy(m)
