"""Specialised kernels on models of many date grids: a program that needs
more bridge nodes than a static walk holds has one general kernel, whatever
the grid, and launches of different shared memory sizes on it in any order
give the interpreter's payoffs bit for bit."""
import numpy as np
import pytest

from gpu_common import Engine, torch
import paper_2108_03076_gb300 as pc
import workloads as W

pytestmark = pytest.mark.gpu

N = 3000
GRIDS = [365, 20, 100, 252, 40, 365, 20]


@pytest.fixture()
def eng():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    e = Engine()
    pc.pc_debug_set_jit_pairs(e.ctx, 1)
    yield e
    e.close()


def spec(n):
    return W.MarketSpec([1.0, 1.1], [0.25, 0.3], W.const_corr(2, 0.4), 0.02, list(range(1, n + 1)))


BARRIER = "(loopif (lt (min (model 0 0) (model 1 0)) 0.8) 0.25 (mult (model 0 0) (payoff 0 0 1)) $0)"
# 18 dates, each pair the later date first: a window of two
READS = [d for i in range(1, 10) for d in (2 * i, 2 * i - 1)]
LOOKBACK = "(mult " + "(add " * (len(READS) - 1) + f"(model 0 {READS[0]})" + \
    "".join(f" (model {j % 2} {o}))" for j, o in enumerate(READS[1:])) + " (payoff 18 0 1))"


@pytest.mark.parametrize("text,grid_param", [(BARRIER, True), (LOOKBACK, False)], ids=["barrier", "lookback"])
@pytest.mark.parametrize("what", ["price", "tangent"])
def test_one_general_kernel_for_all_grids(eng, text, grid_param, what):
    kernels, seen = [], {}
    for n in GRIDS:
        m, k = eng.model(spec(n)), eng.contract(text, [n] if grid_param else [])
        got = {}
        for jit in (False, True):
            pc.pc_set_jit(eng.ctx, jit)
            if what == "price":
                got[jit] = eng.paths(m, k, N, 11)
            else:
                out = torch.zeros(8, dtype=torch.float64, device="cuda")
                x = torch.zeros(3 * N, device="cuda")
                pc.pc_debug_greeks_paths(m, k, N, 0, 11, 0, out.data_ptr(), x.data_ptr())
                torch.cuda.synchronize()
                got[jit] = x.cpu().numpy(), out.cpu().numpy()
        pc.pc_set_jit(eng.ctx, False)
        for a, b in zip(got[False], got[True]):
            np.testing.assert_array_equal(a, b)
        kernels.append(pc.pc_debug_jit_kernels(eng.ctx))
        if n in seen:
            np.testing.assert_array_equal(got[True][0], seen[n])
        seen[n] = got[True][0]
    if not grid_param:  # (the barrier's instructions hold its number of dates)
        assert kernels == [kernels[0]] * len(GRIDS)


def test_compile_leaves_nothing_to_the_first_large_call(eng):
    """A screened barrier has two kernels, for its small launches and for the
    paths left by the screen: pc_jit_compile makes both."""
    m, k = eng.model(spec(240)), eng.contract(BARRIER, [240])
    assert pc.pc_debug_price_kernels(m, k, 1 << 20) == 3 and pc.pc_debug_price_kernels(m, k, 1 << 12) == 1
    pc.pc_set_jit(eng.ctx, True)
    pc.pc_jit_compile(m, k)
    assert pc.pc_debug_jit_kernels(eng.ctx) == 2
    large, small = pc.pc_price(m, k, 1 << 20, 5), pc.pc_price(m, k, 1 << 12, 5)
    assert pc.pc_debug_jit_kernels(eng.ctx) == 2
    pc.pc_set_jit(eng.ctx, False)
    assert (large, small) == (pc.pc_price(m, k, 1 << 20, 5), pc.pc_price(m, k, 1 << 12, 5))


def test_compile_before_the_context_is_switched(eng):
    """pc_jit_compile while the context still interprets compiles the kernel
    that the first specialised call runs."""
    text = "(mult (max (sub (max (model 0 2) (model 1 5)) 1.0) 0.0) (payoff 5 0 1))"
    m, k = eng.model(spec(5)), eng.contract(text)
    plain = pc.pc_price(m, k, 1 << 12, 5)
    pc.pc_jit_compile(m, k)
    compiled = pc.pc_debug_jit_kernels(eng.ctx)
    pc.pc_set_jit(eng.ctx, True)
    assert pc.pc_price(m, k, 1 << 12, 5) == plain
    assert pc.pc_debug_jit_kernels(eng.ctx) == compiled == 1
