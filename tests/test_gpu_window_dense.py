"""The window of dates in HBM, one to four underlyings: where one block an SM
more than the usual launch holds every tile at once, the launch takes it.  At
the edges of that rule paths and sums are those of the window in shared
memory, bit for bit."""
import numpy as np
import pytest

from gpu_common import Engine, torch
import paper_2108_03076_gb300 as pc
import workloads as W

pytestmark = pytest.mark.gpu

TILE, WARPS = 64, 4  # paths a tile, warps a block
USUAL = {1: 7, 2: 6, 3: 5, 4: 5}  # blocks an SM


@pytest.fixture(scope="module")
def eng():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    e = Engine()
    yield e
    pc.pc_set_window_mode(e.ctx, pc.WINDOW_AUTO)
    e.close()


@pytest.mark.parametrize("d", [1, 2, 3, 4])
@pytest.mark.parametrize("more,extra", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_one_block_more_where_it_holds_every_tile(eng, d, more, extra):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    spec = W.MarketSpec([1.0 + 0.1 * i for i in range(d)], [0.25] * d, W.const_corr(d, 0.4), 0.02, list(range(1, 9)))
    terms = [f"(model {i} (tplus $0 {-j}))" for j in range(8) for i in range(d)]
    s = terms[0]
    for t in terms[1:]:
        s = f"(add {s} {t})"
    m, k = eng.model(spec), eng.contract(f"(max (sub (div {s} {8.0 * d}) 1.1) 0.0)", [8])
    n = (USUAL[d] + more) * sms * WARPS * TILE + extra
    out = {}
    for mode in (pc.WINDOW_SHARED, pc.WINDOW_HBM):
        pc.pc_set_window_mode(eng.ctx, mode)
        out[mode] = eng.paths(m, k, n, 0x51) + (pc.pc_price(m, k, n, 0x51),)
        if mode == pc.WINDOW_HBM:
            grid = pc.pc_price_info(m, k, n).grid
    pc.pc_set_window_mode(eng.ctx, pc.WINDOW_AUTO)
    np.testing.assert_array_equal(out[pc.WINDOW_SHARED][0], out[pc.WINDOW_HBM][0])
    np.testing.assert_array_equal(out[pc.WINDOW_SHARED][1], out[pc.WINDOW_HBM][1])
    assert out[pc.WINDOW_SHARED][2] == out[pc.WINDOW_HBM][2]
    dense = (more, extra) in ((0, 1), (1, 0))
    assert grid > USUAL[d] * sms if dense else grid == USUAL[d] * sms
