"""Two underlyings with the window of dates in HBM: the launch takes the
denser kernel (seven blocks an SM) where that holds every tile at once.  At the
edges of that rule the paths and sums are those of the window in shared
memory, bit for bit."""
import numpy as np
import pytest

from gpu_common import Engine, torch
import paper_2108_03076_gb300 as pc
import workloads as W

pytestmark = pytest.mark.gpu

TILE, WARPS = 64, 4  # paths a tile, warps a block


@pytest.fixture(scope="module")
def eng():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    e = Engine()
    yield e
    pc.pc_set_window_mode(e.ctx, pc.WINDOW_AUTO)
    e.close()


@pytest.mark.parametrize("rounds,extra", [(6, 0), (6, 1), (7, 0), (7, 1), (14, 1)])
def test_dense_window_launches_keep_every_path(eng, rounds, extra):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    spec = W.MarketSpec([1.0, 1.2], [0.25, 0.3], W.const_corr(2, 0.4), 0.02, list(range(1, 13)))
    s = "(add (model 0 $0) (model 1 $0))"
    for j in range(1, 12):
        s = f"(add {s} (add (model 0 (tplus $0 {-j})) (model 1 (tplus $0 {-j}))))"
    m, k = eng.model(spec), eng.contract(f"(max (sub (div {s} 24.0) 1.1) 0.0)", [12])
    n = rounds * sms * WARPS * TILE + extra
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
    # past 6 sms blocks the denser kernel's 7 sms hold the rest
    dense = (rounds, extra) in ((6, 1), (7, 0))
    assert grid > 6 * sms if dense else grid == 6 * sms
