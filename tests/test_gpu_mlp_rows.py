"""A network called with fewer rows than it was created for, at a row count
whose weight gradients take more split-k partials than the largest call's:
the same gradients, losses and trained parameters as a network created for
exactly those rows, bit for bit."""
import numpy as np
import pytest

from gpu_common import Engine, torch
import paper_2108_03076_gb300 as pc

pytestmark = pytest.mark.gpu

WIDTHS = [16, 256, 256, 256, 5]


@pytest.fixture(scope="module")
def eng():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    e = Engine()
    yield e
    e.close()


@pytest.mark.parametrize("max_batch", [8192, 16384])
def test_fewer_rows_than_created_for(eng, max_batch):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    taken = {b: pc.pc_debug_mlp_partials(WIDTHS, max_batch, b, sms)[0] for b in range(64, max_batch + 1, 64)}
    rows = max(taken, key=taken.get)
    assert rows < max_batch and taken[rows] > taken[max_batch]
    rng = np.random.default_rng(5)
    x = torch.tensor(rng.normal(size=(rows, WIDTHS[0])).astype(np.float32), device="cuda")
    t = torch.tensor(rng.normal(size=(rows, WIDTHS[-1])).astype(np.float32), device="cuda")
    w = np.ones(WIDTHS[-1], np.float32)
    got = []
    for created_for in (max_batch, rows):
        net = pc.pc_mlp_create(eng.ctx, WIDTHS, created_for, 3)
        try:
            g = torch.full((pc.pc_mlp_query(net).n_params,), float("nan"), dtype=torch.float32, device="cuda")
            torch.cuda.synchronize()
            loss = pc.pc_mlp_gradients(net, x.data_ptr(), t.data_ptr(), w, rows, g.data_ptr())
            trained = pc.pc_mlp_train(net, x.data_ptr(), t.data_ptr(), rows, w, rows, 3, 1e-3, 9)
            got.append((loss, g.cpu().numpy(), trained, pc.pc_mlp_get_params(net)))
        finally:
            pc.pc_mlp_destroy(net)
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
