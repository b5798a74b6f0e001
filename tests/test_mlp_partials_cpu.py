"""Host-side sizes of a network's weight-gradient partials (no GPU): whatever
number of rows a call has, its split-k partials fit the buffer that the
network was created with.  Fewer rows can take more splits (ranges are whole
64-row chunks: 8,192 rows make 64 splits of two chunks, 4,864 rows 76 of one),
so the buffer's size is not that of the largest call."""
import pytest

pc = pytest.importorskip("paper_2108_03076_gb300")

WIDTHS = [[16, 256, 256, 256, 5], [16, 5], [16, 64, 5], [3, 64, 128, 64, 1], [16, 384, 384, 384, 5],
          [16] + [64] * 7 + [5], [16, 1024, 1024, 5]]


@pytest.fixture(scope="session", autouse=True)
def built():
    from paper_2108_03076_gb300 import build
    build.build()


@pytest.mark.parametrize("widths", WIDTHS, ids=lambda w: "-".join(map(str, w)))
@pytest.mark.parametrize("sms", [148, 152])
def test_partials_of_every_batch_fit(widths, sms):
    for max_batch in (1, 64, 65, 1000, 4096, 8192, 16384, 65536):
        over = [(b, *wh) for b in range(min(64, max_batch), max_batch + 1, 64)
                for wh in [pc.pc_debug_mlp_partials(widths, max_batch, b, sms)] if wh[0] > wh[1]]
        assert not over, (max_batch, over[:3])
