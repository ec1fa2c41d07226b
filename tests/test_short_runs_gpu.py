"""Row-ring kernel, few streams: output rows cut into runs of eight and more, last runs of any length, blocks that begin mid-stream."""
import pytest

from paper_1804_10727_b200 import idf
from paper_1804_10727_b200.workloads import conv, POOL
from helpers import assert_close, assert_equal, rand_net, with_shifts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [16, 17, 25, 33, 81])              # two runs and up; 81: ten runs, the last one of a single row
@pytest.mark.parametrize("mode,pool", [("i8", False), ("i8", True), ("bf16", False), ("bf16", True)])
def test_short_runs_match_oracle(orc, mode, pool, H):
    layers = (conv(32, 32, 3, pad=1),) + ((POOL,) if pool else ())
    if mode == "i8":
        layers = with_shifts(layers, 8)
    x, ws, bs = rand_net(mode, layers, H, 20, 32, S=3, seed=H)
    want = orc.forward(mode, layers, x, ws, bs)
    for chunks in (None, [H], [H // 2, H - H // 2], [1, H - 1]):
        net = idf.Net(mode, layers, 20, 32, 3, ws, bs)
        got = idf.infer(net, x, chunks=chunks, last=True)
        assert net.status()[0] > 0
        (assert_equal if mode == "i8" else assert_close)(got, want, f"{mode}/{H}/{chunks}")
        net.close()
