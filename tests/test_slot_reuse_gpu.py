"""Wide channel tiles leave few accumulator slots; blocks that begin with carried rows must not let an epilogue group take a slot's
second row for its first."""
import numpy as np
import pytest

from paper_1804_10727_b200 import idf
from paper_1804_10727_b200.workloads import conv, POOL
from helpers import assert_equal, rand_net, with_shifts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pool", [False, True])
@pytest.mark.parametrize("chunks", [[3] * 9, [4, 5, 6, 2, 7], [2, 9, 3, 8]])
def test_wide_channel_tiles_in_short_blocks(orc, pool, chunks):
    layers = with_shifts((conv(64, 128, 3, pad=1),) + ((POOL,) if pool else ()), 10)
    S, H, W = 500, sum(chunks), 30                               # 125 tiles of four streams: the widest channel tile is taken
    x, ws, bs = rand_net("i8", layers, H, W, 64, S=S, seed=len(chunks))
    pick = np.r_[0:8, 250, 499]
    want = orc.forward("i8", layers, x[pick], ws, bs)
    net = idf.Net("i8", layers, W, 64, S, ws, bs)
    got = idf.infer(net, x, chunks=chunks, last=True)
    assert all(t > 0 for t in net.status()[:1])
    assert_equal(got[pick], want)
    # ... and all streams against one push
    assert np.array_equal(got, idf.infer(net, x, last=True))
    net.close()
