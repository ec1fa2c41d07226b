"""Pooling folded into the emission of rows of odd width: tiles get an even number of positions, the last column has no partner."""
import numpy as np
import pytest

from paper_1804_10727_b200 import idf
from paper_1804_10727_b200.workloads import conv, POOL
from helpers import assert_close, assert_equal, rand_net, with_shifts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [39, 63, 127, 129, 157])           # several streams to a tile, one, two tiles to a row
@pytest.mark.parametrize("mode,cin", [("i8", 16), ("i8", 64), ("bf16", 32)])
def test_pooled_rows_of_odd_width(orc, mode, cin, W):
    layers = (conv(cin, 32, 3, pad=1), POOL)
    if mode == "i8":
        layers = with_shifts(layers, 8)
    S, chunks = 7, [1, 2, 9, 1, 6]
    x, ws, bs = rand_net(mode, layers, sum(chunks), W, cin, S=S, seed=W)
    want = orc.forward(mode, layers, x, ws, bs)
    for c in (chunks, None):
        net = idf.Net(mode, layers, W, cin, S, ws, bs)
        got = idf.infer(net, x, chunks=c, last=True)
        assert net.status()[0] > 0 and net.status()[1] == 0
        (assert_equal if mode == "i8" else assert_close)(got, want, f"{mode}/{W}/{c}")
        net.close()
