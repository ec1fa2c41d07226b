"""Row-ring kernel with two CTAs on an SM: layers of more (position, channel) tiles than there are SMs, on both sides of that line."""
import numpy as np
import pytest

from paper_1804_10727_b200 import idf
from paper_1804_10727_b200.workloads import conv, POOL
from helpers import assert_equal, rand_net, with_shifts

pytestmark = pytest.mark.gpu

LAYERS = {
    "i8_pair_pool": ("i8", 16, (conv(16, 32, 3), POOL)),
    "i8_stride2": ("i8", 32, (conv(32, 64, 3, 2),)),
    "i8_64_to_32": ("i8", 64, (conv(64, 32, 3, pad=1),)),
    "bf16_pool": ("bf16", 32, (conv(32, 32, 3, pad=1), POOL)),
}


@pytest.mark.parametrize("S", [592, 600])                        # 148 and 150 tiles of four streams
@pytest.mark.parametrize("name", sorted(LAYERS))
def test_two_ctas_per_sm(orc, name, S):
    mode, cin, layers = LAYERS[name]
    layers = with_shifts(layers, 9)
    W, chunks = (59 if "stride2" in name else 32 if "pair" not in name else 34), [1, 1, 7, 2, 10]
    x, ws, bs = rand_net(mode, layers, sum(chunks), W, cin, S=S, seed=S)
    pick = np.r_[0:8, 250, S - 1]
    want = orc.forward(mode, layers, x[pick], ws, bs)
    net = idf.Net(mode, layers, W, cin, S, ws, bs)
    got = idf.infer(net, x, chunks=chunks, last=True)
    assert net.status()[0] > 0
    whole = idf.infer(net, x, last=True)                         # every stream, in one push: other row counts per launch
    if mode == "i8":
        assert_equal(got[pick], want)
        assert np.array_equal(got, whole)
    else:                                                        # a bf16 result is off by one rounding, 2^-8 of its size
        np.testing.assert_allclose(got[pick], want, rtol=2 ** -7, atol=2 ** -8 * np.abs(want).max())
        np.testing.assert_allclose(got, whole, rtol=2 ** -7, atol=2 ** -8 * np.abs(want).max())
    net.close()
