"""Infinities and NaN in bf16 input reach the outputs whose receptive field holds them, and no others: tensor-core layers that take
several positions as one must not let a zero weight meet them."""
import numpy as np
import pytest

from paper_1804_10727_b200 import idf
from paper_1804_10727_b200.workloads import conv
from helpers import assert_close, rand_net

pytestmark = pytest.mark.gpu

CASES = [
    # (name, layer, H, W, S)
    ("8ch_3x3", conv(8, 32, 3, pad=1, relu=0), 9, 21, 5),                    # 16-byte positions, an odd number of taps
    ("8ch_5x5", conv(8, 16, 5, pad=2, relu=0), 9, 12, 3),
    ("8ch_4x4", conv(8, 16, 4, pad=1, relu=0), 9, 15, 3),                    # an even one: pairs without zero weights
    ("32ch_stride2_pad", conv(32, 32, 3, stride=2, pad=1, relu=0), 12, 38, 5),
    ("16ch_stride2", conv(16, 32, 3, stride=2, relu=0), 12, 40, 4),
    ("32ch_stride2_even", conv(32, 32, 2, stride=2, relu=0), 12, 40, 4),
    ("32ch_3x3", conv(32, 32, 3, pad=1, relu=0), 9, 21, 5),
]


@pytest.mark.parametrize("name,layer,H,W,S", CASES, ids=[c[0] for c in CASES])
def test_nonfinite_input_stays_in_its_receptive_field(orc, name, layer, H, W, S):
    layers = (layer,)
    for k, value in enumerate((np.inf, -np.inf, np.nan)):
        x, ws, bs = rand_net("bf16", layers, H, W, layer.cin, S=S, seed=k)
        r = np.random.default_rng(k)
        for s in {0, S // 2, S - 1}:                                         # edges and inner positions, even and odd
            for row, col in ((0, 0), (H // 2, W // 2), (H // 2 + 1, max(W // 2 - 3, 0)), (H - 1, W - 1)):
                if r.random() < 0.7:
                    x[s, row, col, r.integers(layer.cin)] = value
        want = orc.forward("bf16", layers, x, ws, bs)
        fine = np.isfinite(want)
        assert not fine.all() and fine.any()
        for chunks in (None, [1] * H, [4, 2, H]):
            net = idf.Net("bf16", layers, W, layer.cin, S, ws, bs)
            got = idf.infer(net, x, chunks=chunks, last=True)
            assert net.status()[0] > 0
            what = f"{name}/{value}/{chunks and len(chunks)}"
            assert np.isfinite(got[fine]).all(), (what, np.count_nonzero(~np.isfinite(got[fine])))
            assert_close(np.where(fine, got, 0), np.where(fine, want, 0), what)
            np.testing.assert_array_equal(got[~fine], want[~fine], what)
            net.close()
