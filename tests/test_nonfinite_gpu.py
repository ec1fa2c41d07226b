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
    ("window_rgb", conv(3, 64, 3, pad=1, relu=0), 9, 60, 70),                # windows of one to eight outputs
    ("window_rgb_one_output", conv(3, 64, 3, pad=1, relu=0), 7, 37, 3),
    ("window_1ch_wide", conv(1, 16, 3, relu=0), 8, 61, 900),                 # 16 channels: two outputs to a piece of 32 columns
    ("window_48", conv(2, 48, 3, relu=0), 7, 90, 300),                       # pieces that straddle two outputs
    ("window_5x5_stride2", conv(2, 32, 5, stride=2, pad=2, relu=0), 16, 33, 4),
    ("window_1d", conv(1, 32, 9, one_d=True, relu=0), 203, 1, 130),
    ("window_1d_stride2", conv(1, 32, 9, stride=2, one_d=True, relu=0), 203, 1, 1030),
    ("time_1d", conv(32, 32, 9, one_d=True, relu=0), 120, 1, 20),            # shifted views of whole rows: no zero weights
    ("time_1d_stride2_pad", conv(64, 32, 9, stride=2, pad=4, one_d=True, relu=0), 120, 1, 20),
    ("window_1d_pad", conv(2, 48, 5, pad=2, one_d=True, relu=0), 50, 1, 3),
    ("pairs_128ch", conv(64, 128, 3, pad=1, relu=0), 11, 22, 7),             # several streams to a tile, halos between them
    ("pairs_two_k_blocks_5x5", conv(128, 64, 5, pad=4, relu=0), 10, 37, 3),
    ("pairs_two_tiles_a_row", conv(64, 64, 3, relu=0), 9, 133, 2),
]


@pytest.mark.parametrize("name,layer,H,W,S", CASES, ids=[c[0] for c in CASES])
def test_nonfinite_input_stays_in_its_receptive_field(orc, debug_flags, name, layer, H, W, S):
    layers = (layer,)
    pairs = name.startswith("pairs")
    debug_flags(idf.DEBUG_FORCE_CTA_PAIRS if pairs else 0)
    for k, value in enumerate((np.inf, -np.inf, np.nan)):
        x, ws, bs = rand_net("bf16", layers, H, W, layer.cin, S=S, seed=k)
        r = np.random.default_rng(k)
        pick = sorted({0, S // 2, S - 1})                                    # streams the oracle recomputes
        for s in pick:                                                       # edges and inner positions, even and odd
            for row, col in ((0, 0), (H // 2, W // 2), (H // 3, max(W // 2 - 3, 0)), (H - 1, W - 1)):
                if r.random() < 0.7:
                    x[s, row, col, r.integers(layer.cin)] = value
        want = orc.forward("bf16", layers, x[pick], ws, bs)
        fine = np.isfinite(want)
        assert not fine.all() and fine.any()
        for chunks in (None, [1] * H, [4, 2, H]):
            net = idf.Net("bf16", layers, W, layer.cin, S, ws, bs)
            whole = idf.infer(net, x, chunks=chunks, last=True)
            assert net.status()[0] > 0 and (not pairs or net.pair_launches()[0] > 0)
            got = whole[pick]
            assert np.isfinite(np.delete(whole, pick, 0)).all()
            what = f"{name}/{value}/{chunks and len(chunks)}"
            assert np.isfinite(got[fine]).all(), (what, np.count_nonzero(~np.isfinite(got[fine])))
            assert_close(np.where(fine, got, 0), np.where(fine, want, 0), what)
            np.testing.assert_array_equal(got[~fine], want[~fine], what)
            net.close()
