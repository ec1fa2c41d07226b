"""Window kernel (thin layers): window widths from one output to a whole instruction, runs of every compiled length and the
general form, ragged last windows and tiles, blocks that begin, continue and end streams, event counts."""
import numpy as np
import pytest

from paper_1804_10727_b200 import idf
from paper_1804_10727_b200.workloads import conv
from helpers import assert_close, assert_equal, rand_net, with_shifts

pytestmark = pytest.mark.gpu

CASES = [
    # (name, mode, layers, H, W, S): the first layer takes the window kernel
    ("bf16_rgb_9_words", "bf16", (conv(3, 64, 3, pad=1),), 6, 224, 64),             # four outputs per window, four K steps
    ("bf16_rgb_one_output", "bf16", (conv(3, 64, 3, pad=1),), 7, 37, 3),
    ("i8_polarity_wide", "i8", (conv(2, 32, 3), conv(32, 32, 3)), 9, 61, 850),      # eight outputs; last window of three
    ("i8_grey_13_outputs", "i8", (conv(1, 16, 3),), 8, 28, 3200),                   # 208 columns: half a chunk of 32
    ("i8_48_channels", "i8", (conv(1, 48, 3, relu=0),), 7, 130, 130),               # 32 columns straddle two outputs
    ("i8_5x5_general_runs", "i8", (conv(4, 32, 5, pad=2), conv(32, 16, 3)), 13, 30, 5),
    ("bf16_5x5_stride2", "bf16", (conv(2, 32, 5, stride=2, pad=2),), 16, 33, 4),
    ("i8_stride2_dense", "i8", (conv(3, 32, 3, stride=2, pad=1, path=1),), 12, 51, 3),
    ("bf16_1d_stride2", "bf16", (conv(1, 32, 9, stride=2, one_d=True),), 203, 1, 1030),
    ("bf16_1d_few", "bf16", (conv(2, 48, 5, pad=2, one_d=True),), 50, 1, 3),
    ("bf16_1d_all_exchange", "bf16", (conv(1, 128, 9, one_d=True),), 64, 1, 19),    # short blocks: every row meets the ring, carried ones from a copy
    ("i8_1d_all_exchange", "i8", (conv(8, 96, 9, pad=4, one_d=True),), 64, 1, 14),
    ("bf16_5x5_all_exchange", "bf16", (conv(2, 32, 5, pad=2),), 24, 27, 40),
    ("i8_1d", "i8", (conv(3, 16, 9, stride=3, one_d=True, path=1),), 100, 1, 140),
]


@pytest.mark.parametrize("name,mode,layers,H,W,S", CASES, ids=[c[0] for c in CASES])
def test_window_kernel_matches_oracle(orc, name, mode, layers, H, W, S):
    if mode == "i8":
        layers = with_shifts(layers, 8)
    x, ws, bs = rand_net(mode, layers, H, W, layers[0].cin, S=S, seed=len(name), bias="48" in name or "1d" in name, zero_frac=0.9)
    pick = np.unique(np.r_[0, 1 % S, S // 2, S - 1])                                # streams the oracle recomputes
    want = orc.forward(mode, layers, x[pick], ws, bs)
    first = None
    for chunks, rb, last in ((None, 0, True), ([1] * H, 0, True), ([H // 2 + 1], 0, False), ([4, 2, 7], 3, True)):
        net = idf.Net(mode, layers, W, layers[0].cin, S, ws, bs, row_block=rb)
        got = idf.infer(net, x, chunks=chunks, last=last)
        tc = net.status()
        what = f"{name}/{chunks and len(chunks)}/{rb}"
        assert tc[0] > 0, what
        if mode == "i8":
            assert_equal(got[pick], want, what)
            first = got if first is None else first
            assert np.array_equal(got, first), what
        else:
            assert_close(got[pick], want, what)                                     # one layer: fp32 output, no hidden rounding
        if mode == "i8" and W > 1 and layers[0].path == 0:
            assert net.event_counts()[0] == int((x != 0).sum()), what
        net.close()
