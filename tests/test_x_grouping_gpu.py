"""Tensor-core layers whose input positions are taken in groups: 16-byte positions two to a K step, x-strided layers with a
stride's worth of positions as one; kx taps of 32- and 64-byte rows read row-shifted from one box.  Tile edges, odd widths, pools."""
import numpy as np
import pytest

from paper_1804_10727_b200 import idf
from paper_1804_10727_b200.workloads import conv, POOL
from helpers import assert_close, assert_equal, rand_net, with_shifts

pytestmark = pytest.mark.gpu

CASES = [
    # (name, mode, layers, H, W, S)
    ("bf16_8ch_pairs", "bf16", (conv(8, 32, 3, pad=1),), 9, 21, 5),
    ("i8_16ch_pairs_two_tiles", "i8", (conv(16, 32, 3, pad=1), POOL), 8, 134, 2),
    ("i8_16ch_pairs_exact_tile", "i8", (conv(16, 16, 3),), 7, 127, 2),               # 125 outputs and three halo positions
    ("i8_16ch_k5_pairs", "i8", (conv(16, 32, 5, pad=2),), 11, 9, 40),
    ("i8_16ch_1x1", "i8", (conv(16, 32, 1),), 5, 17, 9),
    ("i8_stride2_even", "i8", (conv(32, 64, 3, stride=2),), 13, 254, 2),
    ("i8_stride2_odd_second_layer", "i8", (conv(16, 32, 3), conv(32, 64, 3, stride=2), POOL), 19, 57, 4),   # the last group spills
    ("i8_stride2_pad_odd", "i8", (conv(16, 32, 3), conv(32, 32, 3, stride=2, pad=1)), 14, 41, 3),           # right padding: no groups
    ("bf16_stride2_pad", "bf16", (conv(32, 32, 3, stride=2, pad=1),), 12, 38, 5),
    ("i8_stride3", "i8", (conv(64, 32, 4, stride=3),), 17, 33, 6),
    ("i8_64ch_shifted", "i8", (conv(64, 64, 3, pad=1), POOL), 10, 126, 3),
    ("i8_16ch_pairs_pool_packed", "i8", (conv(16, 32, 3, pad=1), POOL), 9, 26, 7),
    ("bf16_64ch_even_kernel_pool", "bf16", (conv(64, 16, 4, pad=1), POOL), 11, 21, 9),      # odd halo: streams start on odd lanes
    ("i8_32ch_packed_streams", "i8", (conv(32, 32, 3),), 9, 12, 100),
]


@pytest.mark.parametrize("name,mode,layers,H,W,S", CASES, ids=[c[0] for c in CASES])
def test_grouped_positions_match_oracle(orc, name, mode, layers, H, W, S):
    if mode == "i8":
        layers = with_shifts(layers, 9)
    x, ws, bs = rand_net(mode, layers, H, W, layers[0].cin, S=S, seed=len(name))
    want = orc.forward(mode, layers, x, ws, bs)
    for chunks, rb in ((None, 0), ([1] * H, 0), ([3, 2, 5], 3)):
        net = idf.Net(mode, layers, W, layers[0].cin, S, ws, bs, row_block=rb)
        got = idf.infer(net, x, chunks=chunks, last=rb == 0)
        tc = net.status()
        assert all(t > 0 for t, l in zip(tc, layers) if l.kind == "conv"), (name, tc)
        (assert_equal if mode == "i8" else assert_close)(got, want, f"{name}/{chunks and len(chunks)}/{rb}")
        net.close()
