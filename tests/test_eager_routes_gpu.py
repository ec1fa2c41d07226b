"""Eager emission: which nets take the tiled kernel (one launch per push) and which the plain ones (a launch per layer and one for
the input), on both sides of the line, against the oracle."""
import numpy as np
import pytest

from paper_1804_10727_b200 import idf
from paper_1804_10727_b200.workloads import conv, POOL
from helpers import assert_close, assert_equal, rand_net, with_shifts

pytestmark = pytest.mark.gpu

CASES = [
    # (name, mode, layers, H, W, S, tiled)
    ("few_streams_wide_rows", "bf16", (conv(2, 128, 3, pad=1),), 6, 224, 4, False),
    ("few_streams_wide_rows_pool", "f32", (conv(16, 96, 3, pad=1), POOL), 6, 115, 3, False),
    ("one_d_many_channels", "i8", (conv(3, 128, 9, one_d=True),), 20, 1, 64, False),
    ("one_d_narrow", "f32", (conv(1, 8, 3, one_d=True), conv(8, 8, 3, one_d=True)), 20, 1, 5, True),
    ("classifier", "i8", (conv(1, 16, 3), conv(16, 32, 3), POOL), 12, 28, 300, True),
]


@pytest.mark.parametrize("name,mode,layers,H,W,S,tiled", CASES, ids=[c[0] for c in CASES])
def test_eager_route(orc, name, mode, layers, H, W, S, tiled):
    if mode == "i8":
        layers = with_shifts(layers, 8)
    x, ws, bs = rand_net(mode, layers, H, W, layers[0].cin, S=S, seed=len(name))
    net = idf.Net(mode, layers, W, layers[0].cin, S, ws, bs, eager=True)
    seg = idf.segments_from_maps(x, mode).cuda()
    out = net.alloc_out(H)
    net.open()
    for r in range(H - 1):
        net.push(seg[r:r + 1], out)
    assert net.launches == (H - 1) * (1 if tiled else len(layers) + 1), net.launches
    rows = net.push_last(seg[H - 1:], out)
    net.status()
    pick = np.unique(np.r_[0, S // 2, S - 1])
    (assert_equal if mode == "i8" else assert_close)(out[:, :rows].cpu().numpy()[pick], orc.forward(mode, layers, x[pick], ws, bs), name)
    net.close()
