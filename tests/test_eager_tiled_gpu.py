"""Tiled eager kernels against the plain ones (a thread per unit), push by push: rows of one and of several runs of 32 positions,
stream groups with a remainder, four and eight channels per thread, quads of input channels and single ones, pools on pools."""
import numpy as np
import pytest
import torch

from paper_1804_10727_b200 import idf
from paper_1804_10727_b200.workloads import conv, POOL
from helpers import rand_net, with_shifts

pytestmark = pytest.mark.gpu

CASES = [
    # (name, mode, layers, H, W, S)
    ("i8_classifier", "i8", (conv(1, 16, 3), conv(16, 32, 3), POOL, conv(32, 32, 3)), 20, 28, 7),
    ("i8_wide_rows", "i8", (conv(2, 8, 3, pad=1), conv(8, 12, 3, stride=2)), 13, 75, 3),
    ("i8_pool_on_pool", "i8", (conv(3, 8, 3, pad=1), POOL, POOL, conv(8, 8, 3)), 25, 37, 5),
    ("i8_k5", "i8", (conv(4, 16, 5, pad=2), conv(16, 4, 3, pad=1)), 14, 16, 33),
    ("f32_1d", "f32", (conv(1, 8, 3, one_d=True), conv(8, 8, 3, one_d=True), conv(8, 4, 3, one_d=True)), 40, 1, 70),
    ("f32_2d_pool", "f32", (conv(3, 8, 3, pad=1), POOL, conv(8, 12, 3)), 17, 23, 6),
    ("bf16_2d", "bf16", (conv(2, 8, 3), conv(8, 16, 3), POOL), 16, 40, 3),
]


@pytest.mark.parametrize("name,mode,layers,H,W,S", CASES, ids=[c[0] for c in CASES])
def test_tiled_kernels_equal_the_plain_ones(orc, debug_flags, name, mode, layers, H, W, S):
    if mode == "i8":
        layers = with_shifts(layers, 7)
    x, ws, bs = rand_net(mode, layers, H, W, layers[0].cin, S=S, seed=len(name), zero_frac=0.8)
    seg = idf.segments_from_maps(x, mode).cuda()
    # a segment buffer that starts on an odd element: the first layer must not rely on word alignment
    odd = torch.empty(seg.numel() + 1, dtype=seg.dtype, device="cuda")[1:].view(seg.shape)
    odd.copy_(seg)
    runs = []
    for flags, s in ((0, seg), (0, odd), (idf.DEBUG_NO_TILED_EAGER, seg)):
        debug_flags(flags)
        net = idf.Net(mode, layers, W, layers[0].cin, S, ws, bs, eager=True)
        out = net.alloc_out(H)
        net.open()
        snaps = []
        for r in range(H - 1):
            net.push(s[r:r + 1], out)
            snaps.append(out.clone())
        rows = net.push_last(s[H - 1:], out)
        snaps.append(out.clone())
        runs.append((torch.stack(snaps).cpu().numpy(), net.event_counts(), rows, net.launches))
        net.status()
        net.close()
    assert runs[0][3] < runs[2][3]                      # the tiled kernels ran: no launch of their own for the input
    for got, events, rows, _ in runs[:2]:
        assert rows == runs[2][2] and events == runs[2][1], name
        # the same sums in the same order (a fused multiply-add may round differently): int nets bit for bit
        if mode == "i8":
            assert np.array_equal(got, runs[2][0]), name
        else:
            assert np.allclose(got, runs[2][0], rtol=1e-5, atol=1e-5) or mode == "bf16" and np.abs(got - runs[2][0]).max() < 0.06, name
    # ... and the end of it is Eq. 1's result
    want = orc.forward(mode, layers, x, ws, bs)
    got = runs[0][0][-1][:, :runs[0][2]]
    assert np.array_equal(got, want) if mode == "i8" else np.abs(got - want).max() < (0.06 if mode == "bf16" else 1e-4 + 1e-3 * np.abs(want).max())
