"""1D layers on the kernel that tiles time x streams: row counts around the tile sizes (16 rows an M tile, 64 an item), strides, ragged
stream groups, weight tiles resident and streamed, one and several K blocks, channel counts with odd slices, blocks that begin,
continue and end streams (rows carried through the ring), in one item per stream group and in many."""
import numpy as np
import pytest

from paper_1804_10727_b200 import idf
from paper_1804_10727_b200.workloads import Layer, conv
from helpers import assert_close, assert_equal, rand_net, with_shifts

pytestmark = pytest.mark.gpu


def c1(cin, cout, k, s=1, pad=0, relu=1):
    return conv(cin, cout, k, s, pad, one_d=True, relu=relu)


CASES = [
    # (name, mode, layer, H, S)
    ("bf16_128_128_k9", "bf16", c1(128, 128, 9), 150, 11),
    ("bf16_64_128_k9", "bf16", c1(64, 128, 9), 72, 8),            # exactly 64 output rows
    ("bf16_32_64_s2", "bf16", c1(32, 64, 9, 2), 139, 3),          # 66 rows: one item and a bit
    ("bf16_64_64_s2_pad", "bf16", c1(64, 64, 9, 2, 4), 64, 17),
    ("bf16_16_16_k3", "bf16", c1(16, 16, 3), 18, 1),
    ("bf16_256_256", "bf16", c1(256, 256, 5), 40, 9),             # four K blocks, two channel slices
    ("bf16_32_96_s3", "bf16", c1(32, 96, 7, 3, 2, 0), 100, 20),
    ("i8_64_128", "i8", c1(64, 128, 9), 100, 10),
    ("i8_128_80", "i8", c1(128, 80, 3, 1, 1, 0), 65, 5),
    ("i8_32_144_s4", "i8", c1(32, 144, 9, 4), 130, 6),            # channel slices of 16
    ("i8_64_96", "i8", c1(64, 96, 5), 77, 4),                     # slices of 48, some of them between 32-byte boundaries
    ("i8_64_96_many", "i8", c1(64, 96, 3, 1, 1), 100, 820),       # slices of 96, also in shares of 48
    ("i8_32_160", "i8", c1(32, 160, 3, 1, 1), 80, 9),             # of 80
    ("i8_32_192", "i8", c1(32, 192, 3, 1, 1, 0), 66, 7),          # of 96 and 48
    ("i8_32_224", "i8", c1(32, 224, 5, 2, 2), 140, 5),            # of 112
]


@pytest.mark.parametrize("name,mode,layer,H,S", CASES, ids=[c[0] for c in CASES])
def test_time_tiles_match_oracle(orc, debug_flags, name, mode, layer, H, S):
    layers = with_shifts((layer,), 9) if mode == "i8" else (layer,)
    x, ws, bs = rand_net(mode, layers, H, 1, layer.cin, S=S, seed=len(name))
    want = orc.forward(mode, layers, x, ws, bs)
    check = assert_equal if mode == "i8" else assert_close           # (one layer: fp32 output)
    for chunks, rb, last in ((None, 0, True), (None, 0, False), ([1] * H, 0, True), ([17, 33, 5, 1, 29], 0, True), ([H // 2], 24, False)):
        net = idf.Net(mode, layers, 1, layer.cin, S, ws, bs, row_block=rb)
        got = idf.infer(net, x, chunks=chunks, last=last)
        assert net.status()[0] > 0
        check(got, want, f"{name}/{chunks and len(chunks)}/{rb}/{last}")
        net.close()
    if mode == "i8":
        debug_flags(idf.DEBUG_NO_TIME_TILES)                         # the row-ring kernel gives the same bytes
        net = idf.Net(mode, layers, 1, layer.cin, S, ws, bs)
        assert_equal(idf.infer(net, x, chunks=[40, 3], last=True), want, name + "/row ring")
        net.close()


def test_slow_kernel_in_front(orc):
    """A layer whose events are scattered one by one takes long over an input without zeros (0.7 s here); the launch that depends on it starts
    early and must not give up meanwhile, though its weight tiles do not all fit."""
    layers = with_shifts((Layer("conv", 512, 512, 9, 1, 1, 0, 1, 0, idf.PATH_SPARSE), conv(512, 256, 9, one_d=True)), 12)
    x, ws, bs = rand_net("i8", layers, 190, 1, 512, S=1, seed=9, zero_frac=0.0)
    net = idf.Net("i8", layers, 1, 512, 1, ws, bs, row_block=256)
    assert_equal(idf.infer(net, x, last=True), orc.forward("i8", layers, x, ws, bs), "slow first layer")
    assert net.status()[1] > 0
    net.close()
