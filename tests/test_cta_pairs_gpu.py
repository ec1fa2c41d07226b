"""Wide layers on CTA pairs (M = 256 tensor-core instructions over two CTAs): positions around the tile sizes (several streams to a tile,
one, several tiles to a row, an odd last tile), rows of an item and remainders, one and several K blocks, channel slices, blocks that
begin, continue and end streams (rows carried through the ring, also from its copy), pooled rows with pairs split across launches, odd
widths, rows that wait only for padding; the row-ring kernel gives the same bytes (int8)."""
import numpy as np
import pytest
import torch

from paper_1804_10727_b200 import idf
from paper_1804_10727_b200.workloads import Layer, conv, POOL
from helpers import assert_close, assert_equal, rand_net, with_shifts
from test_full_size_gpu import _bf16_down_up

pytestmark = pytest.mark.gpu


def rect(cin, cout, kh, kw, pad=0, relu=1):
    return Layer("conv", cin, cout, kh, kw, 1, pad, relu, 0, 0)


CASES = [
    # (name, mode, layers, H, W, S)
    ("bf16_64_64", "bf16", (conv(64, 64, 3, pad=1),), 19, 20, 13),
    ("bf16_128_256_one_position_tile", "bf16", (conv(128, 256, 3, pad=1),), 9, 126, 1),
    ("bf16_256_128_two_tiles_a_row", "bf16", (conv(256, 128, 3, pad=1),), 7, 130, 2),
    ("bf16_128_96", "bf16", (conv(128, 96, 3),), 12, 39, 5),                     # slices of 32
    ("bf16_64_64_k5", "bf16", (conv(64, 64, 5, pad=4),), 11, 24, 3),             # rows and columns of nothing but padding beside the map
    ("bf16_64_64_k5x2", "bf16", (rect(64, 64, 5, 2, 1, 0),), 14, 30, 2),
    ("bf16_pool_f32", "bf16", (conv(64, 64, 3, pad=1), POOL), 13, 30, 5),
    ("bf16_pool_odd", "bf16", (conv(128, 128, 3, pad=1), POOL), 18, 65, 3),      # odd width, one stream to a tile
    ("i8_64_64", "i8", (conv(64, 64, 3),), 15, 27, 9),                           # 64-byte positions
    ("i8_128_256", "i8", (conv(128, 256, 3, pad=1),), 10, 18, 7),
    ("i8_pool", "i8", (conv(128, 64, 3, pad=1), POOL), 17, 34, 4),
    ("i8_pool_odd_rows", "i8", (conv(64, 128, 3), POOL), 18, 131, 1),
]


@pytest.mark.parametrize("name,mode,layers,H,W,S", CASES, ids=[c[0] for c in CASES])
def test_cta_pairs_match_oracle(orc, debug_flags, name, mode, layers, H, W, S):
    layers = with_shifts(layers, 9) if mode == "i8" else layers
    x, ws, bs = rand_net(mode, layers, H, W, layers[0].cin, S=S, seed=len(name))
    want = orc.forward(mode, layers, x, ws, bs)
    check = assert_equal if mode == "i8" else assert_close                       # (one conv layer: fp32 output)
    debug_flags(idf.DEBUG_FORCE_CTA_PAIRS)
    for chunks, rb, last in ((None, 0, True), (None, 0, False), ([1] * H, 0, True), ([5, 1, 2], 0, True), ([H // 2], 4, False)):
        net = idf.Net(mode, layers, W, layers[0].cin, S, ws, bs, row_block=rb)
        got = idf.infer(net, x, chunks=chunks, last=last)
        assert net.pair_launches()[0] == net.status()[0] > 0                     # every launch that brings rows
        check(got, want, f"{name}/{chunks and len(chunks)}/{rb}/{last}")
        net.close()
    if mode == "i8":
        debug_flags(idf.DEBUG_NO_CTA_PAIRS)
        net = idf.Net(mode, layers, W, layers[0].cin, S, ws, bs)
        assert_equal(idf.infer(net, x, chunks=[4, 3], last=True), want, name + "/row ring")
        assert net.status()[0] > 0 and net.pair_launches()[0] == 0
        net.close()


@pytest.mark.parametrize("S", [72, 76])                                          # 144 and 152 tiles of the row-ring kernel: one turn of the SMs, two
def test_rows_one_by_one(orc, S):
    """The rule for launches of few rows, on both sides of its line."""
    layers = (conv(256, 256, 3, pad=1),)
    x, ws, bs = rand_net("bf16", layers, 6, 30, 256, S=S, seed=S)
    pick = np.r_[0:4, S - 1]
    want = orc.forward("bf16", layers, x[pick], ws, bs)
    net = idf.Net("bf16", layers, 30, 256, S, ws, bs)
    for chunks in ([1] * 6, [2, 3, 1], [4, 2], [6]):
        assert_close(idf.infer(net, x, chunks=chunks, last=True)[pick], want, f"{S}/{len(chunks)}")
        few = sum(n < 6 for n in chunks)
        assert net.pair_launches()[0] == len(chunks) - (few if S == 72 else 0) and net.status()[0] == len(chunks)
    net.close()


@pytest.mark.parametrize("cin,S,chunks", [(64, 296, (15, 16)), (64, 192, (7, 8)), (128, 140, (11, 12))])    # 148, 96 and 140 tiles: full turns and not
def test_rows_in_one_turn(orc, cin, S, chunks):
    """The rule where the row-ring kernel takes a launch in one turn of the SMs, on both sides of its line."""
    layers = (conv(cin, 128, 3, pad=1),)
    x, ws, bs = rand_net("bf16", layers, sum(chunks), 30, cin, S=S, seed=S)
    pick = np.r_[0:3, S - 1]
    net = idf.Net("bf16", layers, 30, cin, S, ws, bs)
    assert_close(idf.infer(net, x, chunks=chunks, last=True)[pick], orc.forward("bf16", layers, x[pick], ws, bs), f"{cin}/{S}")
    assert net.pair_launches() == [1] and net.status() == [2]
    net.close()


def test_hidden_rows(orc, debug_flags):
    """bf16 rows between layers, emitted and pooled by pairs: against the row-ring kernels, off by one rounding (2^-8 of the value; the
    sums of the next layer average that out, so twice it over the largest output bounds them)."""
    layers = (conv(64, 128, 3, pad=1), POOL, conv(128, 128, 3, pad=1), conv(128, 64, 3, pad=1), POOL)
    x, ws, bs = rand_net("bf16", layers, 24, 40, 64, S=6, seed=3)
    outs = []
    for flags in (idf.DEBUG_FORCE_CTA_PAIRS, idf.DEBUG_NO_CTA_PAIRS):
        debug_flags(flags)
        net = idf.Net("bf16", layers, 40, 64, 6, ws, bs)
        outs.append([])
        for c in (None, [1] * 24, [7, 2, 9]):
            outs[-1].append(idf.infer(net, x, chunks=c, last=True))
            tc, pairs = net.status(), net.pair_launches()
            assert all(tc[i] > 0 and pairs[i] == (tc[i] if flags == idf.DEBUG_FORCE_CTA_PAIRS else 0) for i in (0, 2, 3)), (flags, c, tc, pairs)
        net.close()
    for got, want in zip(*outs):
        assert np.abs(got - want).max() <= 2.0 ** -7 * np.abs(want).max()


@pytest.mark.parametrize("push", [14, 36, 40])
def test_pool_rows_taken_and_parked_in_one_launch(debug_flags, push):
    """Launches that begin with a pair's second row and end with a pair's first (rows [35, 71), [71, 107)): the row an earlier launch left in
    the pool state and the one parked there belong to different clusters, in no order; with shares that straddle columns of work the parking
    cluster comes first.  The row-ring kernel gives the same bytes, every time."""
    layers = with_shifts((conv(128, 128, 3, pad=1), POOL), 12)
    S, H, W = 64, 112, 112
    g = torch.Generator(device="cuda").manual_seed(push)
    seg = torch.randint(-127, 128, (H, S, W, 128), generator=g, device="cuda", dtype=torch.int8)
    _, ws, bs = rand_net("i8", layers, 1, 1, 128, S=1, seed=push)
    net = idf.Net("i8", layers, W, 128, S, ws, bs)
    net.open()
    outs = []
    for rep in range(11):
        debug_flags(idf.DEBUG_NO_CTA_PAIRS if rep == 0 else idf.DEBUG_FORCE_CTA_PAIRS if push < 16 else 0)
        out = net.alloc_out(H)
        net.reset()
        for r in range(0, H - push, push):
            net.push(seg[r:r + push], out)
        r = (H - 1) // push * push
        net.push_last(seg[r:], out)
        net.status()
        assert (net.pair_launches()[0] > 0) == (rep > 0)
        outs.append(out)
        assert torch.equal(out, outs[0]), f"{push} rows a push, run {rep}: {int((out != outs[0]).sum())} of {out.numel()} differ"
    assert int(outs[0].ne(0).sum()) > outs[0].numel() // 4
    net.close()


def test_hidden_rows_match_oracle(orc, debug_flags):
    """Rows between layers, emitted and pooled by pairs, against the oracle: int8 nets exactly; a bf16 layer's rounded rows, passed on by a 1x1
    identity layer, are the rounding of some value within the strict tolerance of the oracle's unrounded one."""
    debug_flags(idf.DEBUG_FORCE_CTA_PAIRS)
    layers = with_shifts((conv(128, 128, 3, pad=1), POOL, conv(128, 256, 3, pad=1), conv(256, 64, 3, pad=1), POOL), 11)
    x, ws, bs = rand_net("i8", layers, 24, 40, 128, S=6, seed=3)
    want = orc.forward("i8", layers, x, ws, bs)
    net = idf.Net("i8", layers, 40, 128, 6, ws, bs)
    for chunks in (None, [1] * 24, [7, 2, 9]):
        assert_equal(idf.infer(net, x, chunks=chunks, last=True), want, f"i8/{chunks and len(chunks)}")
        assert all(net.pair_launches()[i] > 0 for i in (0, 2, 3))
    net.close()
    for layer, pool in ((conv(64, 128, 3, pad=1), False), (conv(128, 128, 3, pad=1, relu=0), True), (conv(128, 64, 5), True)):
        layers = (layer,) + ((POOL,) if pool else ()) + (conv(layer.cout, layer.cout, 1, relu=0),)
        x, ws, bs = rand_net("bf16", layers, 17, 34, layer.cin, S=5, seed=layer.cin + layer.cout)
        ws[-1], bs[-1] = np.eye(layer.cout, dtype=np.float32).reshape(layer.cout, 1, 1, layer.cout), None
        want = orc.conv_layer("bf16", layer, x, ws[0], bs[0])
        want = orc.pool_layer("bf16", want) if pool else want
        tol = 1e-4 + 1e-3 * np.abs(want)
        lo, hi = _bf16_down_up(want - tol)[0], _bf16_down_up(want + tol)[1]
        net = idf.Net("bf16", layers, 34, layer.cin, 5, ws, bs)
        for chunks in (None, [1] * 17, [7, 2, 3]):
            got = idf.infer(net, x, chunks=chunks, last=True).astype(np.float64)
            assert net.pair_launches()[0] > 0 and got.shape == want.shape
            bad = (got < lo) | (got > hi)
            assert not bad.any(), (layer, pool, chunks, int(bad.sum()), bad.size)
        net.close()


def test_slow_kernel_in_front(orc):
    """A layer whose events are scattered one by one takes long over an input without zeros; the launch that depends on it starts early and must
    not give up meanwhile."""
    layers = with_shifts((Layer("conv", 128, 256, 4, 4, 1, 0, 1, 0, idf.PATH_SPARSE), conv(256, 128, 3, pad=1)), 11)
    x, ws, bs = rand_net("i8", layers, 20, 68, 128, S=1, seed=9, zero_frac=0.0)
    net = idf.Net("i8", layers, 68, 128, 1, ws, bs, row_block=16)
    assert_equal(idf.infer(net, x, last=True), orc.forward("i8", layers, x, ws, bs), "slow first layer")
    assert net.pair_launches()[1] > 0
    net.close()
