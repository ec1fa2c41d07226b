"""One stream advanced by the per-layer tensor-core kernels and by the all-layers launch in turn: pushes of many rows take the
former, pushes of one or two rows of a small net the latter (the library's own choice).  A row that a push completes leaves its old
partial sum in its ring slot; the row that takes the slot next must not start from it, whichever launch begins it."""
import numpy as np
import pytest

from paper_1804_10727_b200 import idf, workloads
from paper_1804_10727_b200.workloads import conv, POOL
from helpers import assert_close, assert_equal, rand_net, with_shifts

pytestmark = [pytest.mark.gpu, pytest.mark.own_routing]


def c1(cin, cout, k, s=1, pad=0, path=0):
    return conv(cin, cout, k, s, pad, one_d=True, path=path)


CASES = [
    # (name, mode, layers, W, pushes)
    ("window_1d", "bf16", (c1(1, 32, 9),), 1, (20, 20, 1, 1, 13, 2, 30, 1, 2)),
    ("window_time_1d", "bf16", (c1(1, 16, 9), c1(16, 32, 9, 2), c1(32, 16, 5, 1, 2)), 1, (160, 1, 2, 160, 1, 1, 40, 2)),
    ("time_1d_i8", "i8", (c1(3, 16, 5, path=1), c1(16, 32, 9, 3, 4), c1(32, 16, 3, 1, 1)), 1, (40, 1, 2, 70, 1, 1, 33, 2, 1)),
    ("window_ring_pool_2d", "bf16", (conv(3, 16, 3, pad=1), conv(16, 32, 3, pad=1), POOL, conv(32, 16, 3)), 8, (5, 5, 1, 7, 1, 2, 6, 1)),
    ("window_ring_stride_2d", "bf16", (conv(3, 16, 3), conv(16, 32, 5, 2, 2)), 13, (5, 6, 1, 7, 2, 1, 6, 1, 1)),
    ("events_ring_pool_2d_i8", "i8", (conv(1, 16, 3), conv(16, 32, 3), POOL, conv(32, 32, 3)), 12, (5, 5, 1, 7, 1, 2, 6, 1)),
    ("ring_stride3_2d_i8", "i8", (conv(16, 16, 4, 3, 1), conv(16, 32, 3, 1, 1)), 13, (9, 8, 1, 1, 7, 2, 1, 12, 1)),
]


def _check(mode, n_conv, got, want, what):
    if mode == "i8":
        assert_equal(got, want, what)
    elif n_conv == 1:
        assert_close(got, want, what)                # fp32 output, no hidden rounding
    else:                                            # a hidden value that rounds to its other neighbour moves an output by 2^-8 of its size
        err = np.abs(got - want)
        assert (err <= 1e-4 + 1e-3 * np.abs(want)).mean() > 0.97 and err.max() < 2 ** -7 * np.abs(want).max(), (what, err.max(), np.abs(want).max())


@pytest.mark.parametrize("S", [1, 3])
@pytest.mark.parametrize("name,mode,layers,W,pushes", CASES, ids=[c[0] for c in CASES])
def test_routes_take_turns(orc, name, mode, layers, W, pushes, S):
    if mode == "i8":
        layers = with_shifts(layers, 8)
    H, n_conv = sum(pushes), sum(l.kind == "conv" for l in layers)
    x, ws, bs = rand_net(mode, layers, H, W, layers[0].cin, S=S, seed=len(name))
    want = orc.forward(mode, layers, x, ws, bs)
    for forced in (False, True):
        net = idf.Net(mode, layers, W, layers[0].cin, S, ws, bs)
        seg = idf.segments_from_maps(x, mode).cuda()
        out = net.alloc_out(H)
        net.open()
        pos = 0
        for i, n in enumerate(pushes):
            if forced:                               # every other push, whatever its size
                idf.set_debug_flags(idf.DEBUG_NO_FUSED if i % 2 == 0 else idf.DEBUG_FORCE_FUSED)
            before = net.launches
            (net.push_last if i + 1 == len(pushes) else net.push)(seg[pos:pos + n], out)
            assert forced or n > 1 or net.launches == before + 1                         # one row: the single launch, by itself
            pos += n
        idf.set_debug_flags(0)
        tc = net.status()
        assert all(t > 0 for t, l in zip(tc, layers) if l.kind == "conv"), tc            # both routes ran
        _check(mode, n_conv, out.cpu().numpy()[:, :want.shape[1]], want, f"{name}/S={S}/forced={forced}")
        net.close()


@pytest.mark.parametrize("pushes", [(5, 5, 1, 17), (10, 10, 1, 7), (5, 1, 5, 1, 1, 15)])
def test_one_mnist2d_stream(orc, pushes):
    w = workloads.get("mnist2d", n_streams=1)
    x = workloads.make_input(w)
    ws, bs = workloads.make_params(w)
    want = orc.forward(w.dtype, w.layers, x, ws, bs)
    net = idf.net_from_workload(w, ws, bs)
    assert_equal(idf.infer(net, x, chunks=list(pushes), last=True), want, f"mnist2d {pushes}")
    net.close()


@pytest.mark.parametrize("pushes", [(160, 160, 1, 2, 160), (200, 1, 1, 150)])
def test_one_audio1d_stream(orc, pushes):
    """(a one-sample push of the whole net is more work than the single launch takes by itself: forced)"""
    w = workloads.get("audio1d", n_streams=1, H=sum(pushes))
    x = workloads.make_input(w)
    ws, bs = workloads.make_params(w)
    want = orc.forward(w.dtype, w.layers, x, ws, bs)
    net = idf.net_from_workload(w, ws, bs)
    seg = idf.segments_from_maps(x, w.dtype).cuda()
    out = net.alloc_out(w.H)
    net.open()
    pos = 0
    for i, n in enumerate(pushes):
        idf.set_debug_flags(idf.DEBUG_FORCE_FUSED if n <= 2 else idf.DEBUG_NO_FUSED)
        (net.push_last if i + 1 == len(pushes) else net.push)(seg[pos:pos + n], out)
        pos += n
    idf.set_debug_flags(0)
    err = np.abs(out.cpu().numpy()[:, :want.shape[1]] - want)
    assert (err <= 1e-4 + 1e-3 * np.abs(want)).mean() > 0.9 and err.max() < 2 ** -7 * np.abs(want).max(), (err.max(), np.abs(want).max())
    net.close()
