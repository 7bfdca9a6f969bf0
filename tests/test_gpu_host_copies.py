"""Layers on host buffers: the rows go through in pieces whose copies and compute overlap.  The bits are those of one pass
over device buffers: every row is computed by itself, with the same integers and the same roundings."""
import threading

import numpy as np
import pytest
import torch

from paper_2203_15952_b200 import binding as aqt

pytestmark = pytest.mark.gpu

D, FF = 512, 2048


def _weights():
    g = torch.Generator(device="cuda").manual_seed(5)
    w1 = torch.randint(-7, 8, (FF, D), generator=g, device="cuda", dtype=torch.int8)
    w2 = torch.randint(-7, 8, (D, FF), generator=g, device="cuda", dtype=torch.int8)
    return w1, torch.rand(FF, generator=g, device="cuda") * 1e-2, w2, torch.rand(D, generator=g, device="cuda") * 1e-2


def _ffn(w, x, y, ws, stream=None):
    aqt.aqt_ffn_fwd(x, w[0], w[1], aqt.BITS_4_UNPACKED, w[2], w[3], aqt.BITS_4_UNPACKED, y, ws, stream=stream)


def _ws(M):
    return torch.empty(aqt.aqt_workspace_bytes(aqt.OP_FFN_FWD, M, FF, D, 8, 4), dtype=torch.uint8, device="cuda")


# up to 9 rows of 2 KB the one-launch form reads x in place, up to 112 it writes y in place; 976 rows are the last size that
# goes whole with x read in place, 977 the first in two pieces; 6145: a last piece of one row
@pytest.mark.parametrize("M,pinned", [(1, True), (9, True), (10, True), (112, True), (112, False), (113, True), (976, True), (977, True), (1025, True), (6145, True), (12800, True), (60001, True), (6145, False)])
def test_ffn_pieces_give_the_bits_of_one_pass(M, pinned):
    w = _weights()
    x = torch.randn(M, D)
    ref = torch.empty(M, D, device="cuda")
    _ffn(w, x.cuda(), ref, _ws(M))
    xh, yh = (x.pin_memory(), torch.full((M, D), float("nan")).pin_memory()) if pinned else (x, torch.full((M, D), float("nan")))
    ws = _ws(M)
    for _ in range(3):  # back to back on one stream: each call's copies wait for the one before
        _ffn(w, xh, yh, ws)
    torch.cuda.synchronize()
    assert aqt.aqt_device_status() == 0
    assert np.array_equal(yh.numpy().view(np.uint32), ref.cpu().numpy().view(np.uint32))
    # one side on the device
    yd = torch.empty(M, D, device="cuda")
    _ffn(w, xh, yd, ws)
    yh.fill_(float("nan"))
    _ffn(w, x.cuda(), yh, ws)
    torch.cuda.synchronize()
    assert torch.equal(yd, ref) and torch.equal(yh, ref.cpu())


@pytest.mark.parametrize("M", [3, 40, 300, 2000])
def test_ffn_on_parts_of_pinned_buffers(M):
    """Rows from the middle and from the very end of a pinned allocation, read and written in place or copied; the rows around
    them stay as they are."""
    w, total = _weights(), 4096  # 8 MB: the end of the tensor is the end of the allocation
    x, y = torch.randn(total, D).pin_memory(), torch.full((total, D), 7.0).pin_memory()
    ref = torch.empty(M, D, device="cuda")
    for r0 in (0, 17, total - M):
        _ffn(w, x[r0:r0 + M].cuda(), ref, _ws(M))
        y.fill_(7.0)
        _ffn(w, x[r0:r0 + M], y[r0:r0 + M], _ws(M))
        torch.cuda.synchronize()
        assert torch.equal(y[r0:r0 + M], ref.cpu())
        assert bool((y[:r0] == 7.0).all()) and bool((y[r0 + M:] == 7.0).all())
    assert aqt.aqt_device_status() == 0


@pytest.mark.parametrize("scale", [aqt.SCALE_ROW, aqt.SCALE_TENSOR])
def test_linear_host_pieces(scale):
    M, N = 5000, 256
    w = _weights()
    wq, s_w = w[0][:N].contiguous(), w[1][:N].contiguous()
    x = torch.randn(M, D)
    ref = aqt.aqt_linear_fwd(x.cuda(), wq, s_w, a_scale_kind=scale)
    yh = torch.full((M, N), float("nan")).pin_memory()
    ws = torch.empty(aqt.aqt_workspace_bytes(aqt.OP_LINEAR_FWD, M, N, D, 8, 8) + 256 + 4 * M * (D + N) + 512, dtype=torch.uint8, device="cuda")
    aqt.aqt_linear_fwd_host(x.pin_memory(), wq, s_w, None, yh, ws, a_scale_kind=scale)
    torch.cuda.synchronize()
    assert torch.equal(yh, ref.cpu())


def test_ffn_host_from_several_threads_and_streams():
    """More streams than there are pairs of side streams, one thread each, every call with input of its own."""
    M, calls = 4000, 4
    w = _weights()
    xs = [torch.randn(M, D).pin_memory() for _ in range(6)]
    refs = []
    for x in xs:
        y = torch.empty(M, D, device="cuda")
        _ffn(w, x.cuda(), y, _ws(M))
        refs.append(y.cpu())
    torch.cuda.synchronize()
    bad = []

    def work(i):
        s, y, ws = torch.cuda.Stream(), torch.empty(M, D).pin_memory(), _ws(M)
        s.wait_stream(torch.cuda.default_stream())
        for c in range(calls):
            y.fill_(float("nan"))
            _ffn(w, xs[i], y, ws, stream=s)
            s.synchronize()
            if not torch.equal(y, refs[i]):
                bad.append((i, c))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad and aqt.aqt_device_status() == 0


def test_ffn_host_captured_in_a_graph():
    M = 4000
    w, x = _weights(), torch.randn(4000, D)
    ref = torch.empty(M, D, device="cuda")
    _ffn(w, x.cuda(), ref, _ws(M))
    xh, yh, ws, s = x.pin_memory(), torch.empty(M, D).pin_memory(), _ws(M), torch.cuda.Stream()
    _ffn(w, xh, yh, ws, stream=s)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        _ffn(w, xh, yh, ws, stream=s)
    yh.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(yh, ref.cpu())
