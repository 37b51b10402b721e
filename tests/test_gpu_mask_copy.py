"""Masks copied to device memory: by the kernel for small ones, by the
runtime for large or unaligned destinations, back to back on one stream, on
the default stream and inside a captured graph; always the masks themselves."""
import numpy as np
import pytest

from gpu_util import context, torch_cuda

pytestmark = pytest.mark.gpu

REC = [("THR_GT", -1, -1, 0, 0, 0.5, 0.0), ("THR_LT", -1, -1, 0, 0, 0.2, 0.0), ("NEAR", 0, -1, 0, 0, 0.0, 0.0),
       ("NOT", 1, -1, 0, 0, 0.0, 0.0)]
ROOTS = [0, 2, 3, 2]


def _result(ctx, h, w, stream=None):
    F = ctx.compile(REC, ROOTS, 8)
    x = np.random.default_rng(h * 7 + w).random((1, h, w)).astype(np.float32)
    res = ctx.eval(F, [ctx.image(x, stream)], stream)
    assert res.sync() == 0
    return res


def _expected(res, h, w):
    words = np.zeros((len(ROOTS), h, 4 * ((w + 127) // 128)), np.uint32)
    res.masks_into(words, on_device=False)
    return words


@pytest.mark.parametrize("offset", [0, 1, 4])
@pytest.mark.parametrize("h,w", [(1, 1), (3, 129), (240, 240), (1021, 1530), (2048, 8192)])
def test_masks_into_device_memory(h, w, offset):
    torch = torch_cuda()
    ctx = context()
    for stream in (torch.cuda.Stream(), None):
        res = _result(ctx, h, w, stream)
        exp = _expected(res, h, w)
        n = exp.size
        buf = torch.full((2 * n + 16,), 7, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        for k in range(2):  # one right behind the other
            res.masks_into(buf[offset + k * n:offset + (k + 1) * n], True, stream)
        torch.cuda.synchronize()
        got = buf.cpu().numpy().view(np.uint32)
        assert np.array_equal(got[offset:offset + n], exp.ravel())
        assert np.array_equal(got[offset + n:offset + 2 * n], exp.ravel())
        assert (got[:offset] == 7).all() and (got[offset + 2 * n:] == 7).all()


def test_masks_into_device_memory_inside_a_captured_graph():
    torch = torch_cuda()
    ctx = context()
    stream = torch.cuda.Stream()
    res = _result(ctx, 300, 500, stream)
    exp = _expected(res, 300, 500)
    out = torch.zeros((2,) + exp.shape, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        res.masks_into(out[0], True, stream)
        res.masks_into(out[1], True, stream)
    for _ in range(2):
        out.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        for k in range(2):
            assert np.array_equal(out[k].cpu().numpy().view(np.uint32), exp)
