"""Percentile selects in each of their forms: one block per select with the
keys of a bin listed in shared memory, the same with a bin too large for the
list, and many blocks per select; in the executor and per operator, for float
and 16-bit pixels, at the sizes where the choice between them changes."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same, check_formula, context, torch_cuda

pytestmark = pytest.mark.gpu

QS = (0.0, 0.25, 0.5, 0.9, 1.0)


def _records():
    rec = []
    for q in QS:
        rec.append(("PCT_GT", -1, -1, 0, 0, 0.0, q))
        rec.append(("PCT_LT", -1, -1, 0, 0, 0.0, q))
    return rec, list(range(len(rec)))


def _image(h, w, kind, dtype, seed=0):
    rng = np.random.default_rng(1000 * h + w + seed)
    x = rng.normal(size=(1, h, w)).astype(np.float32)
    if kind == "flat":  # most pixels equal: one bin holds nearly all of them
        x = np.where(rng.random((1, h, w)) < 0.9, np.float32(0.25), x)
    elif kind == "special":
        at = rng.random((1, h, w))
        x = np.where(at < 0.1, np.float32(np.inf), x)
        x = np.where(at > 0.9, np.float32(-np.inf), x)
        x = np.where((at > 0.45) & (at < 0.5), np.float32(np.nan), x)
        x = np.where((at > 0.5) & (at < 0.55), np.float32(-0.0), x)
    if dtype == "u16":
        x = np.clip(np.nan_to_num(x, posinf=4, neginf=-4) * 9000 + 30000, 0, 65535).astype(np.uint16)
    return x.astype(np.float32) if dtype == "f32" else x


@pytest.mark.parametrize("dtype", ["f32", "u16"])
@pytest.mark.parametrize("kind", ["normal", "flat", "special"])
@pytest.mark.parametrize("h,w", [(1, 1), (3, 5), (250, 250), (511, 513), (512, 512), (64, 2051), (601, 1021)])
def test_percentiles_of_one_image(h, w, kind, dtype):
    torch_cuda()
    rec, roots = _records()
    check_formula(rec, roots, [_image(h, w, kind, dtype)])


@pytest.mark.parametrize("kind", ["normal", "flat"])
def test_percentiles_of_a_batch_with_a_block_per_select(kind):
    """70 jobs of 5 selects are more than the grid has blocks: a block each,
    also on images that a lone job would split."""
    torch = torch_cuda()
    ctx = context()
    rec, roots = _records()
    F = ctx.compile(rec, roots, 8)
    stream = torch.cuda.Stream()
    host = [_image(520, 510 + k % 3, kind, "f32" if k % 2 else "u16", seed=k) for k in range(4)]
    images = [ctx.image(x, stream) for x in host]
    results = ctx.eval_batch([(F, [images[k % 4]]) for k in range(70)], stream)
    exp = [oracle.evaluate(rec, roots, [x], conn=8).masks for x in host]
    for k in range(70):
        assert results[k].sync() == 0
        assert_same([results[k].mask(r, stream) for r in range(len(roots))], exp[k % 4], f"job {k}")
