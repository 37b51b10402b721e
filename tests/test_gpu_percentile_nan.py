"""Percentiles of channels that hold NaN of any bits (quiet or signalling, either
sign, any payload; all of them sort behind +infinity): alone, in a batch, and
per operator, below and above the size where many blocks share a select."""
import numpy as np
import pytest

from gpu_util import check_formula, torch_cuda

pytestmark = pytest.mark.gpu

QS = (0.0, 0.5, 0.999, 1.0)


@pytest.mark.parametrize("bits", [0xFF800001, 0xFF800002, 0xFF800010, 0xFF800100, 0xFF8FFFFF, 0xFF900000,
                                  0xFFC00000, 0xFFFFFFFF, 0x7F800001, 0x7FC00000])
@pytest.mark.parametrize("h,w", [(1, 5), (65, 129), (512, 512)])
@pytest.mark.parametrize("share", ["one", "many"])
def test_nan_of_any_bits(h, w, bits, share):
    torch_cuda()
    rng = np.random.default_rng(h + w)
    x = rng.normal(size=(1, h, w)).astype(np.float32)
    b = x.view(np.uint32).reshape(-1)
    if share == "one":
        b[rng.integers(0, b.size)] = bits
    else:
        b[rng.random(b.size) < 0.3] = bits
    rec = []
    for q in QS:
        rec.append(("PCT_GT", -1, -1, 0, 0, 0.0, q))
        rec.append(("PCT_LT", -1, -1, 0, 0, 0.0, q))
    check_formula(rec, list(range(len(rec))), [x])
