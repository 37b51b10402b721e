"""Number-term programs with few and with many live values: the executor gives
a thread four, two or one vectors of pixels, and half of the threads the work,
as the registers leave room; ragged rows, both pixel formats."""
import numpy as np
import pytest

from gpu_util import check_formula, torch_cuda

pytestmark = pytest.mark.gpu


def _program(live):
    """`live` sums that are all made before the first is used, then multiplied
    up from the last one; thresholds on the product and on a quotient."""
    rec = [("VALUE", -1, -1, 0, 0, 0.0, 0.0)]
    for k in range(live):
        rec.append(("ADD", 0, -1, 0, 0, 0.25 + 0.125 * k, 0.0))
    at = live
    for k in range(live - 1, 0, -1):
        rec.append(("MUL", at, k, 0, 0, 0.0, 0.0))
        at = len(rec) - 1
    rec.append(("DIV", at, 1, 0, 0, 0.0, 0.0))
    rec.append(("THR_GT", at, -1, 0, 0, 1.5, 0.0))
    rec.append(("THR_LT", len(rec) - 2, -1, 0, 0, 1.25, 0.0))
    return rec, [len(rec) - 2, len(rec) - 1]


@pytest.mark.parametrize("dtype", ["f32", "u16"])
@pytest.mark.parametrize("live", [1, 2, 3, 6, 10, 13])
def test_programs_of_every_register_count(live, dtype):
    torch_cuda()
    rec, roots = _program(live)
    for h, w in ((1, 1), (5, 3), (9, 130), (302, 519)):
        x = np.random.default_rng(live * h + w).random((1, h, w)).astype(np.float32)
        if dtype == "u16":
            x = (x * 3).astype(np.uint16)
        check_formula(rec, roots, [x])
