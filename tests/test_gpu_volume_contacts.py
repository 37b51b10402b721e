"""Contacts between the slices of a volume: labels of sparse, even and dense
noise, and of salt on blobs, at widths around words and vectors and with dense
slices whose contacts exceed a block's list, against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import context, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("conn", [26, 6])
@pytest.mark.parametrize("shape", [(2, 3, 3), (3, 5, 31), (4, 7, 33), (5, 9, 64), (3, 40, 129), (2, 64, 515)])
@pytest.mark.parametrize("p", [0.03, 0.12, 0.3, 0.5, 0.75, 0.95])
def test_labels_across_slices(conn, shape, p):
    torch = torch_cuda()
    ctx = context()
    rng = np.random.default_rng(int(1000 * p) + conn + sum(shape))
    for k in range(4):
        m = (rng.random(shape) < p).astype(np.uint8)
        if k == 1:  # slices that touch only side by side or diagonally
            m[1::2] &= 1 - m[::2][:m[1::2].shape[0]]
        elif k == 2:  # full blocks with holes
            m[:, : shape[1] // 2 + 1, : shape[2] // 2 + 1] = 1
            m[rng.random(shape) < 0.1] = 0
        elif k == 3:  # checkerboards shifted from slice to slice
            z, y, x = np.indices(shape)
            m = (((x + y + z) % 2 == 0) & (rng.random(shape) < 0.5 + p / 2)).astype(np.uint8)
        mv = ctx.mask_volume(m)
        lab = torch.empty(m.size, dtype=torch.int32, device="cuda")
        ctx.ccl(mv, lab, conn)
        assert ctx.ccl_status() == 0, ctx.last_error()
        exp, _ = oracle.ccl3(m, conn)
        np.testing.assert_array_equal(lab.cpu().numpy().reshape(shape), exp)
