"""The step timeline lists the steps of the plan, whichever way the launch runs
its percentile selects."""
import numpy as np
import pytest

import workloads as wl
from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [(120, 200), (512, 512), (700, 901)])
def test_timeline_rows_are_the_plans_steps(side):
    torch = torch_cuda()
    import paper_2010_07284_gb300 as vg
    ctx = vg.Context(trace=True)
    f = wl.config4_formula()
    F = ctx.compile(wl.formula_to_records(f), f.roots, 8)
    kinds = [st["kind"] for st in F.plan()["steps"]]
    assert 0 in kinds
    stream = torch.cuda.Stream()
    imgs = [np.stack([wl.uniform_image(*side, seed=4 * k + c)[0] for c in range(4)]) for k in range(2)]
    b = ctx.batch([(F, [ctx.image(im, stream)]) for im in imgs], stream)
    for _ in range(2):
        b.run(stream)
    stream.synchronize()
    t = b.trace()
    n = len(kinds)
    assert t[:, 0].tolist() == [0] * n + [1] * n
    assert t[:, 1].tolist() == list(range(n)) * 2
    assert t[:, 2].tolist() == kinds * 2
    assert np.all(t[:, 3] > 0) and np.all(t[:, 4] >= t[:, 3])
    assert np.all(t[:, 5] > 0) and np.all(t[:, 6] >= 0)
    deps = F.plan()["deps"]
    for j in range(2):
        for q, dep in enumerate(deps):
            for d in dep:
                # (an item's end is read behind its count, a little late)
                assert t[j * n + q, 3] >= t[j * n + d, 4] - 5000, "a step starts before one it waits for ends"
    b.close()
    ctx.close()
