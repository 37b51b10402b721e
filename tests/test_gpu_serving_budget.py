"""Device memory a served query is admitted with: the buffers that a batch gives
it, neither more (queries that fit would wait) nor less."""
import numpy as np
import pytest

import workloads as wl
from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

SLACK = 1 << 20  # tables, alignment


def buffers(F, h, w):
    """Bytes of a job's buffers and result masks, from its plan."""
    wp = (w + 127) // 128 * 4
    mask, px = 4 * h * wp, h * w
    plan = F.plan()
    sz = plan["sizes"]
    sets = 1 + max([s["scratch"] for s in plan["selects"]], default=-1)
    tiles = -(-h // 32) * -(-wp // 32)
    state = 4 * tiles * 16 * min(32, wp) * 32
    nums = sum(1 for a in plan["arith"] if a["op"] == 5)
    split = h * w >= 1 << 18
    return (mask * (sz["n_inter_slots"] + sz["n_root_slots"] + sz["n_rank_planes"]) + sets * (8 * px + state)
            + 4 * h * 32 * wp * nums + (65600 * len(plan["pct"]) if split else 0)), sets * state // 4


def formulas():
    f = wl.random_dag(300, seed=3, max_depth=60)
    g = wl.arith_dag(60, seed=5)
    return {"masks": (wl.formula_to_records(f), f.roots, 1), "terms": (wl.formula_to_records(g), g.roots, 2)}


@pytest.mark.parametrize("h,w", [(1500, 1500), (1111, 2049)])
@pytest.mark.parametrize("kind", ["masks", "terms"])
def test_a_query_is_admitted_with_its_buffers(kind, h, w):
    torch_cuda()
    import paper_2010_07284_gb300 as vg
    ctx = vg.Context()
    rec, roots, channels = formulas()[kind]
    F = ctx.compile(rec, roots, 8)
    img = ctx.image(np.stack([wl.uniform_image(h, w, seed=c)[0] for c in range(channels)]))
    need, flags = buffers(F, h, w)
    assert kind == "terms" or flags > 2 * SLACK
    srv = vg.Server(ctx, max_inflight_batches=1, max_batch_jobs=4)
    st, res = srv.wait(srv.submit(F, [img]), timeout_us=60_000_000)
    assert st == 0
    peak = srv.stats()["peak_bytes"]
    assert need - SLACK <= peak <= need + SLACK, (peak, need)
    res.close()
    srv.close()
    ctx.close()
