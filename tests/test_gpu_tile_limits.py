"""Tile shapes at the edges of what is accepted: tall tiles of few words and tiles
whose words are no multiple of four run and give the oracle's masks, beside
contexts of other shapes; a tile table may name such shapes, and shapes whose
buffers do not fit."""
import re

import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_util import assert_same, check_formula, context, torch_cuda

pytestmark = pytest.mark.gpu


def _formula():
    f = wl.random_dag(200, seed=11, max_depth=50)
    return wl.formula_to_records(f), f.roots


@pytest.mark.parametrize("rows,words", [(545, 1), (1024, 1), (1024, 4), (600, 4), (825, 5), (512, 8), (80, 44),
                                        (33, 7), (6, 200), (1, 250)])
def test_tall_tiles_match_oracle(rows, words):
    torch_cuda()
    rec, roots = _formula()
    ctx = context(tile_rows=rows, tile_words=words)
    for h, w in ((1100, 131), (70, 1500)):
        img = wl.uniform_image(h, w, seed=h)
        check_formula(rec, roots, [img], ctx=ctx, modes=("fused",))
        check_formula(rec, roots, [img], ctx=context(), modes=("fused",))


def test_refused_shapes():
    torch_cuda()
    import paper_2010_07284_gb300 as vg
    for rows, words in ((1024, 5), (1024, 256), (300, 64), (1025, 1), (1, 257)):
        with pytest.raises(vg.VlError):
            vg.Context(tile_rows=rows, tile_words=words)


@pytest.mark.parametrize("rows,words,runs", [(33, 32, True), (44, 32, True), (128, 8, True), (20, 7, True),
                                             (322, 4, True), (600, 1, True), (2, 112, False)])
def test_tables_name_tall_narrow_and_wide_shapes(tmp_path, rows, words, runs):
    torch_cuda()
    import paper_2010_07284_gb300 as vg
    rec, roots = _formula()
    imgs = [wl.uniform_image(640, 900 + 40 * k, seed=k) for k in range(2)]
    ctx = vg.Context()
    F = ctx.compile(rec, roots, 8)
    jobs = [(F, [ctx.image(im)]) for im in imgs]
    plain = ctx.tile_shape(jobs)
    ctx.autotune(jobs, reps=1)
    path = tmp_path / "tiles.txt"
    ctx.save_tuning(path)
    lines = path.read_text().splitlines()
    key = re.match(r"[0-9a-f]{16}", lines[1]).group(0)
    path.write_text(f"{lines[0]}\n{key} {rows} {words} 2\n")
    ctx = vg.Context()
    F = ctx.compile(rec, roots, 8)
    jobs = [(F, [ctx.image(im)]) for im in imgs]
    ctx.load_tuning(path)
    got = ctx.tile_shape(jobs)
    assert got["tuned"] == runs
    want = (rows, words) if runs else (plain["tile_rows"], plain["tile_words"])
    assert (got["tile_rows"], got["tile_words"]) == want
    results = ctx.eval_batch(jobs)
    for im, res in zip(imgs, results):
        assert res.sync() == 0
        exp = oracle.evaluate(rec, roots, [im], conn=8).masks
        assert_same([res.mask(r) for r in range(len(roots))], exp, f"{rows} x {words}")
    for rows, words in ((64, 64), (45, 32), (0, 8)):  # more than a table may name
        path.write_text(f"{lines[0]}\n{key} {rows} {words} 2\n")
        with pytest.raises(vg.VlError):
            ctx.load_tuning(path)


def test_autotuner_tries_one_wave_heights_again():
    """A 3000 x 4096 image on two CTAs an SM: tiles of 32 words fit one wave of
    the grid from about forty rows on."""
    torch = torch_cuda()
    import paper_2010_07284_gb300 as vg
    ctx = vg.Context()
    rec, roots = [("THR_GT", -1, -1, 0, 0, 0.5, 0.0), ("NEAR", 0, -1, 0, 0, 0.0, 0.0)], [1]
    F = ctx.compile(rec, roots, 8)
    img = wl.uniform_image(3000, 4096, seed=1)
    jobs = [(F, [ctx.image(img)])]
    s = torch.cuda.Stream()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per_col = 2 * sms // 4
    rows = -(-3000 // per_col)
    assert 34 <= rows <= 44
    trials = ctx.autotune(jobs, stream=s, reps=1)["trials"]
    tall = [t for t in trials if (t["tile_rows"], t["tile_words"]) == (rows, 32)]
    assert len(tall) == 2 and all(t["status"] == 0 for t in tall)
