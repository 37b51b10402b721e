"""Barrier placement inside fused groups, replayed on the CPU under the layout
that the interpreter has (csrc/dev_group.cuh): buffers are rows of 16-byte
vectors (the tile's words and one vector on either side), and vector v belongs
to thread v mod 512.

Every instruction's shared-memory accesses are replayed word by word, each with
the thread that makes it:
  * loads, constants, connectives and rank thresholds read and write whole
    vectors of their own (a load's masks and the staged planes are fetched by
    the thread that uses them);
  * N reads its own vector in three rows, and the word left and right of it in
    those rows: a tile with no more vectors than threads takes these by
    shuffles from the lanes beside, whose rows' vectors all take part, and only
    the first and the last lane of a warp read them; any other tile reads them;
  * a store reads its own core vectors, or nothing where it is done together
    with the instruction before it;
  * the float threshold writes single words, each by a lane of the warp that
    loads it.
A word that two threads touch, one of them writing, needs a barrier in between.
"""
from __future__ import annotations

import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_group_barriers import _plans

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_07284_gb300", "csrc")
# rows and words of a tile (words in fours), and of the last one in its column /
# row (0: the same)
SHAPES = [(32, 32, 0, 0), (64, 16, 0, 0), (16, 32, 0, 0), (16, 16, 0, 0), (64, 8, 0, 0), (16, 8, 0, 0),
          (14, 32, 0, 0), (27, 16, 0, 0), (40, 32, 0, 0), (32, 32, 4, 0), (16, 32, 1, 8), (7, 4, 0, 0),
          (154, 4, 0, 0), (6, 120, 0, 0), (40, 32, 0, 4)]
UNR = 8  # loads a lane of the float threshold has in flight: a warp takes 4 * UNR words


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    out = str(tmp_path_factory.mktemp("group") / "libgroup.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(ROOT, "tests", "group_shim.cpp"), "-o", out], check=True)
    return C.CDLL(out)


class Words:
    """Who has read and written the words of the buffers since the last barrier
    (-1: nobody, -2: several threads)."""

    def __init__(self, n):
        self.n = n
        self.clear()

    def clear(self):
        self.w, self.r = {}, {}

    def of(self, d, b):
        if b not in d:
            d[b] = np.full(self.n, -1, np.int32)
        return d[b]

    def read(self, b, at, thread):
        w = self.of(self.w, b)[at]
        r = self.of(self.r, b)
        old = r[at]
        r[at] = np.where((old == -1) | (old == thread), thread, -2)
        return bool(np.any((w != -1) & (w != thread)))

    def write(self, b, at, thread):
        w, r = self.of(self.w, b), self.of(self.r, b)
        bad = np.any((w[at] != -1) & (w[at] != thread)) or np.any((r[at] != -1) & (r[at] != thread))
        w[at] = np.where((w[at] == -1) | (w[at] == thread), thread, -2)
        return bool(bad)


def replay(plan, step, shape, layout, drop=None):
    """Yields (instruction, what) for every conflict of one group step; `drop`:
    an instruction whose barrier is left out."""
    rows_t, words_t, th, tww = shape
    th, tww = th or rows_t, tww or words_t
    NT, seg, nv = layout.group_threads(), layout.group_segment(), layout.group_row_vecs(words_t)
    halo = step["halo"]
    rows = th + 2 * halo
    one = rows * nv <= NT
    W = Words(rows * nv * 4)
    v = np.arange(rows * nv)
    row, col = v // nv, v % nv
    side = (col == 0) | (col == nv - 1)
    row_need = np.maximum(halo - row, row - (halo + th - 1))
    need = np.maximum(row_need, side)
    owner = v % NT
    core = (need <= 0) & (4 * (col - 1) < tww)

    def vec(sel):  # words and threads of whole vectors
        return (4 * v[sel, None] + np.arange(4)).ravel(), np.repeat(owner[sel], 4)

    first, last = step["insn_off"], step["insn_off"] + step["insn_cnt"]
    done = set()
    for k in range(first, last):
        ins = plan["insns"][k]
        if (k - first) % seg == 0:
            W.clear()
        if k in done:
            continue
        if ins["sync"] and k != drop:
            W.clear()
        op, h, d = ins["op"], ins["halo"], ins["dst"]
        mine = need <= h
        if op == 8:
            if W.read(ins["a"], *vec(core)):
                yield k, "a store reads words another thread wrote"
            continue
        if op == 1:  # float threshold, word by word
            s = 1 if h > 0 else 0
            bw = tww + 2 * s
            idx = np.arange((th + 2 * h) * bw)
            warp, in_warp = (idx // (4 * UNR)) % (NT // 32), idx % (4 * UNR)
            # of 16 words, word 4 * (part / 2) + quad goes to lane 8 * quad + part
            thread = 32 * warp + 8 * (in_warp % 4) + 2 * (in_warp % 16 // 4)
            at = (halo - h) * nv * 4 + 4 - s + (idx // bw) * nv * 4 + idx % bw
            if W.write(d, at, thread):
                yield k, "a float threshold writes words another thread touched"
            continue
        bad = False
        if op in (3, 4, 5, 9):
            for b in [ins["a"]] + ([ins["b"]] if op != 3 else []):
                bad |= W.read(b, *vec(mine))
        elif op == 6:
            b = ins["a"]
            if one:
                for dr in (-1, 0, 1):  # every vector of the rows
                    sel = row_need <= h
                    at = 4 * (v[sel, None] + dr * nv) + np.arange(4)
                    assert at.min() >= 0 and at.max() < W.n
                    bad |= W.read(b, at.ravel(), np.repeat(owner[sel], 4))
                lanes = ((mine & (col > 0) & (v % 32 == 0), -1), (mine & (col < nv - 1) & (v % 32 == 31), 4))
            else:
                for dr in (-1, 0, 1):
                    at = 4 * (v[mine, None] + dr * nv) + np.arange(4)
                    bad |= W.read(b, at.ravel(), np.repeat(owner[mine], 4))
                lanes = ((mine & (col > 0), -1), (mine & (col < nv - 1), 4))
            for sel, off in lanes:
                for dr in (-1, 0, 1):
                    bad |= W.read(b, 4 * (v[sel] + dr * nv) + off, owner[sel])
        if bad:
            yield k, "reads words another thread wrote"
        if W.write(d, *vec(mine)):
            yield k, "writes words another thread touched"
        if one and k + 1 < last and (k + 1 - first) % seg:
            n = plan["insns"][k + 1]
            if n["op"] == 8 and not n["sync"] and n["a"] == d:
                done.add(k + 1)  # the store takes the value as it is


def conflicts(plan, shape, layout, steps=None):
    for si, st in enumerate(plan["steps"]):
        if st["kind"] == 1 and (steps is None or si in steps):
            for k, what in replay(plan, st, shape, layout):
                yield si, k, what


@pytest.fixture(scope="module")
def plans():
    return _plans()


def test_layout_is_the_one_modelled(layout):
    assert layout.group_threads() == 512
    assert [layout.group_row_vecs(w) for w in (1, 3, 4, 5, 16, 32)] == [3, 3, 3, 4, 6, 10]


@pytest.mark.parametrize("shape", SHAPES)
def test_no_unsynchronised_conflicts(plans, layout, shape):
    for name, plan in plans:
        bad = next(conflicts(plan, shape, layout), None)
        assert bad is None, f"{name} tile {shape}: {bad}"


@pytest.mark.parametrize("shape", [(32, 32, 0, 0), (14, 32, 0, 0), (6, 120, 0, 0)])
def test_a_missing_barrier_is_seen(plans, layout, shape):
    """The barrier before an N whose operand was written since the barrier
    before: without it the rows above and below are another thread's."""
    seen = 0
    for name, plan in plans:
        for st in plan["steps"]:
            if st["kind"] != 1:
                continue
            first, last = st["insn_off"], st["insn_off"] + st["insn_cnt"]
            written = set()
            for k in range(first, last):
                ins = plan["insns"][k]
                if (k - first) % layout.group_segment() == 0:
                    written = set()
                elif ins["sync"]:
                    if ins["op"] == 6 and ins["a"] in written and seen < 60:
                        seen += 1
                        assert any(True for _ in replay(plan, st, shape, layout, drop=k)), (name, k)
                    written = set()
                if ins["op"] != 8:
                    written.add(ins["dst"])
    assert seen > 20
