"""Range arithmetic of the percentile selects (csrc/select_range.h) on the
host: keys are ordered like the floats with every NaN last, and from any guess
a select is down to the wanted key after at most three histograms -- also where
the range ends at the highest keys (negative NaN with small payloads)."""
from __future__ import annotations

import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_07284_gb300", "csrc")
ROUNDS = 3
TOP = 0xFFFFFFFF


@pytest.fixture(scope="module")
def sel(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    out = str(tmp_path_factory.mktemp("select") / "libselect.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(ROOT, "tests", "select_shim.cpp"), "-o", out], check=True)
    lib = C.CDLL(out)
    lib.sel_key_of.restype = lib.sel_bits_of.restype = C.c_uint
    return lib


def keys_of(sel, bits):
    return np.array([sel.sel_key_of(C.c_uint(int(b))) for b in bits], dtype=np.uint32)


def check(sel, keys, k, lo, hi, top=TOP):
    keys = np.ascontiguousarray(keys, dtype=np.uint32)
    out = C.c_uint(0)
    n = sel.sel_run(keys.ctypes.data_as(C.POINTER(C.c_uint)), len(keys), C.c_longlong(k),
                    C.c_uint(lo), C.c_uint(hi), C.c_uint(top), ROUNDS, C.byref(out))
    assert n >= 0, f"rank {k} from [{lo:#x}, {hi:#x}]: not down to one key after {ROUNDS} histograms"
    assert out.value == np.sort(keys)[k]


def test_keys_are_ordered_like_floats(sel):
    bits = np.array([0xFF800000, 0xFF7FFFFF, 0xBF800000, 0x80000001, 0x80000000, 0x00000000, 0x00000001,
                     0x3F800000, 0x7F7FFFFF, 0x7F800000, 0x7F800001, 0x7FC00000, 0x7FFFFFFF, 0xFFFFFFFF,
                     0xFFC00000, 0xFF900000, 0xFF800002, 0xFF800001], dtype=np.uint32)
    keys = keys_of(sel, bits)
    assert np.all(np.diff(keys.astype(np.int64)) > 0)
    assert keys[0] == 0 and keys[-1] == TOP
    assert [sel.sel_bits_of(C.c_uint(int(k))) for k in keys] == bits.tolist()


@pytest.mark.parametrize("bits", [0xFF800001, 0xFF800002, 0xFF800010, 0xFF800100, 0xFF880000, 0xFF8FFFFF,
                                  0xFF900000, 0xFFC00000, 0xFFFFFFFF, 0x7FFFFFFF, 0x7FC00000, 0x7F800001,
                                  0x7F800000, 0xFF800000, 0x80000000, 0x00000000])
@pytest.mark.parametrize("others", ["none", "uniform", "signed"])
def test_pixels_of_any_bits(sel, bits, others):
    rng = np.random.default_rng(3)
    x = rng.random(4000, dtype=np.float32) - np.float32(0.5 if others == "signed" else 0.0)
    b = np.full(5, bits, np.uint32) if others == "none" else np.append(x.view(np.uint32), np.uint32(bits))
    keys = keys_of(sel, b)
    order = np.sort(keys)
    at = int(np.searchsorted(order, keys[-1]))
    guesses = [(0, TOP), (int(order[0]), int(order[-1])),
               (int(order[len(order) // 2]), TOP), (int(order[-2]), TOP), (int(order[0]), int(order[1]))]
    for k in (0, len(b) // 2, at, len(b) - 1):
        for lo, hi in guesses:
            check(sel, keys, k, lo, hi)


@pytest.mark.parametrize("seed", range(40))
def test_random_ranges(sel, seed):
    rng = np.random.default_rng(seed)
    top = TOP if seed % 4 else 0xFFFF
    base = int(rng.integers(0, 2)) * (top - min(top, 1 << int(rng.integers(1, 33))) + 1)
    keys = base + (rng.random(300) * (top - base + 1)).astype(np.uint64)
    keys = np.minimum(np.append(keys, [top, top - 1]), top).astype(np.uint32)
    for _ in range(20):
        lo, hi = sorted(int(v) for v in rng.choice(keys, 2))
        if rng.random() < 0.2:
            hi = top
        if rng.random() < 0.2:
            lo = 0
        check(sel, keys, int(rng.integers(0, len(keys))), lo, hi, top)
