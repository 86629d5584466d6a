"""The rules of the work estimate and the path-segment planner (csrc/plan_rules.h), compiled for the host."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "plan_rules.h"
extern "C" void cells(int n, const float *x, uint32_t *out) {
    for (int i = 0; i < n; i++) out[i] = hg::lattice_cell(x[i] * hg::kLatticeScale - hg::kLatticeShift);
}
extern "C" void cuts(int n, const float *t, const int32_t *leaf, float t0, int32_t leaf0, uint8_t *out) {
    for (int c = 0; c < n; c++) out[c] = hg::cut_made(t, leaf, c, t0, leaf0);
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wall", "-Werror", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1311_0705_gb300", "csrc"), str(d / "rules.cpp"), "-o", str(d / "rules.so")],
                   check=True)
    return ctypes.CDLL(str(d / "rules.so"))


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def test_every_coordinate_counts_for_its_cell(rules):
    x = np.concatenate([np.arange(0, 16, 0.01), np.linspace(1e-4, 0.9999, 999), [15.98, 15.9999]]).astype(np.float32)
    # the domain's faces, and past them by a rounding of the coordinates (a few 2^-24 of the domain, 16 cells)
    face = np.array([0.0, -0.0, -4e-6, 4e-6, 16.0, 16 - 4e-6, 16 + 4e-6], np.float32)
    x = np.concatenate([x, face])
    out = np.empty(len(x), np.uint32)
    rules.cells(len(x), _p(x), _p(out))
    inner = (np.abs(x - np.round(x)) < 2.0 ** -12) & (x > 0.5) & (x < 15.5)  # such a coordinate may count for either side
    np.testing.assert_array_equal(out[~inner], np.clip(np.floor(x[~inner]), 0, 15).astype(np.uint32))
    assert (np.abs(out[inner] + 0.5 - x[inner]) < 0.501).all()


def test_any_coordinate_gives_a_cell(rules):
    x = np.array([-40.0, 1e30, -1e30, np.nan, np.inf, -np.inf], np.float32)
    out = np.empty(len(x), np.uint32)
    rules.cells(len(x), _p(x), _p(out))
    assert (out < 16).all()


def _cuts(rules, t, leaf, t0, leaf0):
    t, leaf, out = np.array(t, np.float32), np.array(leaf, np.int32), np.zeros(len(t), np.uint8)
    rules.cuts(len(t), _p(t), _p(leaf), ctypes.c_float(t0), leaf0, _p(out))
    return [j for j in range(len(t)) if out[j]]


def test_cuts_follow_each_other(rules):
    none = -np.inf
    assert _cuts(rules, [1, 2, 3], [5, 6, 7], 0.0, 4) == [0, 1, 2]
    assert _cuts(rules, [1, none, 3], [5, -1, 7], 0.0, 4) == [0, 2]
    assert _cuts(rules, [none, none], [-1, -1], 0.0, 4) == []
    assert _cuts(rules, [1, 1, 2], [5, 5, 6], 0.0, 4) == [0, 2]  # the same leaf twice
    assert _cuts(rules, [1, 2], [4, 6], 0.0, 4) == [1]           # the first leaf
    # a time out of order, and one between: segments must not run backwards
    assert _cuts(rules, [1, 3, 2, 2.5, 4], [5, 7, 6, 8, 9], 0.0, 4) == [0, 1, 4]
    rng = np.random.default_rng(1)
    for _ in range(200):
        t, leaf = rng.integers(0, 20, 15).astype(float), rng.integers(0, 9, 15)
        t[rng.random(15) < 0.2] = none
        made = _cuts(rules, t, leaf, 1.0, 3)
        assert (np.diff([1.0] + list(t[made])) > 0).all()
        assert (np.diff([3] + list(leaf[made])) != 0).all()
