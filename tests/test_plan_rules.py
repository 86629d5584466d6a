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
