"""The contractions that the bench credits a phase with are those performed:
compact tips are lookups, with or without a table of Q P."""
import os
import sys

import pytest

import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("N,S,C,precision,pre,tables", [
    (10, 61, 100, "fp32", 2 * 8 + 10, False),  # small: a' Q of every tip
    (96, 61, 513, "fp32", 2 * 94, True),
    (10, 122, 100, "fp32", 2 * 8, True),
    (10, 61, 100, "fp64", 2 * 8, False),
    (10, 122, 100, "fp64", 3 * 8, False),
    (10, 20, 100, "fp32", 2 * 8, False),
    (10, 20, 100, "fp64", 3 * 8, False),
    (10, 4, 100, "fp64", 2 * 8, False),
])
def test_products(N, S, C, precision, pre, tables):
    sys.path.insert(0, ROOT)
    import bench
    R = 4
    w = synth.small_workload(N, S, R, C, seed=1)
    fl = bench.contraction_flops(w, precision)
    one = 2 * S * S * R * C
    assert fl["post"] == (N - 2) * one
    assert fl["pre"] == pre * one
    assert fl["pmat"] == (2 * S ** 3 * N * R if tables else 0)
