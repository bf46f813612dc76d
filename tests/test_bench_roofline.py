"""The evaluator's roof counts the columns that its walk reads, not those its early end leaves out."""
import os
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

from paper_1807_09932_gb300 import synth


def walk(X, c):
    """The walk of one segment: column 0, then two at a time while a row still follows."""
    follows = ~np.isnan(X[:, c[0]])
    read = 1
    k = 1
    while k < len(c) and follows.any():
        for j in (k, k + 1):
            if j < len(c):
                follows &= X[:, c[j]] >= X[:, c[j - 1]]
                read += 1
        k += 2
    return read


def test_columns_of_the_walk():
    import bench
    rng = np.random.default_rng(3)
    X = rng.standard_normal((1024 * 3 + 100, 30)).astype(np.float32)
    X[rng.random(X.shape) < 0.02] = np.nan
    X[:1024, 3] = np.nan
    cols, offs = synth.make_population(2, 40, 30, 1, 24)
    want = np.mean([walk(X[1024 * s:1024 * (s + 1)], cols[offs[i]:offs[i + 1]])
                    for i in range(40) for s in range(3)])
    assert bench.walked_columns(X, [(cols, offs)]) == pytest.approx(want, abs=1e-12)


def test_every_row_follows_every_column_is_read():
    import bench
    X = np.tile(np.arange(16, dtype=np.float32), (2048, 1))
    cols = np.arange(16, dtype=np.uint16)
    assert bench.walked_columns(X, [(cols, np.array([0, 15, 16], np.uint32))]) == 8.0
