"""The pair-table build vs the oracle, pair by pair: every ordered pair and single of a matrix
scored through the table (whole numbers, so equality), at the edges of its 64-word ranges, its 32
columns a and 16 columns b per block, and of every number of planes and slab height."""
import numpy as np
import pytest

import oracle
from paper_1807_09932_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols", [
    (1, 1), (5, 2), (64, 7), (2047, 15), (2048, 16), (2049, 17), (4100, 31), (33, 32), (700, 33),
    (16384, 20), (16385, 21), (513, 63), (1030, 64), (300, 65), (520, 128), (260, 209), (40, 257),
    (70, 370)])
def test_every_pair(rows, cols):
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    rng = np.random.default_rng(rows * 1009 + cols)
    X = np.round(rng.standard_normal((rows, cols)).astype(np.float32) * 3)  # many ties
    X[rng.random(X.shape) < 0.1] = np.nan
    X[0] = rng.permutation(cols)  # every code
    if cols <= 65:
        lists = [[a, b] if a != b else [a] for a in range(cols) for b in range(cols)]
    else:
        pick = sorted(set([0, 15, 16, 31, 32, 33, 63, 64, cols - 2, cols - 1]
                          + rng.integers(0, cols, 30).tolist()))
        lists = [[a, b] if a != b else [a] for a in pick for b in pick]
    c, o = synth.population_from_lists(lists)
    with ebic.Matrix(X) as m:
        m.build_pairs()
        cnt, bm = ebic.eval_population(m, c, o)
    ecnt, ebm = oracle.eval_population(X, c, o)
    assert np.array_equal(cnt, ecnt)
    assert np.array_equal(bm, ebm)
