"""The overlap kernel vs the oracle (whole numbers, so equality): sizes at the edges of its
256-word segments, its two candidates per warp and its 32-member groups, and bitmaps whose words
are none, few (on both sides of the line of 6 non-zero words per member) and all non-zero."""
import numpy as np
import pytest

import oracle
from paper_1807_09932_gb300 import synth

pytestmark = pytest.mark.gpu


def sparse_bitmaps(rng, n, rows, n_members):
    """n bitmaps: candidate i has about few[i % 7] non-zero words per 256-word segment."""
    W = (rows + 31) // 32
    bm = np.zeros((n, W), dtype=np.uint32)
    line = min(6 * n_members, 128)
    for i in range(n):
        want = (0, 1, line - 1, line, line + 1, 200, 256)[i % 7]
        for s in range(0, W, 256):
            span = min(256, W - s)
            at = s + rng.permutation(span)[:min(want, span)]
            bm[i, at] = rng.integers(1, 1 << 32, size=len(at), dtype=np.uint64).astype(np.uint32)
    if rows % 32:
        bm[:, -1] &= np.uint32((1 << (rows % 32)) - 1)
    return bm


@pytest.mark.parametrize("rows,n_cand,n_members", [
    (1, 1, 1), (31, 15, 2), (32 * 255 + 1, 16, 3), (32 * 256, 17, 20), (32 * 257, 33, 31),
    (20000, 40, 40), (32 * 512 + 7, 21, 32), (9000, 7, 33), (8192, 9, 70),
    (32 * 2048 + 5, 1599, 20),      # two candidates per warp, an odd count
    (32 * 768, 4100, 5),            # the same, few members
])
def test_overlaps_and_fitness(rows, n_cand, n_members):
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    rng = np.random.default_rng(rows * 31 + n_cand)
    X = rng.standard_normal((rows, 12), dtype=np.float32)
    cols, offs = synth.make_population(n_cand, n_cand, 12, 1, 8)
    acols, aoffs = synth.make_population(n_members + 5, n_members, 12, 1, 8)
    bm = sparse_bitmaps(rng, n_cand, rows, n_members)
    abm = synth.random_bitmaps(7, n_members, rows, density=0.4)
    counts = np.bitwise_count(bm).sum(axis=1).astype(np.uint32)
    with ebic.Matrix(X) as m:
        fit, ov = ebic.fitness(m, cols, offs, counts, bm, acols, aoffs, abm)
    efit, eov = oracle.fitness(rows, cols, offs, counts, bm, acols, aoffs, abm)
    assert np.array_equal(ov, eov)
    assert np.array_equal(fit, efit)
