"""The evaluator's walk by the height of its row tiles (1, 2 and 4 slabs of 512 rows: several candidates a
warp, one, one with two words a lane) at the edges of tiles, with lists that end on an odd and on an
even column and lists whose rows all follow, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1807_09932_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [1, 2, 4])
@pytest.mark.parametrize("rows,cols", [(1, 1), (512, 2), (2048, 3), (2049, 9), (1025, 31),
                                       (4097, 52), (6143, 33), (2561, 104), (1537, 127)])
@pytest.mark.parametrize("negative", [False, True])
def test_tiles(rows, cols, tile, negative):
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    rng = np.random.default_rng(rows + cols)
    X = np.round(rng.standard_normal((rows, cols)).astype(np.float32) * 4)
    X[::2] = np.sort(X[::2], axis=1)            # rows that every increasing list of columns follows
    X[rng.random(X.shape) < 0.02] = np.nan
    lists = [list(range(k)) for k in range(1, min(cols, 40) + 1)]
    lists += [list(rng.permutation(cols)[:k]) for k in range(1, min(cols, 12) + 1) for _ in range(3)]
    c, o = synth.population_from_lists(lists)
    want_c, want_b = oracle.eval_population(X, c, o, negative=negative)
    with ebic.Matrix(X) as m:
        try:
            m.set_tile(tile)
        except ebic.EbicError:
            pytest.skip("the tile does not fit")
        got_c, got_b = ebic.eval_population(m, c, o, negative=negative, direct=True)
        assert np.array_equal(got_c, want_c) and np.array_equal(got_b, want_b)
        m.set_chunk_cols(64)                     # chunks that end at every few lists
        got_c, _ = ebic.eval_population(m, c, o, negative=negative, direct=True, want_bitmaps=False)
        assert np.array_equal(got_c, want_c)
