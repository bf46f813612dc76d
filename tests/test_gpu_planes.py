"""The bit-plane rank layout and its evaluator vs the oracle (whole numbers, so equality), at the
column counts where the number of planes or the slab height changes and at row counts around a
word, a slab and a tile; the same matrices in one batch without pair tables (the walk that takes
its layout at run time)."""
import numpy as np
import pytest

import oracle
from paper_1807_09932_gb300 import synth

pytestmark = pytest.mark.gpu

# (columns, rows): 1-10 planes; slabs of 16 words up to 208 columns, 8 up to 369, 4 up to 665
SHAPES = [(1, 33), (3, 512), (7, 513), (15, 1), (31, 2049), (32, 4097), (63, 1024), (64, 1025),
          (104, 1537), (105, 700), (127, 513), (128, 512), (208, 1030), (209, 257), (255, 300),
          (256, 255), (369, 513), (370, 129), (511, 200), (512, 127), (665, 131), (666, 65),
          (832, 190)]


@pytest.fixture(scope="module")
def ebic():
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic as e
    return e


def values(cols, rows):
    """Few distinct values (ties, so ranks well below the column count) in odd rows, all distinct
    ones in even rows, 2 % missing."""
    rng = np.random.default_rng(cols * 7919 + rows)
    X = rng.standard_normal((rows, cols), dtype=np.float32)
    X[1::2] = np.round(X[1::2] * 2)
    X[rng.random(X.shape) < 0.02] = np.nan
    if rows > 2:
        X[2] = np.nan
        X[0] = np.arange(cols)  # every code up to the largest
    return X


def population(cols, seed):
    rng = np.random.default_rng(seed)
    lists = [rng.permutation(cols)[:min(cols, L)].tolist()
             for L in (1, 2, 3, 4, 5, 8, 17, 64) for _ in range(5)]
    lists += [np.arange(min(cols, n)).tolist() for n in (2, 33, 64)]  # row 0 follows these
    return synth.population_from_lists(lists)


@pytest.mark.parametrize("cols,rows", SHAPES)
def test_evaluator_and_rank_export(ebic, cols, rows):
    X = values(cols, rows)
    c, o = population(cols, cols)
    for exclude in (True, False):
        with ebic.Matrix(X, exclude_missing=exclude, fill_value=0.5) as m:
            for negative in (False, True):
                cnt, bm = ebic.eval_population(m, c, o, negative=negative)
                ecnt, ebm = oracle.eval_population(X, c, o, exclude_missing=exclude,
                                                   fill_value=0.5, negative=negative)
                assert np.array_equal(cnt, ecnt) and np.array_equal(bm, ebm)
                cnt2, _ = ebic.eval_population(m, c, o, negative=negative, want_bitmaps=False)
                assert np.array_equal(cnt2, ecnt)
            got = m.ranks()
        F = np.where(np.isnan(X), np.float32(0.5), X) if not exclude else X
        for r in range(rows):
            ok = ~np.isnan(F[r])
            want = np.full(cols, 0xFFFF, dtype=np.uint16)
            want[ok] = np.unique(F[r][ok], return_inverse=True)[1]
            assert np.array_equal(got[r], want), r


def test_batch_without_pair_tables(ebic):
    import torch
    ms, items, alone = [], [], []
    for i, (cols, rows) in enumerate(SHAPES):
        X = values(cols, rows)
        m = ebic.Matrix(X)
        ms.append(m)
        c, o = population(cols, i)
        neg = i % 2 == 1
        alone.append(ebic.eval_population(m, c, o, negative=neg))
        dc = torch.from_numpy(c.view(np.int16)).cuda()
        do = torch.from_numpy(o.view(np.int32)).cuda()
        n = len(o) - 1
        items.append((m.handle, dc, do, n, ebic.EBIC_NEGATIVE_TRENDS if neg else 0,
                      torch.full((n,), 7, dtype=torch.int32, device="cuda"),
                      torch.full((n, m.words), 7, dtype=torch.int32, device="cuda")))
    reqs = ebic.make_requests(items)
    b = ebic.ebic_batch_create(len(items))
    try:
        assert ebic.ebic_batch_run(b, reqs, len(items)) == 0
        assert ebic.ebic_batch_status(b, len(items))[0] == 0
        for it, (cnt, bm) in zip(items, alone):
            assert np.array_equal(it[5].cpu().numpy().view(np.uint32), cnt)
            assert np.array_equal(it[6].cpu().numpy().view(np.uint32), bm)
    finally:
        ebic.ebic_batch_free(b)
        for m in ms:
            m.close()


@pytest.mark.parametrize("rows,n_cand,chunk", [(40000, 1, 0), (512, 3000, 64), (100000, 700, 128)])
def test_work_split_covers_every_candidate_and_row(ebic, rows, n_cand, chunk):
    """Fewer candidates than CTAs, many chunks on one tile, many chunks on many tiles."""
    X = values(64, rows)
    c, o = synth.make_population(5, n_cand, 64, 1, 6)
    with ebic.Matrix(X) as m:
        m.set_chunk_cols(chunk)
        cnt, bm = ebic.eval_population(m, c, o)
    ecnt, ebm = oracle.eval_population(X, c, o)
    assert np.array_equal(cnt, ecnt) and np.array_equal(bm, ebm)
