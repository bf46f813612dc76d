"""The one-launch scoring of small calls vs the oracle (whole numbers, so equality) at the edges of
its 128-word parts and of its candidates per block, for every output the call can be asked for;
and the sizes just past its limits, which take the pass."""
import numpy as np
import pytest

import oracle
from paper_1807_09932_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,n_cand,k,negative", [
    (1, 3, 1, 1, False), (31, 8, 7, 0, False), (1000, 50, 200, 20, False),
    (4096, 64, 9, 64, False), (4096, 70, 8, 33, True), (4097, 20, 17, 3, False),
    (4097, 20, 17, 3, True), (12289, 30, 40, 7, True), (20000, 66, 33, 20, True),
    (28672, 65, 5, 2, True), (32768, 40, 31, 64, True), (32769, 40, 31, 64, True),
    (6000, 40, 8001, 4, True),
])
def test_scores(rows, cols, n_cand, k, negative):
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    rng = np.random.default_rng(rows + n_cand)
    X = np.round(rng.standard_normal((rows, cols)).astype(np.float32) * 8)
    X[rng.random(X.shape) < 0.02] = np.nan
    order = rng.permutation(cols)[:min(cols, 40)]
    X[::3, order] = np.sort(X[::3, order], axis=1)  # rows that long chains still match
    c, o = synth.make_population(rows, n_cand, cols, 1, min(cols, 12))
    longest = order.astype(np.uint16)  # and a chain past one step of terms
    c, o = np.concatenate([c, longest]), np.append(o, o[-1] + len(longest)).astype(np.uint32)
    ac, ao = synth.make_population(rows + 1, max(k, 1), cols, 1, min(cols, 6))
    ac, ao = (ac, ao) if k else (ac, ao[:1])
    cnt, bm = oracle.eval_population(X, c, o, negative=negative)
    _, abm = oracle.eval_population(X, ac, ao, negative=negative) if k else (None, None)
    if k == 0:
        abm = np.zeros((1, bm.shape[1]), np.uint32)
    fit, over = oracle.fitness(rows, c, o, cnt, bm, ac, ao, abm[:k])
    with ebic.Matrix(X) as m:
        m.build_pairs()
        for wb, wo in ((False, False), (True, True)):
            gc, gb, gf, go = ebic.eval_fitness(m, c, o, ac, ao, abm, negative=negative,
                                               want_bitmaps=wb, want_overlaps=wo)
            assert np.array_equal(gc, cnt) and np.array_equal(gf, fit)
            assert not wb or np.array_equal(gb, bm)
            assert not wo or k == 0 or np.array_equal(go, over)
        # device lists and outputs: a rejected list writes no fitness
        dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a).view(t)).cuda()  # noqa: E731
        n = len(o) - 1
        f = torch.full((n,), 5, dtype=torch.int64, device="cuda")
        counts = torch.zeros(n, dtype=torch.int32, device="cuda")
        bad = c.copy()
        bad[-1] = cols
        args = (dev(ac, np.int16), dev(ao, np.int32), dev(abm, np.int32), k, counts, None, f, None)
        flags = ebic.EBIC_NEGATIVE_TRENDS if negative else 0
        assert ebic.ebic_eval_fitness(m.handle, dev(bad, np.int16), dev(o, np.int32), n, flags,
                                      *args) == 0
        assert m.status() == ebic.EBIC_ERR_INVALID_ARG
        assert bool((f == 5).all())
        assert ebic.ebic_eval_fitness(m.handle, dev(c, np.int16), dev(o, np.int32), n, flags,
                                      *args) == 0
        assert m.status() == ebic.EBIC_OK
        assert np.array_equal(f.cpu().numpy().view(np.uint64), fit)
        assert np.array_equal(counts.cpu().numpy().view(np.uint32), cnt)
