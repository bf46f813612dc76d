"""Batched requests whose archives differ in every way the batch's archive copy and fitness see:
none, no members, odd and even member counts up to 64, rows of one and several copy units, and
requests without a fitness between them. Equal to the oracle (whole numbers)."""
import numpy as np
import pytest

import oracle
from paper_1807_09932_gb300 import synth

pytestmark = pytest.mark.gpu


def test_mixed_archives():
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a).view(t)).cuda()  # noqa: E731
    rng = np.random.default_rng(11)
    mats, items, want = [], [], []
    for rows, cols in ((97, 9), (16385, 40), (40000, 70)):
        X = np.round(rng.standard_normal((rows, cols)).astype(np.float32) * 4)
        X[rng.random(X.shape) < 0.02] = np.nan
        m = ebic.Matrix(X)
        m.build_pairs()
        mats.append(m)
        for n_cand, k, fit, neg in ((1, 3, True, False), (33, None, False, True),
                                    (257, 64, True, True), (40, 0, True, False),
                                    (100, 33, True, False), (65, 20, True, True)):
            c, o = synth.make_population(rows + n_cand, n_cand, cols, 1, 9)
            ecnt, ebm = oracle.eval_population(X, c, o, negative=neg)
            cnt = torch.full((n_cand,), 3, dtype=torch.int32, device="cuda")
            f = torch.full((n_cand,), 3, dtype=torch.int64, device="cuda") if fit else None
            arch = (None, None, None, 0)
            efit = None
            if fit:
                ac, ao = synth.make_population(rows + 7, k, cols, 1, 6) if k else \
                    (np.zeros(1, np.uint16), np.zeros(1, np.uint32))
                abm = synth.random_bitmaps(rows + k, max(k, 1), rows, 0.2)
                efit, _ = oracle.fitness(rows, c, o, ecnt, ebm, ac, ao, abm[:k])
                arch = (dev(ac, np.int16), dev(ao, np.int32), dev(abm, np.int32), k)
            items.append((m.handle, dev(c, np.int16), dev(o, np.int32), n_cand,
                          ebic.EBIC_NEGATIVE_TRENDS if neg else 0, cnt, None, *arch, f))
            want.append((ecnt, efit))
    b = ebic.ebic_batch_create(len(items))
    try:
        for _ in range(2):  # the second replay finds the first one's scratch
            assert ebic.ebic_batch_run(b, ebic.make_requests(items), len(items)) == 0
            assert ebic.ebic_batch_status(b, len(items))[0] == 0
            for it, (ecnt, efit) in zip(items, want):
                assert np.array_equal(it[5].cpu().numpy().view(np.uint32), ecnt)
                if efit is not None:
                    assert np.array_equal(it[11].cpu().numpy().view(np.uint64), efit)
    finally:
        ebic.ebic_batch_free(b)
        for m in mats:
            m.close()
