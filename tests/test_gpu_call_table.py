"""Populations scored through a pair table built for the call (a matrix without one) against the
evaluator and, on a sample, the oracle: one range of rows and several, both trends, with and
without bitmaps, and a size just below each limit."""
import numpy as np
import pytest

import oracle
from paper_1807_09932_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,n_cand,negative", [
    (436444, 8, 300, False),        # one range, ragged last word
    (60001, 200, 13334, True),      # 256 MB limit: ranges of 1,536 words, two of them
    (40000, 300, 30000, False),     # ranges of 512 words, three of them
    (60001, 200, 13333, False),     # one candidate below cols * cols / 3: the evaluator
    (127968, 30, 1000, False),      # 3,999,000 candidates times words: the evaluator
    (128032, 30, 1000, True),       # 4,001,000: the table
])
def test_same_as_the_evaluator(rows, cols, n_cand, negative):
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    X = torch.randn(rows, cols, generator=torch.Generator("cuda").manual_seed(rows), device="cuda")
    X[torch.rand(rows, cols, device="cuda") < 0.01] = float("nan")
    X[::7] = (X[::7] * 2).round()
    lens = np.random.default_rng(n_cand).integers(1, min(cols, 7) + 1, n_cand)
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint32)
    picks = np.random.default_rng(1).random((n_cand, cols)).argsort(axis=1)
    c = np.concatenate([picks[i, :lens[i]] for i in range(n_cand)]).astype(np.uint16)
    dc = torch.from_numpy(c.view(np.int16)).cuda()
    do = torch.from_numpy(offs.view(np.int32)).cuda()
    with ebic.Matrix(X) as m:
        out = []
        for direct in (True, False):
            cnt = torch.full((n_cand,), 9, dtype=torch.int32, device="cuda")
            bm = torch.full((n_cand, m.words), 9, dtype=torch.int32, device="cuda")
            ebic.eval_population(m, dc, do, negative=negative, counts=cnt, bitmaps=bm,
                                 direct=direct)
            assert m.status() == 0
            out.append((cnt, bm))
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
        cnt = torch.zeros(n_cand, dtype=torch.int32, device="cuda")
        ebic.eval_population(m, dc, do, negative=negative, counts=cnt, want_bitmaps=False)
        assert torch.equal(cnt, out[0][0])
    few = 40
    ecnt, _ = oracle.eval_population(X.cpu().numpy(), c[:offs[few]], offs[:few + 1],
                                     negative=negative)
    assert np.array_equal(out[1][0][:few].cpu().numpy().view(np.uint32), ecnt)
