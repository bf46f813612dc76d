"""Device lists that the preparation rejects: what the call leaves is there for the next operation
in the stream, also when the list has no column at all and the evaluator therefore no work."""
import numpy as np
import pytest

import oracle
from paper_1807_09932_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 300, 2_000_000])
@pytest.mark.parametrize("noalloc", [False, True])
def test_list_without_columns(n, noalloc):
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    X = np.random.default_rng(n).standard_normal((700, 20)).astype(np.float32)
    good_c, good_o = synth.make_population(3, 50, 20, 2, 6)
    want, _ = oracle.eval_population(X, good_c, good_o)
    dc = torch.from_numpy(good_c.view(np.int16)).cuda()
    do = torch.from_numpy(good_o.astype(np.uint32).view(np.int32)).cuda()
    none = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    with ebic.Matrix(X) as m:
        def run(c, o, count, out):
            if noalloc:
                rc = ebic.ebic_eval_population_noalloc(m.handle, c, o, count, 0, out, None)
            else:
                rc = ebic.ebic_eval_population(m.handle, c, o, count, ebic.EBIC_EVAL_DIRECT, out,
                                               None)
            assert rc == ebic.EBIC_OK
        torch.cuda.synchronize()
        s = torch.cuda.default_stream()
        with torch.cuda.stream(s):
            for _ in range(3):
                cnt = torch.full((n,), -1, dtype=torch.int32, device="cuda")
                run(dc, none, n, cnt)
                after = cnt.clone()  # the next operation in the stream
                assert m.status() == ebic.EBIC_ERR_INVALID_ARG
                assert not after.any()
                got = torch.full((50,), -1, dtype=torch.int32, device="cuda")
                run(dc, do, 50, got)
                assert m.status() == ebic.EBIC_OK
                assert np.array_equal(got.cpu().numpy().view(np.uint32), want)
