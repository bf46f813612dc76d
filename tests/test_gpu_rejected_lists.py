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


def test_archive_list_whose_total_is_past_its_columns():
    """The last offset of a device archive list is wrong: the list is rejected (its columns are not
    read up to that total), nothing is written, and the next call is right."""
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    X = np.random.default_rng(5).standard_normal((900, 20)).astype(np.float32)
    c, o = synth.make_population(3, 50, 20, 2, 6)
    ac, ao = synth.make_population(4, 20, 20, 2, 6)
    cnt, bm = oracle.eval_population(X, c, o)
    _, abm = oracle.eval_population(X, ac, ao)
    fit, _ = oracle.fitness(900, c, o, cnt, bm, ac, ao, abm)
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a).view(t)).cuda()  # noqa: E731
    with ebic.Matrix(X) as m:
        m.build_pairs()
        for total in (int(ao[-1]) + 100, 20 * 64, 2**31):
            bad = ao.astype(np.uint32).copy()
            bad[-1] = total
            for offs, status in ((bad, ebic.EBIC_ERR_INVALID_ARG), (ao, ebic.EBIC_OK)):
                f = torch.full((50,), 5, dtype=torch.int64, device="cuda")
                n = torch.zeros(50, dtype=torch.int32, device="cuda")
                rc = ebic.ebic_eval_fitness(m.handle, dev(c, np.int16), dev(o, np.int32), 50, 0,
                                            dev(ac, np.int16), dev(offs, np.int32),
                                            dev(abm, np.int32), 20, n, None, f, None)
                assert rc == ebic.EBIC_OK and m.status() == status
                if status == ebic.EBIC_OK:
                    assert np.array_equal(f.cpu().numpy().view(np.uint64), fit)
                else:
                    assert bool((f == 5).all())
