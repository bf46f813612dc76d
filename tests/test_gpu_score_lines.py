"""Scoring on either side of the lines between the kernels that do it: one launch and the pass (by
parts, warps and wanted members), 24 and 28 warps in the pass; and the one launch with members side
by side (up to 32 and up to 64 words). The two sides' results are compared with the evaluator's and
the overlap kernel's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [  # rows, cols, candidates, members, both trends
    (32, 12, 40, 64, False), (1000, 12, 300, 64, True), (1024, 12, 300, 61, False),
    (1025, 30, 300, 64, False), (2048, 30, 300, 63, True), (2049, 30, 300, 64, True),
    (1000, 12, 8000, 64, False), (1000, 12, 8001, 64, False),      # one part, at most 32 words
    (6000, 30, 2490, 64, True), (6000, 30, 4000, 64, True),         # two parts
    (20000, 30, 900, 64, True), (20000, 30, 1000, 64, True),        # five parts
    (20000, 30, 1500, 0, True), (20000, 30, 1700, 0, True),
    (20000, 30, 1600, 20, False), (20000, 30, 6000, 20, False),     # the pass, 24 and 28 warps
    (60000, 30, 1600, 20, False),
]


@pytest.mark.parametrize("rows,cols,n,k,negative", CASES)
def test_same_on_both_sides(rows, cols, n, k, negative):
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic, synth
    g = torch.Generator("cuda").manual_seed(rows + n)
    x = (torch.randn(rows, cols, generator=g, device="cuda") * 8).round()
    x[torch.rand(rows, cols, generator=g, device="cuda") < 0.02] = float("nan")
    c, o = synth.make_population(n, n, cols, 1, 7)
    ac, ao = synth.make_population(n + 1, max(k, 1), cols, 1, 3)
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a).view(t)).cuda()  # noqa: E731
    dc, do = dev(c, np.int16), dev(o.astype(np.uint32), np.int32)
    dac, dao = dev(ac, np.int16), dev(ao.astype(np.uint32), np.int32)
    flags = ebic.EBIC_NEGATIVE_TRENDS if negative else 0
    with ebic.Matrix(x) as m:
        abm = torch.zeros((max(k, 1), m.words), dtype=torch.int32, device="cuda")
        acnt = torch.zeros(max(k, 1), dtype=torch.int32, device="cuda")
        ebic.ebic_eval_population(m.handle, dac, dao, max(k, 1), flags | ebic.EBIC_EVAL_DIRECT, acnt,
                                  abm)
        out = []
        m.build_pairs()
        for f, overlaps in ((flags | ebic.EBIC_EVAL_DIRECT, True), (flags, True), (flags, False)):
            cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
            bm = torch.zeros((n, m.words), dtype=torch.int32, device="cuda")
            fit = torch.zeros(n, dtype=torch.int64, device="cuda")
            ov = torch.zeros((n, max(k, 1)), dtype=torch.int32, device="cuda")
            rc = ebic.ebic_eval_fitness(m.handle, dc, do, n, f, dac, dao, abm, k, cnt, bm, fit,
                                        ov if overlaps and k else None)
            assert rc == ebic.EBIC_OK and m.status() == ebic.EBIC_OK
            out.append((cnt, bm, fit, ov))
        for a, b in zip(out[0], out[1]):
            assert torch.equal(a, b)
        for a, b in zip(out[0][:3], out[2][:3]):
            assert torch.equal(a, b)
