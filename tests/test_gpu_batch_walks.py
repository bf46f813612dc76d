"""A batch's rank-code pass has a walk per stored layout and tile: requests of every one of them, both
trend options, with and without bitmaps, in one batch, against the evaluator's single calls."""
import numpy as np
import pytest

from paper_1807_09932_gb300 import synth

pytestmark = pytest.mark.gpu

# columns (1 to 10 bit planes, slabs of 16, 8, 4 and 2 words), rows, tile (0: the default)
SHAPES = [(1, 5000, 4), (3, 2049, 4), (7, 4100, 4), (15, 2100, 4), (31, 8200, 4), (52, 6000, 4),
          (63, 3000, 2), (104, 2050, 2), (127, 1500, 1), (200, 1100, 0), (240, 700, 0),
          (369, 600, 0), (500, 400, 0), (600, 300, 0), (832, 200, 0), (20, 1000, 2), (40, 300, 1),
          (12, 31, 0)]


def test_every_walk():
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a).view(t)).cuda()  # noqa: E731
    ms, items, want, out = [], [], [], []
    for i, (cols, rows, tile) in enumerate(SHAPES):
        g = torch.Generator("cuda").manual_seed(i)
        x = (torch.randn(rows, cols, generator=g, device="cuda") * 4).round()
        x[::2] = x[::2].sort(dim=1)[0]
        x[torch.rand(rows, cols, generator=g, device="cuda") < 0.01] = float("nan")
        m = ebic.Matrix(x)
        ms.append(m)
        if tile:
            m.set_tile(tile)
        n = 70 + i
        c, o = synth.make_population(i, n, cols, 1, min(cols, 24))
        c = np.sort(c) if cols == 1 else c
        dc, do = dev(c, np.int16), dev(o.astype(np.uint32), np.int32)
        for flags in (0, ebic.EBIC_NEGATIVE_TRENDS):
            for bitmaps in (True, False):
                cnt = torch.full((n,), -1, dtype=torch.int32, device="cuda")
                bm = torch.full((n, m.words), -1, dtype=torch.int32, device="cuda")
                items.append((m.handle, dc, do, n, flags, cnt, bm if bitmaps else None))
                out.append((cnt, bm if bitmaps else None))
                a, b = torch.zeros_like(cnt), torch.zeros_like(bm)
                rc = ebic.ebic_eval_population(m.handle, dc, do, n, flags | ebic.EBIC_EVAL_DIRECT, a,
                                               b)
                assert rc == ebic.EBIC_OK
                want.append((a, b))
    batch = ebic.ebic_batch_create(len(items))
    assert ebic.ebic_batch_run(batch, ebic.make_requests(items), len(items), None) == ebic.EBIC_OK
    rc, status = ebic.ebic_batch_status(batch, len(items))
    assert rc == ebic.EBIC_OK and not any(status)
    for (cnt, bm), (a, b) in zip(out, want):
        assert torch.equal(cnt, a) and (bm is None or torch.equal(bm, b))
    ebic.ebic_batch_free(batch)
    for m in ms:
        m.close()
