"""The memory that the library's pools keep: given back on request, and bounded when they start
empty (a matrix's, a pair table's and a call's pair table)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _held(torch, free0):
    torch.cuda.synchronize()
    return free0 - torch.cuda.mem_get_info()[0]


def test_kept_then_released():
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic, synth
    x = torch.randn(30000, 500, device="cuda")   # 1 GB of table
    y = torch.randn(436444, 16, device="cuda")
    c, o = synth.make_population(1, 400, 16, 2, 6)
    dc = torch.from_numpy(c.view(np.int16)).cuda()
    do = torch.from_numpy(o.astype(np.uint32).view(np.int32)).cuda()
    cnt = torch.zeros(400, dtype=torch.int32, device="cuda")
    ebic.Matrix(x[:64].contiguous()).close()     # the kernels' code is loaded
    ebic.ebic_release_memory()
    free0 = torch.cuda.mem_get_info()[0]
    slack = 256 << 20                            # the driver's granularity, code
    for n in (1, 4):
        ms = [ebic.Matrix(x) for _ in range(n)]
        for m in ms:
            m.build_pairs()
        with ebic.Matrix(y) as m:                # a table for the call
            ebic.eval_population(m, dc, do, counts=cnt, want_bitmaps=False)
        for m in ms:
            m.close()
        held = _held(torch, free0)
        assert held <= (2 << 30) + (512 << 20) + slack, held
        if n == 1:
            assert held > 512 << 20              # kept for the next matrix
    ebic.ebic_release_memory()
    assert _held(torch, free0) <= slack
