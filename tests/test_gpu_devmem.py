"""The pool behind matrices and pair tables: what it keeps is bounded, and threads that open and
close matrices on their own streams never see each other's memory."""
import threading

import numpy as np
import pytest

import oracle
from paper_1807_09932_gb300 import synth

pytestmark = pytest.mark.gpu


def test_kept_memory_is_bounded():
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    x = torch.randn(30000, 500, device="cuda")  # 1 GB of table
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for n in (1, 4):
        ms = [ebic.Matrix(x) for _ in range(n)]
        for m in ms:
            m.build_pairs()
        for m in ms:
            m.close()
        torch.cuda.synchronize()
        held = free0 - torch.cuda.mem_get_info()[0]
        assert held <= (2 << 30) + (256 << 20), held  # the limit, and the driver's granularity


def test_threads_open_and_close():
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    sets = []
    for i in range(4):
        X = np.random.default_rng(i).standard_normal((2000 + 513 * i, 30 + i)).astype(np.float32)
        c, o = synth.make_population(i, 100, 30, 2, 8)
        sets.append((X, c, o, oracle.eval_population(X, c, o)))
    wrong = []

    def work(X, c, o, want):
        s = torch.cuda.Stream().cuda_stream
        for k in range(20):
            m = ebic.Matrix(X, stream=s)
            m.build_pairs(stream=s)
            cnt, bm = ebic.eval_population(m, c, o, stream=s, direct=k % 2 == 0)
            if not (np.array_equal(cnt, want[0]) and np.array_equal(bm, want[1])):
                wrong.append((X.shape, k))
            m.close()

    ts = [threading.Thread(target=work, args=a) for a in sets]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not wrong
