"""The autotuner times the evaluator, the kernel that its tiles shape, whatever route a plain call on
the matrix would take; winners of another evaluator or layout are not taken from the cache."""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_1807_09932_gb300 import autotune, synth


@pytest.mark.parametrize("negative", [False, True])
def test_the_timed_call_asks_for_the_evaluator(monkeypatch, negative):
    import torch

    from paper_1807_09932_gb300 import ebic
    flags = []

    class Event:
        def __init__(self, enable_timing):
            pass

        def record(self, stream):
            pass

        def synchronize(self):
            pass

        def elapsed_time(self, other):
            return 1.0

    monkeypatch.setattr(torch.cuda, "Event", Event)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=0))
    monkeypatch.setattr(ebic, "ebic_eval_population",
                        lambda h, c, o, n, f, *rest: flags.append(f) or 0)
    m = SimpleNamespace(handle=None, set_tile=lambda t: None, set_chunk_cols=lambda c: None)
    measure = autotune.gpu_measure(m, None, None, 10, None, None, negative, iters=1)
    assert measure(1, 0) == 1.0
    want = ebic.EBIC_EVAL_DIRECT | (ebic.EBIC_NEGATIVE_TRENDS if negative else 0)
    assert flags == [want, want]


def test_winners_of_another_layout_are_not_taken():
    # the key of the evaluator that read ranks as bytes and halves
    assert autotune.shape_key(8, 64, 436444, 1600, 9.0, False) != "w8-c64-r19-p11-l9-n0"
    assert autotune.shape_key(8, 64, 436444, 1600, 9.0, False).endswith("-w8-c64-r19-p11-l9-n0")


@pytest.mark.gpu
def test_a_population_large_enough_for_a_table():
    """120,000 x 40, 1,600 candidates: a plain call builds a table for itself (no evaluator launch),
    the tuner's calls don't."""
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    x = torch.randn(120000, 40, device="cuda")
    cols, offs = synth.make_population(4, 1600, 40, 2, 10)
    dc = torch.from_numpy(cols.view(np.int16)).cuda()
    do = torch.from_numpy(offs.astype(np.uint32).view(np.int32)).cuda()
    cnt = torch.zeros(1600, dtype=torch.int32, device="cuda")
    with ebic.Matrix(x) as m:
        ebic.ebic_timing_enable(True)
        try:
            ebic.eval_population(m, dc, do, counts=cnt, want_bitmaps=False)
            want = cnt.clone()
            assert ebic.ebic_timing_read(ebic.EBIC_TIMING_PAIR_EVALUATE)[1] == 1
            ebic.ebic_timing_enable(True)   # (drops what was recorded)
            tile, chunk, ms, hit = autotune.tune_matrix(m, dc, do, 1600, 6.0, cnt, None, iters=2)
            tiles = len(autotune.allowed_tiles(m))
            assert ebic.ebic_timing_read(ebic.EBIC_TIMING_PAIR_EVALUATE)[1] == 0
            assert ebic.ebic_timing_read(ebic.EBIC_TIMING_EVALUATE)[1] == \
                3 * tiles * len(autotune.CHUNKS)
        finally:
            ebic.ebic_timing_enable(False)
        assert not hit and torch.equal(cnt, want)
