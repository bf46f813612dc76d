"""Matrices are closed, tables dropped and memory released while other streams are being captured in
thread-local and relaxed mode: the captures end well, and so do a batch's and a device search's own
beside threads that open and close matrices. A close waits for work of other streams on the matrix."""
import threading

import numpy as np
import pytest

import oracle
from paper_1807_09932_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["thread_local", "relaxed"])
def test_captures_survive(mode):
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    X = np.random.default_rng(1).standard_normal((5000, 20)).astype(np.float32)
    ms = [ebic.Matrix(X) for _ in range(3)]
    for m in ms:
        m.build_pairs()
    y = torch.zeros(100, device="cuda")
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    errors = []

    def close():
        try:
            ms[0].drop_pairs()
            for m in ms:
                m.close()
            ebic.ebic_release_memory()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    with torch.cuda.graph(g, capture_error_mode=mode):
        y += 1
        t = threading.Thread(target=close)
        t.start()
        t.join()
        y += 1
    assert not errors
    g.replay()
    torch.cuda.synchronize()
    assert bool((y == 2).all())


def test_searches_and_batches_beside_closing_threads():
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    X = np.random.default_rng(2).standard_normal((4000, 24)).astype(np.float32)
    small = np.random.default_rng(3).standard_normal((500, 12)).astype(np.float32)
    with ebic.Matrix(X) as m:
        m.build_pairs()
        kw = dict(population=60, generations=8, archive_size=8, elite=4, tournament=3,
                  max_init_len=5, max_len=12, seed=5)
        want = ebic.ebic_run(m.handle, ebic.ebic_params_default(**kw))
        stop, errors = threading.Event(), []

        def churn():
            try:
                s = torch.cuda.Stream().cuda_stream
                while not stop.is_set():
                    k = ebic.Matrix(small, stream=s)
                    k.build_pairs(stream=s)
                    k.close()
            except Exception as e:  # noqa: BLE001
                errors.append(e)

        ts = [threading.Thread(target=churn) for _ in range(2)]
        for t in ts:
            t.start()
        try:
            for _ in range(10):
                got = ebic.ebic_run(m.handle, ebic.ebic_params_default(
                    flags=ebic.EBIC_RUN_ON_DEVICE, **kw))
                assert got["members"] == want["members"]
                assert np.array_equal(got["counts"], want["counts"])
                ebic.ebic_batch_free(ebic.ebic_batch_create(4))
        finally:
            stop.set()
            for t in ts:
                t.join()
        assert not errors


def test_close_waits_for_other_streams():
    """Scoring queued on a stream behind other work, the matrix closed at once and its memory taken by
    new matrices: the scores are those of the closed matrix."""
    import torch
    torch.cuda.init()
    from paper_1807_09932_gb300 import ebic
    X = np.random.default_rng(4).standard_normal((20000, 30)).astype(np.float32)
    c, o = synth.make_population(1, 200, 30, 2, 6)
    want, _ = oracle.eval_population(X, c, o)
    dc = torch.from_numpy(c.view(np.int16)).cuda()
    do = torch.from_numpy(o.astype(np.uint32).view(np.int32)).cuda()
    other = np.zeros((20000, 30), np.float32)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        cnt = torch.zeros(200, dtype=torch.int32, device="cuda")
        m = ebic.Matrix(X)
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)
            ebic.eval_population(m, dc, do, counts=cnt, want_bitmaps=False, direct=True,
                                 stream=s.cuda_stream)
        m.close()
        ks = [ebic.Matrix(other) for _ in range(3)]
        torch.cuda.synchronize()
        assert np.array_equal(cnt.cpu().numpy().view(np.uint32), want)
        for k in ks:
            k.close()
