"""What the host code does when device memory runs out, on a fake CUDA runtime: an allocation that a
call needs has the pools give back what they hold and is tried once more; a population's table for
the call, which it can do without, leaves the call to the evaluator."""
import ctypes

import numpy as np
import pytest

import native_build

POOL, ASYNC, MALLOC, TABLE = 0, 1, 2, 3  # matrices' pool, default pool, cudaMalloc, calls' tables' pool
OK, OOM = 0, -2
CUDA_OOM = 2                     # cudaErrorMemoryAllocation
P = ctypes.c_void_p


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    lib = native_build.load(tmp_path_factory.mktemp("native"), "fake_cuda",
                            ["capi.cpp", "devmem.cpp"])
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_live.restype = ctypes.c_size_t
    lib.fake_limit.restype = ctypes.c_uint64
    lib.fake_device.restype = P
    lib.fake_device.argtypes = [ctypes.c_size_t]
    lib.fake_device_free.argtypes = [P]
    lib.fake_scratch.argtypes = lib.fake_fixed.argtypes = [ctypes.c_size_t]
    lib.ebic_load_matrix.argtypes = [P, ctypes.c_int64, ctypes.c_int32, ctypes.c_int64,
                                     ctypes.c_uint32, ctypes.c_float, P, ctypes.POINTER(P)]
    lib.ebic_eval_population.argtypes = [P, P, P, ctypes.c_uint32, ctypes.c_uint32, P, P, P]
    lib.ebic_matrix_build_pairs.argtypes = [P, ctypes.c_uint64, P, P]
    lib.ebic_free_matrix.argtypes = [P]
    lib.ebic_matrix_drop_pairs.argtypes = [P]
    lib.fake_reset()
    return lib


def log(lib):
    return lib.fake_log().decode().splitlines()


def given_back(lib):
    first = log(lib)[:4]
    return first[0] == "sync" and {"trim library 0", "trim default 0"} <= set(first[1:])


def load(lib, rows, cols):
    x = np.zeros((rows, cols), np.float32)
    h = P()
    rc = lib.ebic_load_matrix(x.ctypes.data, rows, cols, cols, 1, 0.0, None, ctypes.byref(h))
    return rc, h


class Population:
    def __init__(self, n):
        self.n = n
        self.cols = np.tile(np.array([0, 1], np.uint16), n)
        self.offs = np.arange(0, 2 * n + 1, 2, dtype=np.uint32)
        self.counts = np.zeros(n, np.uint32)

    def score(self, lib, h, flags=0):
        return lib.ebic_eval_population(h, self.cols.ctypes.data, self.offs.ctypes.data, self.n,
                                        flags, self.counts.ctypes.data, None, None)


def test_matrix_and_table_tried_again(lib):
    rc, h = load(lib, 3000, 20)
    assert rc == OK
    lib.fake_reset()
    lib.fake_fail(POOL, 0, 1)
    rc, h2 = load(lib, 3000, 20)
    assert rc == OK and given_back(lib)
    lib.fake_reset()
    lib.fake_fail(POOL, 0, 1)
    assert lib.ebic_matrix_build_pairs(h, 1 << 40, None, None) == OK
    assert given_back(lib)
    lib.fake_reset()
    lib.fake_fail(POOL, 0, 2)
    assert lib.ebic_matrix_build_pairs(h2, 1 << 40, None, None) == OOM
    rc, h3 = load(lib, 3000, 20)
    assert rc == OK
    for m in (h, h2, h3):
        lib.ebic_free_matrix(m)
    assert lib.fake_live(POOL) == 0


def test_scratch_tried_again(lib):
    rc, h = load(lib, 3000, 20)
    pop = Population(10)
    lib.fake_reset()
    assert pop.score(lib, h) == OK
    held, calls = lib.fake_live(ASYNC), lib.fake_seen(ASYNC)
    assert held == 0 and calls >= 3 and "trim library 0" not in log(lib)
    for k in range(calls):  # each of the call's allocations in turn
        lib.fake_reset()
        lib.fake_fail(ASYNC, k, 1)
        assert pop.score(lib, h) == OK
        assert {"trim library 0", "trim default 0"} <= set(log(lib))
        lib.fake_reset()
        lib.fake_fail(ASYNC, k, 2)
        assert pop.score(lib, h) == OOM
        assert lib.fake_live(ASYNC) == 0  # nothing stays behind
    lib.ebic_free_matrix(h)


@pytest.mark.parametrize("kind,call", [(ASYNC, "fake_scratch"), (MALLOC, "fake_fixed")])
def test_the_batch_allocations_tried_again(lib, kind, call):
    lib.fake_reset()
    lib.fake_fail(kind, 0, 1)
    assert getattr(lib, call)(1 << 20) == OK and given_back(lib)
    lib.fake_reset()
    lib.fake_fail(kind, 0, 2)
    assert getattr(lib, call)(1 << 20) == CUDA_OOM


def test_a_capture_is_left_alone(lib):
    lib.fake_reset()
    lib.fake_capture(1)
    lib.fake_fail(ASYNC, 0, 1)
    assert lib.fake_scratch(1 << 20) == CUDA_OOM
    assert log(lib) == []
    lib.fake_reset()


# 140,000 rows, 1,000 candidates of 20 columns: above the line for a table built for the call
BIG = (140000, 20, 1000)


def test_call_table_leaves_a_bounded_amount(lib):
    rows, cols, n = BIG
    rc, h = load(lib, rows, cols)
    pop = Population(n)
    lib.fake_reset()
    assert pop.score(lib, h) == OK
    assert [x for x in log(lib) if x != "sync"] == ["prepare", "pair build", "pair evaluate"]
    assert lib.fake_seen(TABLE) == 2 and lib.fake_seen(POOL) == 0  # the table and its term lists
    assert lib.fake_limit(TABLE) == 512 << 20
    other = lib.fake_seen(ASYNC)
    lib.fake_reset()
    assert pop.score(lib, h, flags=2) == OK   # EBIC_EVAL_DIRECT: the rest of the scratch
    assert lib.fake_seen(ASYNC) == other and lib.fake_seen(TABLE) == 0
    assert lib.fake_live(ASYNC) == lib.fake_live(TABLE) == 0
    lib.ebic_free_matrix(h)


@pytest.mark.parametrize("which", [0, 1])    # the table, its term lists
def test_call_table_without_memory_falls_back(lib, which):
    rows, cols, n = BIG
    rc, h = load(lib, rows, cols)
    pop = Population(n)
    lib.fake_reset()
    lib.fake_fail(TABLE, which, 1)
    assert pop.score(lib, h) == OK
    assert not any(x.startswith("trim") for x in log(lib))   # nor does the call wait for memory
    assert [x for x in log(lib) if x in ("pair build", "pair evaluate", "evaluate")] == ["evaluate"]
    assert lib.fake_live(TABLE) == 0
    lib.ebic_free_matrix(h)


def test_captured_call_takes_no_table(lib):
    rows, cols, n = BIG
    rc, h = load(lib, rows, cols)
    dev = {}
    for name, a in (("cols", Population(n).cols), ("offs", Population(n).offs),
                    ("counts", np.zeros(n, np.uint32))):
        dev[name] = lib.fake_device(a.nbytes)
        ctypes.memmove(dev[name], a.ctypes.data, a.nbytes)
    lib.fake_reset()
    lib.fake_capture(1)
    rc = lib.ebic_eval_population(h, dev["cols"], dev["offs"], n, 0, dev["counts"], None, None)
    assert rc == OK and log(lib) == ["prepare", "evaluate"] and lib.fake_seen(TABLE) == 0
    lib.fake_reset()
    rc = lib.ebic_eval_population(h, dev["cols"], dev["offs"], n, 0, dev["counts"], None, None)
    assert rc == OK and log(lib) == ["prepare", "pair build", "pair evaluate"]
    for d in dev.values():
        lib.fake_device_free(d)
    lib.ebic_free_matrix(h)


def test_release(lib):
    rows, cols, n = BIG
    rc, h = load(lib, rows, cols)
    assert Population(n).score(lib, h) == OK
    lib.ebic_free_matrix(h)
    lib.fake_reset()
    assert lib.ebic_release_memory(ctypes.c_int32(-1)) == OK
    assert log(lib)[0] == "idle"
    assert set(log(lib)[1:]) == {"trim library 0", "trim tables 0", "trim default 0"}
    assert lib.ebic_release_memory(ctypes.c_int32(7)) == -1


SHAPES = [(1, 1), (1000, 20), (4097, 33), (300, 52), (5000, 64), (70001, 127), (513, 128),
          (9000, 208), (9000, 209), (3000, 457), (100, 666), (65, 832)]


@pytest.mark.parametrize("rows,cols", SHAPES)
def test_admission_counts_what_a_run_allocates(lib, rows, cols):
    """The server's footprint of a run without an archive is its matrix, its pair table (within the
    budget) or else its population's bitmaps, and 4 KB; the matrix and table as the library
    allocates them."""
    from paper_1807_09932_gb300 import ebic, serve
    lib.fake_reset()
    before = lib.fake_live(POOL)
    rc, h = load(lib, rows, cols)
    matrix = lib.fake_live(POOL) - before
    assert rc == OK and lib.ebic_matrix_build_pairs(h, 1 << 60, None, None) == OK
    table = lib.fake_live(POOL) - before - matrix
    lib.ebic_free_matrix(h)
    assert ebic.ebic_matrix_bytes(rows, cols) == (matrix, table)
    spec = serve.RunSpec(run_id=0, X=np.empty((rows, cols), np.float32), max_cand=10)
    be = object.__new__(serve.GpuBackend)
    be.ebic = ebic
    be.pair_budget = 0
    assert be.footprint(spec) == matrix + 10 * ((rows + 31) // 32) * 4 + 4096
    be.pair_budget = table
    assert be.footprint(spec) == matrix + table + 4096


def test_a_closed_run_leaves_its_memory_to_every_allocator():
    from types import SimpleNamespace as NS

    from paper_1807_09932_gb300 import serve
    calls = []
    be = object.__new__(serve.GpuBackend)
    be.dev = NS(index=0)
    be.torch = NS(cuda=NS(synchronize=lambda d: calls.append("sync")))
    be.ebic = NS(ebic_release_memory=lambda d: calls.append(("release", d)))
    be.runs = {3: {"m": NS(close=lambda: calls.append("close"))}}
    be.close_run(3)
    assert calls == ["sync", "close", ("release", 0)]


def test_closing_beside_another_threads_capture(lib):
    """Closing a matrix, dropping its table and releasing memory wait for the device in a way that a
    thread-local or relaxed capture of another thread (ebic_batch_create's, a device search's) survives."""
    rc, h = load(lib, 3000, 20)
    assert rc == OK and lib.ebic_matrix_build_pairs(h, 1 << 40, None, None) == OK
    lib.fake_reset()
    lib.fake_other_capture(1)
    assert lib.ebic_matrix_drop_pairs(h) == OK and log(lib) == ["idle"]
    assert lib.ebic_free_matrix(h) == OK and log(lib) == ["idle", "idle"]
    assert lib.ebic_release_memory(ctypes.c_int32(-1)) == OK
    assert not lib.fake_other_broken() and lib.fake_live(POOL) == 0


def test_memory_that_cannot_be_freed_now_is_freed_later(lib):
    """Beside a capture in global mode nothing may wait for the device: the close fails, and its memory,
    which other streams may still use, is neither freed nor lost."""
    rc, h = load(lib, 3000, 20)
    rc2, h2 = load(lib, 500, 20)
    held = lib.fake_live(POOL)
    assert rc == rc2 == OK and held > 0
    lib.fake_reset()
    lib.fake_other_capture(2)
    assert lib.ebic_free_matrix(h) == -3        # EBIC_ERR_CUDA
    assert lib.fake_live(POOL) == held
    lib.fake_other_capture(0)
    assert lib.ebic_free_matrix(h2) == OK
    assert lib.fake_live(POOL) == 0


def test_closing_without_a_byte_left(lib):
    rc, h = load(lib, 3000, 20)
    lib.fake_reset()
    lib.fake_fail(MALLOC, 0, 100)
    assert lib.ebic_free_matrix(h) == OK and log(lib) == ["device sync"]
    assert lib.fake_live(POOL) == 0
