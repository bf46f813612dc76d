"""Which entries of an archive list the fused preparation reads: every entry of a list in order, each
for the member that holds it; of a list whose offsets are wrong only what a member with offsets of
its own in order covers, so never past the columns because of a wrong total."""
import ctypes

import numpy as np
import pytest

import native_build


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return native_build.load(tmp_path_factory.mktemp("native"), "list_entries")


def members(lib, offs):
    offs = np.ascontiguousarray(offs, dtype=np.uint32)
    n, total = len(offs) - 1, int(offs[-1])
    out = np.full(total, 0xFFFFFFFF, np.uint32)
    p = ctypes.POINTER(ctypes.c_uint32)
    lib.list_entries(offs.ctypes.data_as(p), ctypes.c_uint32(n), ctypes.c_uint32(total),
                     out.ctypes.data_as(p))
    return out, n


def test_lists_in_order(lib):
    rng = np.random.default_rng(0)
    for n in (1, 2, 3, 20, 63, 64):
        offs = np.concatenate([[0], np.cumsum(rng.integers(1, 65, n))])
        got, _ = members(lib, offs)
        assert np.array_equal(got, np.repeat(np.arange(n), np.diff(offs)))


def test_wrong_total(lib):
    # two members of 2 and 3 columns; the last offset, and so the total, is far past them
    got, n = members(lib, [0, 2, 128])
    assert list(got[:2]) == [0, 0] and np.all(got[2:] == n)


def test_wrong_offsets_read_only_members_in_order(lib):
    rng = np.random.default_rng(1)
    for _ in range(300):
        n = int(rng.integers(1, 65))
        offs = np.concatenate([[0], np.cumsum(rng.integers(1, 65, n))])
        for _ in range(int(rng.integers(1, 4))):
            offs[rng.integers(0, n + 1)] = rng.integers(0, 64 * n + 200)
        got, n = members(lib, offs)
        total = int(offs[-1])
        for t, m in enumerate(got):
            if m == n:
                continue
            lo, hi = int(offs[m]), int(offs[m + 1])
            assert lo <= t < hi and hi - lo <= 64 and hi <= total and (m > 0 or lo == 0)
