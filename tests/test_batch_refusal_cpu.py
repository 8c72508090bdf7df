"""perm_f3_batch refuses an entry above 2 with PF3_EDOMAIN and leaves its
outputs alone, with a device or without one, and before it works on a large
matrix."""
import time

import numpy as np
import pytest

from paper_2407_20205_gb300 import inputs


@pytest.fixture(scope="module")
def pf3():
    from paper_2407_20205_gb300 import build
    build.build()
    from paper_2407_20205_gb300 import binding
    return binding


def call(pf3, ns, at=None, value=3):
    flat, nsa = pf3.pack_batch([inputs.uniform_matrix(7000 + n, n) for n in ns])
    if at is not None:
        flat[at] = value
    res, hist = np.full(len(ns), 77, np.uint8), np.full(3, 77, np.uint64)
    rc = pf3._lib_batch(flat.ctypes.data_as(pf3._u8p), nsa.ctypes.data_as(pf3._i32p), len(ns),
                        res.ctypes.data_as(pf3._u8p), hist.ctypes.data_as(pf3._u64p))
    return rc, res, hist


@pytest.mark.parametrize("value", [3, 4, 7, 128, 255])
@pytest.mark.parametrize("ns", [(3,), (5, 4), (3, 17, 24), (2, 33)])
def test_bad_entry_at_every_place_of_a_word(pf3, ns, value):
    total = sum(n * n for n in ns)
    for at in sorted({*range(min(total, 20)), *range(max(0, total - 12), total)}):
        rc, res, hist = call(pf3, ns, at, value)
        assert rc == pf3.PF3_EDOMAIN, at
        assert (res == 77).all() and (hist == 77).all()


@pytest.mark.parametrize("ns", [(3,), (5, 4), (3, 17, 24), (2, 33)])
def test_good_entries_are_not_refused(pf3, ns):
    rc = call(pf3, ns)[0]
    assert rc in (pf3.PF3_OK, pf3.PF3_ECUDA)  # the latter without a device


@pytest.mark.gpu
def test_refused_before_a_large_matrix_is_worked_on(pf3):
    """52 x 52 takes about two seconds."""
    call(pf3, (5,))
    t0 = time.perf_counter()
    rc, res, hist = call(pf3, (52, 5), 52 * 52 + 7)
    assert rc == pf3.PF3_EDOMAIN and (res == 77).all() and (hist == 77).all()
    assert time.perf_counter() - t0 < 0.5
