"""Ranges of more than 2^48 indices run as graphs of equal launch sequences that
find their place by a counter: the counts equal those of pieces short enough to
be launched one by one, and the asynchronous call returns long before they are
done."""
import time

import numpy as np
import pytest

from paper_2407_20205_gb300 import inputs
from test_gpu_meet import by_pieces, counts

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf3():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_20205_gb300 import binding
    return binding


@pytest.mark.parametrize("kind,first,length", [
    ("uniform", 0, (1 << 48) + 1),                          # one sequence more than 64
    ("uniform", (1 << 50) + 12345, (1 << 48) + (1 << 42)),  # 64 with one before and one behind them
    ("uniform", (1 << 51) - 987654321, (1 << 50) + (1 << 49) + (1 << 44) + 777),  # 256, twice 64 and a rest
    ("merged", (1 << 50) + 12345, (1 << 48) + (1 << 42))])
def test_equal_to_pieces(pf3, kind, first, length):
    n = 53
    A = inputs.uniform_matrix(7300, n) if kind == "uniform" else inputs.pooled_columns(7301, n, 24, 12)
    last = first + length - 1
    assert counts(pf3, A, first, last) == by_pieces(pf3, A, first, last, 1 << 46)


def test_bad_entry(pf3):
    import torch
    A = inputs.uniform_matrix(7302, 53)
    A[52, 52] = 3
    out = torch.zeros(3, dtype=torch.int64, device="cuda")
    pf3.perm_f3_range_counts_async(torch.from_numpy(A).cuda(), 53, 5, 1 << 50, out, None)
    assert out.tolist() == [0, 0, -1]
    A[52, 52] = 2
    assert counts(pf3, A, 0, 1 << 30) == by_pieces(pf3, A, 0, 1 << 30, 1 << 26)


def test_asynchronous_calls_return_at_once(pf3):
    """2^51 indices take about two seconds, and 2^52 four; one call behind the
    other, while the first still runs."""
    import torch
    A = inputs.uniform_matrix(7303, 53)
    dA, out = torch.from_numpy(A).cuda(), torch.zeros((2, 3), dtype=torch.int64, device="cuda")
    counts(pf3, A, 0, 1 << 30)
    t0 = time.perf_counter()
    for k in range(2):
        pf3.perm_f3_range_counts_async(dA, 53, 0, (1 << (51 + k)) - 1, out[k], torch.cuda.current_stream())
    returned = time.perf_counter() - t0
    torch.cuda.synchronize()
    done = time.perf_counter() - t0
    assert returned < 0.25 and done > 4 * returned, (returned, done)
    p, m, r = out[1].tolist()
    assert r == pf3.perm_from_counts(53, p, m) and p > out[0, 0] > 0
