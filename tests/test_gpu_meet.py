"""Long Gray ranges are counted by meeting low and high row subsets instead of
walking every index; the +1/-1 counts are the same integers (tolerance 0).
Each split of the range between low and high rows is compared with ranges
short enough for the walk or the next smaller split, at ragged ends, at the top
of the 64-bit index space, and for matrices whose subsets fall into few
classes (zero and repeated columns, zero rows, rank one)."""
import numpy as np
import pytest

from conftest import rank_one_counts
from paper_2407_20205_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf3():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_20205_gb300 import binding
    return binding


def counts(pf3, A, first, last):
    import torch
    dA = torch.from_numpy(np.ascontiguousarray(A)).cuda()
    out = torch.zeros(3, dtype=torch.int64, device="cuda")
    pf3.perm_f3_range_counts_async(dA, A.shape[0], first, last, out, None)
    torch.cuda.synchronize()
    p, m, r = (int(x) % (1 << 64) for x in out.cpu())
    assert r == pf3.perm_from_counts(A.shape[0], p, m)
    return p, m


def by_pieces(pf3, A, first, last, piece):
    total = [0, 0]
    while first <= last:
        stop = min(last, first + piece - 1)
        for k, x in enumerate(counts(pf3, A, first, stop)):
            total[k] += x
        first = stop + 1
    return tuple(total)


def matrix(kind, n):
    A = inputs.uniform_matrix(900 + n, n)
    if kind == "zero column":
        A[:, 1] = 0
    elif kind == "zero rows":
        A[:20] = 0
    elif kind == "few columns":
        A = inputs.pooled_columns(901, n, 5, 4)
    elif kind == "sparse":
        A = inputs.sparse_matrix_from_stream(inputs.Stream(902, n), n)
    elif kind == "mostly nonzero":
        A = ((np.ones((n, n)) + np.eye(n)) % 3).astype(np.uint8)  # distinct columns, a third of the terms nonzero
    return A


KINDS = ["uniform", "zero column", "zero rows", "few columns", "sparse", "mostly nonzero"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [30, 33, 48, 64])
def test_shortest_ranges_equal_the_walk(pf3, kind, n):
    """2^29 indices and a little more, ragged at both ends, against ranges of
    2^26 that are walked."""
    A = matrix(kind, n)
    first = 12345 if n == 30 else (1 << (n - 1)) - 98765
    last = first + (1 << 29) + 4321
    assert counts(pf3, A, first, last) == by_pieces(pf3, A, first, last, 1 << 26)


@pytest.mark.parametrize("n,log2", [(31, 31), (40, 34), (64, 37)])
def test_larger_splits_equal_the_smaller(pf3, n, log2):
    A = matrix("sparse", n)
    if n == 64:
        A = inputs.pooled_columns(903, n, 20, 8)
    first, last = (0, (1 << n) - 1) if n == 31 else ((1 << 39) + 7, (1 << 39) + (1 << log2) + 99)
    if n == 64:
        first, last = (1 << 64) - (1 << log2) - 3, (1 << 64) - 1
    got = counts(pf3, A, first, last)
    assert sum(got) > 0
    assert got == by_pieces(pf3, A, first, last, 1 << (log2 - 2))


@pytest.mark.parametrize("n", [29, 32, 35, 38])
def test_rank_one_closed_form(pf3, n):
    rng = np.random.default_rng(n)
    d, e = rng.choice([1, -1], n), rng.choice([1, -1], n)
    A = ((d[:, None] * e[None, :]) % 3).astype(np.uint8)
    assert counts(pf3, A, 0, (1 << n) - 1) == rank_one_counts(d, e)


def test_against_the_oracle(pf3, oracle):
    A = matrix("uniform", 36)
    first, last = (1 << 33) + 17, (1 << 33) + (1 << 29) + 9000
    want = oracle.ryser_range_par(np.ascontiguousarray(A.T), first, last)
    assert sum(want) > 0 and counts(pf3, A, first, last) == want


def test_bad_entry_leaves_the_next_call_intact(pf3):
    import torch
    A = matrix("uniform", 34)
    B = A.copy()
    B[3, 4] = 7
    out = torch.zeros(3, dtype=torch.int64, device="cuda")
    pf3.perm_f3_range_counts_async(torch.from_numpy(B).cuda(), 34, 0, (1 << 34) - 1, out, None)
    torch.cuda.synchronize()
    assert [int(x) for x in out.cpu()] == [0, 0, -1]
    assert counts(pf3, A, 0, (1 << 30) - 1) == by_pieces(pf3, A, 0, (1 << 30) - 1, 1 << 26)


@pytest.mark.parametrize("n,pool", [(30, 1), (30, 4), (31, 7), (33, 11), (33, 13), (64, 6)])
def test_columns_merge_on_the_device(pf3, oracle, n, pool):
    """Device-pointer calls on a matrix of few distinct columns: counted by
    characters over the whole range, met on the merged columns over a part of
    it; a window of both equals the walk (of A as it is) and the whole the
    host call, which merges on the host."""
    A = inputs.pooled_columns(950 + n + pool, n, pool, pool)
    if n == 64:
        want = pf3.class_counts(A)
        assert want is None or counts(pf3, A, 0, (1 << 64) - 1) == want
        first = (1 << 63) + 12345
    else:
        got = counts(pf3, A, 0, (1 << n) - 1)
        assert got == pf3.perm_f3_counts(A)
        pf3.set_class_limit(0)  # no characters: the merged matrix is met
        try:
            assert counts(pf3, A, 0, (1 << n) - 1) == got
        finally:
            pf3.set_class_limit(pf3.CLASS_MAX_COLS)
        first = 54321
    last = first + (1 << 29) + 77
    assert counts(pf3, A, first, last) == by_pieces(pf3, A, first, last, 1 << 26)


@pytest.mark.parametrize("log2,L,K", [(29, 16, 7), (31, 17, 8), (34, 19, 9), (37, 20, 10), (39, 22, 11)])
def test_classes_of_every_size(pf3, log2, L, K):
    """Low rows with few entries in the class columns: classes from a handful
    of low subsets (words that repeat over the lanes, 8 or 16 of them) to
    thousands (joined by a whole thread block, many units each)."""
    n = 50
    A = inputs.uniform_matrix(77, n)
    A[:L, :K] *= (np.random.default_rng(5).random((L, K)) < 0.2).astype(np.uint8)
    first = (1 << 45) + 1001
    last = first + (1 << log2) + 5
    assert counts(pf3, A, first, last) == by_pieces(pf3, A, first, last, 1 << (log2 - 2))
