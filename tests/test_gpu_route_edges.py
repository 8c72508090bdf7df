"""Calls on both sides of the lines between the routes: single ranges at 2^24 and
2^27 indices, batches at n = 17 / 18 and 30 / 31 and the most shares a matrix
is cut into (n = 29, 30)."""
import numpy as np
import pytest

from paper_2407_20205_gb300 import inputs
from test_gpu_batch_meet import family
from test_gpu_meet import KINDS, by_pieces, counts, matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf3():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_20205_gb300 import binding
    return binding


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [28, 36, 64])
def test_shortest_met_ranges_equal_the_walk(pf3, kind, n):
    A = matrix(kind, n)
    first = 12345 if n == 28 else (1 << (n - 1)) - 98765
    for length in ((1 << 27) - 1, 1 << 27, (1 << 27) + 1, (1 << 28) - 77):
        last = min(first + length, 1 << n) - 1
        assert counts(pf3, A, first, last) == by_pieces(pf3, A, first, last, 1 << 25), length


def test_shortest_met_range_vs_oracle(pf3, oracle):
    A = matrix("uniform", 30)
    first = (1 << 29) + 4321
    for length in ((1 << 24) - 1, 1 << 24, (1 << 24) + 1, 1 << 27):
        want = oracle.ryser_range_par(np.ascontiguousarray(A.T), first, first + length - 1)
        assert counts(pf3, A, first, first + length - 1) == want, length


@pytest.mark.parametrize("n", [29, 30, 31])
def test_residues_at_the_upper_end(pf3, n):
    mats = family(n, 4800 + n)
    want = [pf3.perm_from_counts(n, *pf3.perm_f3_counts(A)) for A in mats]
    assert list(pf3.perm_f3_batch(mats)) == want


def test_sizes_of_all_routes_in_one_batch(pf3):
    ns = [30, 31, 17, 18, 29, 30, 31, 16, 32, 18, 30]
    mats = [inputs.uniform_matrix(4900, n, k) for k, n in enumerate(ns)]
    want = [pf3.perm_from_counts(n, *pf3.perm_f3_counts(A)) for n, A in zip(ns, mats)]
    res, hist = pf3.perm_f3_batch(mats, with_hist=True)
    assert list(res) == want and [int(h) for h in hist] == [want.count(v) for v in range(3)]
