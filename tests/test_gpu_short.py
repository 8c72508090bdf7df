"""Ranges of fewer than 2^24 - 1 Gray indices are stepped in full by as many
threads as there are: exact counts against the oracle for whole matrices of
every small n, single indices, ranges that start and end anywhere inside a run
of 8 or a thread's share, the top of the 64-bit index space, one and two words,
and matrices of mostly nonzero terms."""
import numpy as np
import pytest

from paper_2407_20205_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf3():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_20205_gb300 import binding
    return binding


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 9, 13, 20, 24, 32, 33, 64])
def test_counts_vs_oracle(pf3, oracle, n):
    import torch
    rng = np.random.default_rng(n)
    top = (1 << n) - 1
    ranges = [(0, min(top, (1 << 20) + 5)), (0, 0), (top, top), (max(0, top - 5000), top)]
    for _ in range(6):
        a = int(rng.integers(0, min(top, 1 << 62) + 1))
        ranges.append((a, min(top, a + int(rng.integers(0, 70000)))))
    if n in (24, 33):
        ranges.append((1 << 10, (1 << 10) + (1 << 24) - 3))  # the longest: 2^24 - 2 indices
    for A in (inputs.uniform_matrix(n, n), inputs.ones_matrix(n)):
        dA = torch.from_numpy(A).cuda()
        for a, b in ranges:
            out = torch.zeros(3, dtype=torch.int64, device="cuda")
            if b > top:
                continue
            pf3.perm_f3_range_counts_async(dA, n, a, b, out, None)
            torch.cuda.synchronize()
            got = [int(x) % (1 << 64) for x in out.cpu()]
            want = oracle.ryser_range_par(np.ascontiguousarray(A.T), a, b)
            assert tuple(got[:2]) == want, (a, b)
            assert got[2] == pf3.perm_from_counts(n, *want)
