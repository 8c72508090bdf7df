"""Large matrices of one size share a launch sequence; those whose columns
merge into few are counted by characters in it, by several thread blocks from
7 columns on.  Such matrices at every place of a group (the first one's words
of scratch are also the group's), groups of nothing else, with bad entries and
with uniform matrices, and the next call on the same scratch."""
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


def few_columns(seed, n, m):
    """n columns, signed copies of m random vectors, each an odd number of
    times: they merge into m (n - m even)."""
    g = np.random.default_rng(seed)
    mult = np.ones(m, int)
    for _ in range((n - m) // 2):
        mult[g.integers(m)] += 2
    cols = g.permutation(np.repeat(np.arange(m), mult))
    return (g.integers(0, 3, (m, n))[cols].T * g.integers(1, 3, n)[None, :] % 3).astype(np.uint8)


def layouts(n, ms):
    """Groups as lists of column counts (0: uniform, -1: an entry above 2)."""
    for m in ms:
        yield [m, m]
        yield [m, 0, 0]
        yield [m, -1]
        yield [0, m, 0, m]
    yield [ms[-1], ms[0], ms[-1], ms[0], -1]
    yield [ms[-1]] * 3 + [0] + [ms[0]]


@pytest.mark.parametrize("n,ms", [(31, (7, 9, 11)), (33, (7, 11)), (34, (8, 10, 12)), (38, (8, 12)), (39, (7,))])
def test_groups_with_few_column_matrices(pf3, n, ms):
    import torch
    U = inputs.uniform_matrix(5100 + n, n)
    dU = torch.from_numpy(U).cuda()
    last = (1 << 30) - 1
    out = torch.zeros(3, dtype=torch.int64, device="cuda")
    pf3.perm_f3_range_counts_async(dU, n, 0, last, out, None)
    torch.cuda.synchronize()
    before = out.tolist()
    stream = torch.cuda.current_stream()
    for layout in layouts(n, ms):
        mats = [few_columns(5200 + 64 * k + m, n, m) if m > 0 else inputs.uniform_matrix(5300 + n, n, k)
                for k, m in enumerate(layout)]
        pf3.set_class_limit(0)  # the reference: met, not counted by characters
        try:
            want = [pf3.perm_f3(A) for A in mats]
        finally:
            pf3.set_class_limit(pf3.CLASS_MAX_COLS)
        for k, m in enumerate(layout):
            if m < 0:
                mats[k][n - 1, 2] = 3
                want[k] = 255
        As = torch.from_numpy(np.concatenate([A.ravel() for A in mats])).cuda()
        ns = np.full(len(mats), n, np.int32)
        res = torch.empty(len(mats), dtype=torch.uint8, device="cuda")
        hist = torch.empty(3, dtype=torch.int64, device="cuda")
        for _ in range(4):
            res.fill_(77)
            hist.fill_(77)
            pf3.perm_f3_batch_async(As, ns, res, hist, stream)
            torch.cuda.synchronize()
            assert res.tolist() == want, layout
            assert hist.tolist() == [want.count(v) for v in range(3)], layout
            # the scratch is as a sequence expects it
            out.zero_()
            pf3.perm_f3_range_counts_async(dU, n, 0, last, out, None)
            torch.cuda.synchronize()
            assert out.tolist() == before, layout
