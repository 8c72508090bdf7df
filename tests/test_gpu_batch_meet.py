"""Batches of 18 <= n <= 32 take the kernel that meets low and high subsets in
Glynn's half sum: the residues are perm(A) mod 3 (exact), at both ends of each
of its two splits (18, 22 and 23, 24), where a matrix is cut into shares (25,
32) and just outside (17, and 33 and 36, which run in launch sequences of several), for uniform matrices and for matrices whose
subsets crowd into few classes."""
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


def family(n, seed):
    """Uniform, sparse, zero row / column, repeated columns, rank one,
    mostly nonzero, monomial, permuted triangular, partly monomial."""
    out = [inputs.uniform_matrix(seed, n, k) for k in range(3)]
    out.append(inputs.sparse_matrix_from_stream(inputs.Stream(seed, 7), n))
    Z = inputs.uniform_matrix(seed, n, 8)
    Z[:, 0] = 0
    out.append(Z)
    Z = inputs.uniform_matrix(seed, n, 9)
    Z[:n // 2] = Z[0]
    out.append(Z)
    out.append(inputs.pooled_columns(seed, n, 3, 2))
    out.append(inputs.ones_matrix(n))
    out.append(((np.ones((n, n)) + np.eye(n)) % 3).astype(np.uint8))
    st = inputs.Stream(seed, 10)
    out.append(inputs.monomial(st, n))
    # rows and columns with a single nonzero entry, alone and one after another
    T = np.triu(inputs.uniform_matrix(seed, n, 11))
    np.fill_diagonal(T, 1 + np.arange(n) % 2)
    out.append(inputs.f3_matmul(inputs.f3_matmul(inputs.monomial(st, n), T), inputs.monomial(st, n)))
    D = inputs.block_diag(inputs.monomial(st, n // 2), inputs.uniform_matrix(seed, n - n // 2, 12))
    D[n // 2:, :3] = inputs.uniform_matrix(seed, n, 13)[n // 2:, :3]
    out.append(D)
    return out


@pytest.mark.parametrize("n", [17, 18, 19, 22, 23, 24])
def test_residues_vs_oracle(pf3, oracle, n):
    mats = family(n, 4000 + n)
    if n > 22:
        mats = mats[:4] + mats[-3:]
    assert list(pf3.perm_f3_batch(mats)) == list(oracle.perm_batch(mats))


@pytest.mark.parametrize("n", [23, 24, 25, 28, 32, 33, 36])
def test_residues_vs_single_matrix_counts(pf3, n):
    mats = family(n, 4100 + n)
    want = [pf3.perm_from_counts(n, *pf3.perm_f3_counts(A)) for A in mats]
    assert list(pf3.perm_f3_batch(mats)) == want


def test_mixed_sizes_bad_entry_and_histogram(pf3):
    """Sizes from all routes in an order that mixes them, one bad entry in a
    whole and one in a cut matrix (device call: 255, not counted), the same
    buffers with new contents."""
    import torch
    ns = [24, 3, 26, 19, 12, 33, 22, 17, 24, 26, 0, 32, 23]
    for seed in (1, 2):
        mats = [inputs.uniform_matrix(4200 + seed, n, k) if n else np.zeros((0, 0), np.uint8)
                for k, n in enumerate(ns)]
        flat, nsa = pf3.pack_batch(mats)
        want = [pf3.perm_f3(A) for A in mats]
        if seed == 1:
            dA = torch.from_numpy(flat).cuda()
            res = torch.zeros(len(ns), dtype=torch.uint8, device="cuda")
            hist = torch.zeros(3, dtype=torch.int64, device="cuda")
        else:
            off = np.concatenate([[0], np.cumsum(nsa.astype(np.int64) ** 2)])
            flat[off[0] + 5] = 3
            flat[off[9] + 600] = 200
            want[0] = want[9] = 255
            dA.copy_(torch.from_numpy(flat))
        pf3.perm_f3_batch_async(dA, nsa, res, hist, torch.cuda.current_stream())
        torch.cuda.synchronize()
        assert res.cpu().tolist() == want
        assert hist.cpu().tolist() == [want.count(v) for v in range(3)]


def test_one_size_and_reordered_batches_agree(pf3):
    """A batch of one size is planned without tables; the same matrices among
    others are not."""
    mats = [inputs.uniform_matrix(4300, 20, k) for k in range(700)]
    alone = pf3.perm_f3_batch(mats)
    other = pf3.perm_f3_batch([inputs.uniform_matrix(4301, 21)] + mats)
    assert list(alone) == list(other[1:])


@pytest.mark.parametrize("chunk_log2,budget_log2", [(22, 22), (23, 33), (26, 28), (36, 30)])
def test_serving_items_shorter_and_longer_than_a_unit(pf3, chunk_log2, budget_log2):
    """A unit runs once the work items issued so far cover it: items of a
    quarter unit, half a unit, several units, a whole request; launches of one
    item; requests of one and two words, merged columns among them."""
    mats = [inputs.uniform_matrix(4400, n, n) for n in (17, 18, 22, 23, 24, 25, 27, 30, 33, 34)]
    mats.append(inputs.pooled_columns(4401, 33, 6, 4))
    mats.append(inputs.sparse_matrix_from_stream(inputs.Stream(4402, 0), 33))
    want = [pf3.perm_f3(A) for A in mats]
    with pf3.ServeContext(chunk_log2=chunk_log2, launch_budget=1 << budget_log2, max_jobs=5) as ctx:
        tickets = [ctx.submit(A) for A in mats]
        assert [ctx.wait(t) for t in tickets] == want


@pytest.mark.parametrize("n", [0, 1, 2, 3, 4, 5, 9, 10, 11, 12, 15, 16, 17])
def test_small_sizes_vs_oracle(pf3, oracle, n):
    """One to 32 lanes per matrix: batches of one size that leave lanes and
    warps of the last unit idle, alone and among other sizes."""
    count = {16: 5, 17: 3}.get(n, 67)
    mats = list(inputs.uniform_matrices(4500 + n, n, count))
    if n > 2:
        mats[0][:] = np.eye(n)
        mats[1][:] = 1
    want = list(oracle.perm_batch(mats))
    assert list(pf3.perm_f3_batch(mats)) == want
    other = [inputs.uniform_matrix(4600, k % 7 + 1, k) for k in range(40)]
    both = [x for pair in zip(mats, other + other) for x in pair]
    got = list(pf3.perm_f3_batch(both))
    assert got[::2] == want[:len(both) // 2]
    assert got[1::2] == list(oracle.perm_batch(both[1::2]))


def test_host_batch_with_a_bad_entry_leaves_outputs_alone(pf3):
    import ctypes
    flat, ns = pf3.pack_batch([inputs.uniform_matrix(4700, n) for n in (5, 20, 33)])
    flat[26] = 3
    res, hist = np.full(3, 77, np.uint8), np.full(3, 77, np.uint64)
    rc = pf3._lib_batch(flat.ctypes.data_as(pf3._u8p), ns.ctypes.data_as(pf3._i32p), 3, res.ctypes.data_as(pf3._u8p),
                        hist.ctypes.data_as(pf3._u64p))
    assert rc == pf3.PF3_EDOMAIN
    assert (res == 77).all() and (hist == 77).all()


@pytest.mark.parametrize("n,count", [(31, 18), (32, 16), (34, 10), (39, 2)])
def test_several_large_matrices_in_one_sequence(pf3, n, count):
    """Sequences of as many matrices as fit and a rest: a bad entry, matrices
    of few columns (counted by characters) and known answers among them."""
    import torch
    mats = [inputs.uniform_matrix(4300 + n, n, k) for k in range(count)]
    mats[-1] = inputs.pooled_columns(4301, n, 3, 2)
    if count > 4:
        mats[1], mats[2] = np.eye(n, dtype=np.uint8), inputs.pooled_columns(4302, n, 11, 2)
        mats[4] = inputs.sparse_matrix_from_stream(inputs.Stream(4303, 7), n)
    want = [pf3.perm_from_counts(n, *pf3.perm_f3_counts(A)) for A in mats]
    if count > 4:
        mats[3][5, 6] = 3
        want[3] = 255
    flat = torch.from_numpy(np.concatenate([A.ravel() for A in mats])).cuda()
    res = torch.zeros(count, dtype=torch.uint8, device="cuda")
    hist = torch.zeros(3, dtype=torch.int64, device="cuda")
    for _ in range(2):  # the second time with the scratch as the first left it
        hist.zero_()
        pf3.perm_f3_batch_async(flat, np.full(count, n, np.int32), res, hist, torch.cuda.current_stream())
        torch.cuda.synchronize()
        assert res.tolist() == want
        assert hist.tolist() == [want.count(r) for r in range(3)]


@pytest.mark.parametrize("class_max_cols", [0, 8])
def test_serving_large_requests_as_a_whole(pf3, class_max_cols):
    """Requests on both sides of 33 and 40 rows, several of one size, some with
    merged columns (walked when class_max_cols is 0) and known answers among
    them, submitted at once and twice."""
    mats = [inputs.uniform_matrix(4400 + n, n, k) for n in (32, 33, 36) for k in range(3)]
    mats += [inputs.uniform_matrix(4500, 40), inputs.pooled_columns(4501, 41, 20, 4), inputs.pooled_columns(4502, 38, 5, 2),
             np.eye(35, dtype=np.uint8), inputs.sparse_matrix_from_stream(inputs.Stream(4503, 7), 37),
             inputs.uniform_matrix(4504, 14), inputs.pooled_columns(4505, 34, 17, 2)]
    want = [pf3.perm_f3(A) for A in mats]
    with pf3.ServeContext(class_max_cols=class_max_cols) as ctx:
        for _ in range(2):
            tickets = [ctx.submit(A) for A in mats]
            assert [ctx.wait(t) for t in tickets] == want
