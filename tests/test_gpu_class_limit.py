"""The class limit (widest merged matrix counted by characters) decides which
route a call takes, for device-pointer calls and batches too, also when it
changes between two calls on the same buffers.  The residues and counts are
the same on both routes, so the routes are told apart by their times: a 36 x 36
matrix of 6 or 8 merged columns is counted by characters in tens of
microseconds and met, with a twelfth and a twenty-fifth of its terms nonzero,
in milliseconds."""
import numpy as np
import pytest

from test_gpu_group_classes import few_columns, pf3  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu

N = 36


def timed(f):
    import torch
    best = float("inf")
    for _ in range(3):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def test_batch_on_the_same_buffers_follows_the_limit(pf3):  # noqa: F811
    import torch
    As = torch.from_numpy(np.concatenate([few_columns(5500 + k, N, 8).ravel() for k in range(4)])).cuda()
    ns = np.full(4, N, np.int32)
    res, hist = torch.zeros(4, dtype=torch.uint8, device="cuda"), torch.zeros(3, dtype=torch.int64, device="cuda")

    def call():
        pf3.perm_f3_batch_async(As, ns, res, hist, torch.cuda.current_stream())
        return res

    first = call().tolist()
    by_characters = timed(call)
    pf3.set_class_limit(0)
    try:
        assert call().tolist() == first
        met = timed(call)
    finally:
        pf3.set_class_limit(pf3.CLASS_MAX_COLS)
    assert call().tolist() == first
    again = timed(call)
    assert met > 3 * by_characters and met > 3 * again, (by_characters, met, again)


@pytest.mark.parametrize("limit,by_characters", [(8, True), (6, True), (5, False), (1, False), (0, False)])
def test_device_call_keeps_a_limit_below_the_default(pf3, limit, by_characters):  # noqa: F811
    """6 merged columns: counted by characters from a limit of 6 on."""
    import torch
    A = few_columns(5600, N, 6)
    dA = torch.from_numpy(np.ascontiguousarray(A)).cuda()  # few_columns gives column-major bytes
    out = torch.zeros(3, dtype=torch.int64, device="cuda")
    want = pf3.perm_f3_counts(A)

    def call():
        pf3.perm_f3_range_counts_async(dA, N, 0, (1 << N) - 1, out, torch.cuda.current_stream())

    fast = timed(call)
    pf3.set_class_limit(limit)
    try:
        t = timed(call)
    finally:
        pf3.set_class_limit(pf3.CLASS_MAX_COLS)
    assert tuple(out.tolist()[:2]) == want
    assert (t < 3 * fast) == by_characters, (t, fast)
