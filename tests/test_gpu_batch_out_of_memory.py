"""A batch for which the device has no room is refused with PF3_ENOMEM, and
the next calls work."""
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


def test_calls_after_a_batch_that_does_not_fit(pf3, oracle):
    import torch
    mats = [inputs.uniform_matrix(7200, n, k) for k in range(3) for n in (5, 12, 20)]
    want = list(oracle.perm_batch(mats))
    assert list(pf3.perm_f3_batch(mats)) == want
    count = 1 << 18  # matrices of 4096 bytes: 1 GiB
    ns = np.full(count, 64, np.int32)
    flat = np.zeros(count * 4096, np.uint8)
    torch.cuda.empty_cache()
    # all of the device but 512 MiB, left untouched
    held = torch.empty(torch.cuda.mem_get_info()[0] - (512 << 20), dtype=torch.uint8, device="cuda")
    try:
        for _ in range(2):
            with pytest.raises(pf3.PF3Error) as e:
                pf3.perm_f3_batch(flat=flat, ns=ns)
            assert e.value.code == pf3.PF3_ENOMEM
            assert list(pf3.perm_f3_batch(mats)) == want
    finally:
        del held
        torch.cuda.empty_cache()
    assert list(pf3.perm_f3_batch(mats)) == want
