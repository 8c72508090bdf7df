"""Matrices of 50 rows and more in a batch take more than 64 launch sequences
each and run behind the batch's captured launches instead of in them."""
import subprocess
import sys

import numpy as np
import pytest

from conftest import ROOT
from paper_2407_20205_gb300 import inputs
from test_gpu_meet import by_pieces

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf3():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_20205_gb300 import binding
    return binding


def test_among_others_and_again(pf3):
    import torch
    ns = np.array([50, 12, 33, 49, 50, 24, 0], np.int32)
    res, hist = torch.zeros(len(ns), dtype=torch.uint8, device="cuda"), torch.zeros(3, dtype=torch.int64, device="cuda")
    dA = torch.zeros(int((ns.astype(np.int64) ** 2).sum()), dtype=torch.uint8, device="cuda")
    for seed in (1, 2):
        mats = [inputs.uniform_matrix(7400 + seed, int(n), k) if n else np.zeros((0, 0), np.uint8)
                for k, n in enumerate(ns)]
        want = [pf3.perm_f3(A) for A in mats]
        # one of the 50 x 50 from its exact counts over short ranges
        assert want[0] == pf3.perm_from_counts(50, *by_pieces(pf3, mats[0], 0, (1 << 50) - 1, 1 << 47))
        if seed == 2:
            mats[4][0, 0], want[4] = 200, 255
        dA.copy_(torch.from_numpy(np.concatenate([A.ravel() for A in mats])))
        for _ in range(2):
            pf3.perm_f3_batch_async(dA, ns, res, hist, torch.cuda.current_stream())
            torch.cuda.synchronize()
            assert res.tolist() == want
            assert hist.tolist() == [want.count(v) for v in range(3)]
        if seed == 1:
            assert list(pf3.perm_f3_batch(mats)) == want


IN_A_NEW_PROCESS = """
import numpy as np, torch
from paper_2407_20205_gb300 import binding as pf3, inputs
dA = torch.from_numpy(inputs.uniform_matrix(7402, 53)).cuda()
res, hist = torch.zeros(1, dtype=torch.uint8, device="cuda"), torch.zeros(3, dtype=torch.int64, device="cuda")
stream = torch.cuda.current_stream()
pf3.perm_f3_batch_async(dA, np.array([33], np.int32), res, hist, stream)
pf3.perm_f3_range_counts_async(dA, 53, 0, 1 << 51, hist, stream)
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
pf3.perm_f3_batch_async(dA, np.array([53], np.int32), res, hist, stream)
torch.cuda.synchronize()
print(before - torch.cuda.mem_get_info()[0])
"""


def test_no_graph_of_thousands_of_nodes(pf3):
    """53 x 53: 1024 sequences, which as a graph take 6 MB of the device.  (Two
    kilobytes a node: 0.8 GB for a 60 x 60 and 13 GB for a 64 x 64.)"""
    out = subprocess.run([sys.executable, "-c", IN_A_NEW_PROCESS], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    assert int(out.stdout) < 4 << 20
