"""The work-item kernel, every variant of it.  Batches are no longer planned as
work items; serving still walks requests so, all of them when the items are
shorter than 2^22 indices: matrices walked whole, in many pieces, by one lane,
on one and two plane words, with merged columns, and on both sides of the
switch to the dense walk."""
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


@pytest.fixture(scope="module")
def requests(pf3, oracle):
    small = [inputs.uniform_matrix(8100 + k, n) for k, n in enumerate((1, 3, 5, 9, 10, 12, 13, 17, 20, 22))]
    small += [np.ones((18, 18), np.uint8), np.eye(16, dtype=np.uint8),
              ((np.ones((19, 19)) + np.eye(19)) % 3).astype(np.uint8)]
    large = [inputs.uniform_matrix(8200 + k, n) for k, n in enumerate((26, 31, 33, 34))]
    large += [inputs.pooled_columns(8300, 33, 6, 4), inputs.pooled_columns(8301, 34, 3, None),
              inputs.pooled_columns(8302, 33, 17, 2), inputs.sparse_matrix_from_stream(inputs.Stream(8303, 7), 33)]
    return small + large, list(oracle.perm_batch(small)) + [pf3.perm_f3(A) for A in large]


@pytest.mark.parametrize("chunk_log2", [13, 18, 21])
def test_every_variant(pf3, requests, chunk_log2):
    mats, want = requests
    keep = {W: pf3.get_variant(pf3.BATCH, W) for W in (1, 2)}
    try:
        for v in range(pf3.variant_count(pf3.BATCH)):
            for W in (1, 2):
                pf3.set_variant(pf3.BATCH, W, v)
            with pf3.ServeContext(chunk_log2=chunk_log2, class_max_cols=0) as ctx:
                tickets = [ctx.submit(A) for A in mats]
                assert [ctx.wait(t) for t in tickets] == want, v
                assert ctx.stats()["items"] >= len(mats) + (4 << (33 - max(chunk_log2, 14)))
    finally:
        for W in (1, 2):
            pf3.set_variant(pf3.BATCH, W, keep[W])
