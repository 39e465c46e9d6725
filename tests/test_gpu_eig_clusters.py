"""Eigenvalues on a device that runs no cluster of 16 blocks: the 8-block reduction, or device memory where the matrix does
not fit in eight blocks, in place of a launch that would fail.

Tolerance: the backward error of the reduction on both sides, as in the other eigenvalue tests.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2205_11852_gb300 as tp
    return tp


# either side of the change to 16 blocks, the largest orders of 8 and of 16 blocks
@pytest.mark.parametrize("n", [2, 95, 96, 120, 457, 460, 628, 640])
@pytest.mark.parametrize("limit", [None, 16, 15, 8])
def test_eigenvalues_without_large_clusters(tp, n, limit, monkeypatch):
    if limit is not None:
        monkeypatch.setenv("TPCF_TEST_MAX_CLUSTER", str(limit))
    ctx = tp.Context(0)
    a = np.random.default_rng(n).standard_normal((2 * n, n))
    C = a.T @ a
    w = ctx.tpcf_eigvalsh(torch.from_numpy(C).to("cuda:0")).cpu().numpy()
    assert ctx.tpcf_sync() == tp.TPCF_OK
    ref = np.linalg.eigvalsh(C)
    assert np.max(np.abs(w - ref)) <= 8.0 * n * 2.0 ** -53 * np.max(np.abs(ref))
    ctx.close()
