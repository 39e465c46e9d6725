"""Eigenvalues of matrices whose blocks do not couple keep each block's own accuracy, however far apart their scales are.

Tolerance: a Sturm count is exact for a matrix within a few last places of each entry, and the bracket ends at two last
places of its ends, so an eigenvalue of a 1 x 1 block is off by at most 2^-50 of itself, one of a 2 x 2 block by 2^-48 of
the block's norm; an exact zero comes back below the bracket's floor of 2^-300 of the matrix's norm.
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


# the three reductions: blocks of 8, of 16, device memory
@pytest.mark.parametrize("n", [2, 3, 9, 40, 120, 640])
@pytest.mark.parametrize("blocks", [1, 2])
def test_eigenvalues_of_blocks_far_apart(tp, n, blocks):
    ctx = tp.Context(0)
    rng = np.random.default_rng(n + blocks)
    C = np.zeros((n, n))
    want, tol = [], []
    i = 0
    while i < n:
        s = 2.0 ** -(8 * int(rng.integers(0, 32))) if i else 1.0
        if blocks == 2 and i + 1 < n and rng.random() < 0.7:
            C[i, i] = C[i + 1, i + 1] = 2.0 * s
            C[i, i + 1] = C[i + 1, i] = s
            want += [s, 3.0 * s]
            tol += [3.0 * s * 2.0 ** -48] * 2
            i += 2
        else:
            v = 0.0 if i and rng.random() < 0.1 else s * float(rng.choice([-1.0, 1.0])) * (1.0 + rng.random())
            C[i, i] = v
            want.append(v)
            tol.append(max(abs(v) * 2.0 ** -50, 2.0 ** -299))
            i += 1
    o = np.argsort(want, kind="stable")
    want, tol = np.array(want)[o], np.array(tol)[o]
    w = ctx.tpcf_eigvalsh(torch.from_numpy(C).to("cuda:0")).cpu().numpy()
    assert ctx.tpcf_sync() == tp.TPCF_OK
    assert np.all(np.abs(w - want) <= tol), np.max(np.abs(w - want) / tol)
    ctx.close()
