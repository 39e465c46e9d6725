"""Gathered projection and the shared-memory eigenvalue reduction at the edges of their ranges.

Tolerances: a projection is one sum of at most n products in float64, so it is within n 2^-53 sum |P x| of the exact
sum, as is numpy's; eigenvalues carry the backward error of the Householder reduction, about n 2^-53 ||C||, on both
sides (a factor 8 covers the constants).
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


@pytest.fixture(scope="module")
def ctx(tp):
    c = tp.Context(0)
    yield c
    c.close()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


# entries per row around the gathered path's 32, outputs and mocks around the 32 x 32 blocks, bins around the 256 that
# are loaded at a time
@pytest.mark.parametrize("n_out,n_mock,nbin,entries", [(1, 1, 1, 1), (31, 33, 32, 5), (32, 32, 255, 32),
                                                       (33, 31, 256, 33), (65, 40, 257, 31), (40, 100, 600, 0)])
def test_project_gathered(tp, ctx, n_out, n_mock, nbin, entries):
    rng = np.random.default_rng(n_out)
    P = np.zeros((n_out, nbin))
    for o in range(n_out):
        k = rng.choice(nbin, size=min(nbin, max(0, entries - (o % 3 if o else 0))), replace=False)
        P[o, k] = rng.standard_normal(len(k))
    x = rng.standard_normal((n_mock, nbin))
    tol = 2.0 * nbin * 2.0 ** -53 * (np.abs(x) @ np.abs(P).T) + 1e-300
    assert np.all(np.abs(ctx.tpcf_project(_dev(P), _dev(x)).cpu().numpy() - x @ P.T) <= tol)
    # a row with a NaN or an infinity spreads as in the full sum (0 inf = NaN)
    x[n_mock // 2, nbin // 2] = np.inf
    x[0, 0] = np.nan
    y = ctx.tpcf_project(_dev(P), _dev(x)).cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = np.array([[np.sum(P[o] * x[m]) for o in range(n_out)] for m in range(n_mock)])
    assert np.array_equal(np.isnan(y), np.isnan(ref))
    ok = np.isfinite(ref)
    assert np.all(np.abs(y[ok] - ref[ok]) <= tol[ok])


# either side of the change from 8 to 16 blocks and of the largest matrix in shared memory; odd remainders of the
# rows per block; matrices with multiple eigenvalues, an exact zero, wide ranges and none but zeros
@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 8, 9, 95, 96, 97, 113, 628, 629])
@pytest.mark.parametrize("kind", ["cov", "multiple", "diagonal", "zero"])
def test_eigvalsh_edges(tp, ctx, n, kind):
    rng = np.random.default_rng(n)
    if kind == "cov":
        a = rng.standard_normal((2 * n, n)) * np.geomspace(1e-3, 1.0, n)
        C = a.T @ a
    elif kind == "multiple":
        q, _ = np.linalg.qr(rng.standard_normal((n, n)))
        w = np.where(np.arange(n) < n // 2, 2.0, 1.0)
        C = (q * w) @ q.T
    elif kind == "diagonal":
        C = np.diag(np.arange(n) * 2.0 ** -30)
    else:
        C = np.zeros((n, n))
    C = 0.5 * (C + C.T)
    w = ctx.tpcf_eigvalsh(_dev(C)).cpu().numpy()
    assert ctx.tpcf_sync() == tp.TPCF_OK
    ref = np.linalg.eigvalsh(C)
    assert np.all(np.diff(w) >= 0.0)
    assert np.max(np.abs(w - ref)) <= 8.0 * n * 2.0 ** -53 * np.max(np.abs(ref))


@pytest.mark.parametrize("n", [1, 2, 3, 40, 120, 629])
def test_eigvalsh_not_finite(tp, ctx, n):
    """A NaN or an infinity in the matrix gives NaN eigenvalues, as on a matrix of NaNs."""
    rng = np.random.default_rng(n)
    a = rng.standard_normal((2 * n, n))
    for value in (np.nan, np.inf):
        for at in ((n - 1, n - 1), (0, n - 1), slice(None)):
            C = a.T @ a
            C[at] = value
            if isinstance(at, tuple):
                C[at[::-1]] = value
            assert np.all(np.isnan(ctx.tpcf_eigvalsh(_dev(C)).cpu().numpy())), (value, at)


def test_eigvalsh_of_a_diagonal_far_below_its_norm(tp, ctx):
    """Entries 2^-80 of a diagonal matrix's norm come back to 2^-88 of the norm (e^2 is held above 2^-180)."""
    d = np.array([1.0, 0.0, 2.0 ** -80, 2.0 ** -80, 3.0 * 2.0 ** -80, 0.0, 0.5, 2.0 ** -40])
    w = ctx.tpcf_eigvalsh(_dev(np.diag(d))).cpu().numpy()
    assert np.max(np.abs(w[:5] - np.sort(d)[:5])) <= 2.0 ** -88
