"""Float64 covariances of columns whose scatter is far below their mean, against exact integer sums.

Entries are 1 + k 2^-g with integers k that sum to zero and g small enough for every partial sum to be exact in float64,
so the mean is exactly 1 and the residuals are exactly k 2^-g.  Tolerance: a float64 sum of n products is within
n 2^-53 sum |y_i y_j| of the exact one, the division by n - 1 and the factor's own rounding add 2^-52 |C|.
"""
import math

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


# a few mocks (two leave the finest grid), the edges of a slice of 16, and several segments of 448
@pytest.mark.parametrize("n", [2, 4, 16, 18, 64, 900])
@pytest.mark.parametrize("scatter", [25, 30, 36, 40, 45])
def test_scatter_far_below_the_mean(tp, ctx, n, scatter):
    g = 52 - math.ceil(math.log2(n)) if n > 2 else 52   # (two mocks: 1 + k and 1 - k)
    top = 2 ** (g - scatter)
    if top < 1:
        pytest.skip("the scatter is below the grid that keeps the mean exact")
    nb = 20
    rng = np.random.default_rng(n + scatter)
    k = rng.integers(-top, top + 1, size=(n // 2, nb))
    k = np.concatenate([k, -k])
    for c in range(nb):
        k[:, c] = k[rng.permutation(n), c]
    k[:, 3] = 0                                     # a constant column
    k[:2, 4], k[2:, 4] = (top, -top), 0             # the scatter in two mocks
    k[:2, 5], k[2:, 5] = (1, -1), 0
    x = 1.0 + k * 2.0 ** -g
    ko = k.astype(object)
    G = ko.T @ ko
    S = np.abs(ko).T @ np.abs(ko)
    want = np.array([[math.ldexp(float(v), -2 * g) for v in row] for row in G]) / (n - 1)
    tol = np.array([[math.ldexp(float(v), -2 * g) for v in row] for row in S]) / (n - 1) * (n + 3) * 2.0 ** -53
    got = ctx.tpcf_sample_cov(_dev(x), tp.TPCF_FP64).cpu().numpy()
    assert ctx.tpcf_sync() == tp.TPCF_OK
    assert np.all(np.abs(got - want) <= tol)
    lc = ctx.tpcf_lc_cov(_dev(x), _dev(x), _dev(x), 1, 50.0, tp.TPCF_FP64)
    for key in ("Ca", "Cb"):
        assert np.all(np.abs(lc[key].cpu().numpy() - want) <= tol), key


def test_two_neighbouring_numbers(tp, ctx):
    """{1, 1 + 2^-52}: the mean rounds to 1, the variance is 2^-104."""
    x = np.array([[1.0, 2.0], [1.0 + 2.0 ** -52, 5.0]])
    got = ctx.tpcf_sample_cov(_dev(x), tp.TPCF_FP64).cpu().numpy()
    assert got[0, 0] == 2.0 ** -104 and got[0, 1] == 1.5 * 2.0 ** -52 and got[1, 1] == 4.5


@pytest.mark.parametrize("n", [2, 40, 3500])
def test_zero_and_constant_columns(tp, ctx, n):
    """Columns of one value have zero covariance with every column, whatever the value's sign."""
    rng = np.random.default_rng(n)
    x = rng.standard_normal((n, 40))
    x[:, 7], x[:, 8], x[:, 9], x[:, 10] = 0.0, -0.0, 0.5, -2.0 ** -700
    got = ctx.tpcf_sample_cov(_dev(x), tp.TPCF_FP64).cpu().numpy()
    for c in (7, 8, 9, 10):
        assert np.all(got[c] == 0.0) and np.all(got[:, c] == 0.0), c
