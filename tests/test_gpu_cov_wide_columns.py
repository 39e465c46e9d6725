"""Float64 covariances of columns whose residuals differ widely in size, element by element.

Reference: sums of the residuals' products in extended precision.  Tolerance per element, with S = sum |y_i y_j|: a
float64 sum in two levels (chains of eight products, three additions, one compensated addition per 32 mocks) is within
12 x 2^-53 S, the residuals' own rounding adds 2 x 2^-53 S, the factor's and the combination's roundings 4, and
means off by d_i (their sums' rounding, at most 64 steps of 2^-53 mean |x| each) add n d_i d_j.
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


def _columns(kind, n, nb, rng):
    x = rng.standard_normal((n, nb))
    if kind.startswith("outliers"):       # two pairs of +- one size, in mocks of their own where there are enough
        for c in range(nb):
            at = (4 * c + np.arange(4)) % n
            x[at, c] = float(kind[8:]) * np.array([1.0, -1.0, 1.0, -1.0])
    elif kind.startswith("halves"):       # the large half of one column meets the small half of the next
        x = np.sign(x) * (1.0 + 0.1 * rng.random((n, nb)))
        x[:n // 2, ::2] *= 2.0 ** -int(kind[6:])
        x[n // 2:, 1::2] *= 2.0 ** -int(kind[6:])
    elif kind == "lognormal":
        x = np.exp(3.0 * x)
    elif kind == "rare":                  # a few events in an otherwise empty column
        x = np.where(rng.random((n, nb)) < 0.02, 1.0 + rng.random((n, nb)), 1e-4 * x)
    elif kind == "one":                   # one such column among ordinary ones
        x[:4, 5] = [1e8, -1e8, 1e8, -1e8]
    return x


@pytest.mark.parametrize("kind", ["outliers1e4", "outliers1e6", "outliers1e12", "halves6", "halves20", "lognormal", "rare",
                                  "one"])
@pytest.mark.parametrize("n,nb", [(5, 17), (33, 40), (400, 24), (1000, 70)])
def test_wide_columns(tp, ctx, kind, n, nb):
    x = _columns(kind, n, nb, np.random.default_rng(n + len(kind)))
    xl = x.astype(np.longdouble)
    y = xl - xl.mean(0)
    y = y - y.mean(0)
    G = y.T @ y
    S = np.abs(y).T @ np.abs(y)
    d = 64.0 * 2.0 ** -53 * np.abs(x).mean(0)
    tol = (18.0 * 2.0 ** -53 * S + n * np.outer(d, d)) / (n - 1)
    got = ctx.tpcf_sample_cov(_dev(x), tp.TPCF_FP64).cpu().numpy()
    assert np.array_equal(got, got.T)
    assert np.all(np.abs(got - G / (n - 1)) <= tol)
    lc = ctx.tpcf_lc_cov(_dev(x), _dev(x), _dev(x), 1, 50.0, tp.TPCF_FP64)
    for key in ("Ca", "Cb"):
        assert np.all(np.abs(lc[key].cpu().numpy() - G / (n - 1)) <= tol), key
    assert ctx.tpcf_sync() == tp.TPCF_OK


# either side of the few mocks and many bins that stay on the tiled float64 kernel
@pytest.mark.parametrize("n,nb", [(2, 1001), (3, 1000), (3, 1001), (19, 1001), (20, 1001)])
def test_few_mocks_and_many_bins(tp, ctx, n, nb):
    x = np.random.default_rng(n + nb).standard_normal((n, nb))
    y = x - x.mean(0)
    S = np.abs(y).T @ np.abs(y) / (n - 1)
    d = 64.0 * 2.0 ** -53 * np.abs(x).mean(0)
    got = ctx.tpcf_sample_cov(_dev(x), tp.TPCF_FP64).cpu().numpy()
    assert np.all(np.abs(got - y.T @ y / (n - 1)) <= 2.0 * (18.0 + n) * 2.0 ** -53 * S + n * np.outer(d, d))
