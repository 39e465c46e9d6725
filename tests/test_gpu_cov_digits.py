"""Float64 covariances on the tensor cores (exact digit splits) against the float64 oracle.

Tolerance: a residual of column i is rounded to 2^(e_i - 56) with 2^e_i <= 2 max |y_i|, so an element of the Gram
matrix is off by at most n 2^(e_i + e_j) 2^-55 + 2^-53 |G_ij| <= n 2^-53 max|y_i| max|y_j| + ..., and max|y_i|^2 <=
G_ii: normalised by sqrt(C_ii C_jj) the error is at most (n + 1) 2^-53; the oracle's own float64 sums have the same
bound, and so have the means.  4 (n + 1) 2^-53 covers all three.
"""
import numpy as np
import pytest

import oracle
import synth

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


def _norm_err(got, ref):
    d = np.sqrt(np.diag(ref))
    d[d == 0.0] = 1.0
    return float(np.max(np.abs(got - ref) / np.outer(d, d)))


# mocks: one slice and its edges, a full segment of 28 slices of 16 and one more mock, several segments; bins: one
# column block, the edges of the 16-column MMA width, of the 64-column and of the 128-row tiles
@pytest.mark.parametrize("n_mock,nbin", [(2, 1), (3, 15), (15, 16), (16, 17), (17, 63), (100, 64), (448, 65),
                                         (449, 127), (897, 128), (64, 129), (333, 193), (40, 321)])
def test_cov_digits_sizes(tp, ctx, n_mock, nbin):
    xs = synth.synthetic_xi_variants(61, n_mock, nbin)
    tol = 4.0 * (n_mock + 1) * 2.0 ** -53
    got = ctx.tpcf_lc_cov(*[_dev(x) for x in xs], 1, 50.0, tp.TPCF_FP64)
    ref = oracle.lc_cov(*xs, 1, 50.0)
    d = np.sqrt(np.diag(ref["Ca"]))
    for k, w in (("Ca", 1.0), ("Cb", 1.0), ("A", 3.0), ("B", 4.0), ("C_lc", 4.0)):   # weights of the combination
        g = got[k].cpu().numpy()
        assert np.array_equal(g, g.T), k
        assert float(np.max(np.abs(g - ref[k]) / np.outer(d, d))) <= w * tol, k
    s = ctx.tpcf_sample_cov(_dev(xs[2]), tp.TPCF_FP64).cpu().numpy()
    assert _norm_err(s, oracle.sample_cov(xs[2])) <= tol
    assert ctx.tpcf_sync() == tp.TPCF_OK


def test_cov_digits_extreme_columns(tp, ctx):
    """Largest digits in every level (full segments of +-(1 - 2^-53)), columns of very different scale, constant
    and zero columns, and columns that are summed in float64 directly: outside 2^+-400, NaN, infinities."""
    n, nb = 896, 40
    rng = np.random.default_rng(5)
    x = rng.normal(size=(n, nb))
    sign = np.where(np.arange(n) % 2 == 0, 1.0, -1.0)
    x[:, 0] = sign * (1.0 - 2.0 ** -53)
    x[:, 1] = sign * (64.0 / 128.0 + 64.0 / 128.0 ** 2 + 64.0 / 128.0 ** 3)
    x[:, 2] *= 2.0 ** 300
    x[:, 3] *= 2.0 ** -300
    x[:, 4] = 0.0
    x[:, 5] = 0.25
    x[:, 6] *= 2.0 ** -420       # below the split range: float64 sums
    x[:, 7] = np.where(np.arange(n) == 17, 2.0 ** 30, x[:, 7])   # one mock dominates the column
    tol = 4.0 * (n + 1) * 2.0 ** -53
    s = ctx.tpcf_sample_cov(_dev(x), tp.TPCF_FP64).cpu().numpy()
    ref = oracle.sample_cov(x)
    assert np.all(s[4] == 0.0) and np.all(s[:, 4] == 0.0) and np.all(s[5] == 0.0)
    assert _norm_err(s, ref) <= tol
    x[3, 8] = np.nan
    x[4, 9] = np.inf
    s = ctx.tpcf_sample_cov(_dev(x), tp.TPCF_FP64).cpu().numpy()
    bad = np.zeros((nb, nb), bool)
    bad[[8, 9]] = True
    bad[:, [8, 9]] = True
    assert np.all(np.isnan(s[bad]))
    ok = [i for i in range(nb) if i not in (8, 9)]
    assert _norm_err(s[np.ix_(ok, ok)], ref[np.ix_(ok, ok)]) <= tol


def test_cov_digits_without_room_for_the_workspace(tp, monkeypatch):
    """A failed allocation of the digit workspace leaves the call to the float64 kernel and its smaller one."""
    xs = synth.synthetic_xi_variants(62, 50, 30)
    monkeypatch.setenv("TPCF_TEST_FAIL_ALLOC", "1")
    ctx = tp.Context(0)
    monkeypatch.delenv("TPCF_TEST_FAIL_ALLOC")
    tol = 4.0 * 51 * 2.0 ** -53
    ref = oracle.lc_cov(*xs, 1, 50.0)
    d = np.sqrt(np.diag(ref["Ca"]))
    for _ in range(2):   # the float64 kernel, then the digits
        got = ctx.tpcf_lc_cov(*[_dev(x) for x in xs], 1, 50.0, tp.TPCF_FP64)["C_lc"].cpu().numpy()
        assert ctx.tpcf_sync() == tp.TPCF_OK
        assert float(np.max(np.abs(got - ref["C_lc"]) / np.outer(d, d))) <= 4.0 * tol
    ctx.close()
