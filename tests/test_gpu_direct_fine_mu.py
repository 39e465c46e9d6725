"""Direct pair counter with one column per |mu| bin (fine mu bins along x) against the brute-force oracle (whole numbers).

The cases are its tables' edges: coincident and nearly coincident points (mu intervals wider than many bins, columns
below the table's first), pairs along and across the line of sight (first and last column), pairs beyond the last edge,
one table per block and two, and the largest binning that fits.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

L = 160.0


@pytest.fixture(scope="module")
def tp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2205_11852_gb300 as tp
    return tp


def _points(seed, n):
    rng = np.random.default_rng(seed)
    x = rng.random((n, 3)) * L
    c = np.mod(rng.random((5, 3))[rng.integers(0, 5, n)] * L + rng.normal(0.0, 3.0, (n, 3)), L)
    line = np.stack([np.linspace(1.0, 60.0, 24), np.full(24, 50.0), np.full(24, 70.0)], 1)     # along x: mu = 1
    out = np.concatenate([x, c, c[:30], np.mod(c[:30] + rng.normal(0.0, 1e-6, c[:30].shape), L), line, line[:, [1, 0, 2]]])
    out[out >= L] = 0.0
    return out


# two tables per block and one
@pytest.mark.parametrize("n_s,ds,n_mu", [(10, 5.0, 32), (30, 1.5, 40), (100, 0.5, 33),
                                                (200, 0.25, 100), (7, 7.0, 128)])
@pytest.mark.parametrize("geometry", ["periodic", "open"])
def test_direct_fine_mu_bins(tp, n_s, ds, n_mu, geometry):
    edges = ds * np.arange(n_s + 1)
    mocks = [(_points(3, 300), [_points(4, 250), _points(5, 333)]), (_points(6, 2), [_points(7, 30), _points(8, 20)])]
    geo_t, geo_o = (tp.TPCF_PERIODIC, oracle.PERIODIC) if geometry == "periodic" else (tp.TPCF_OPEN, oracle.OPEN)
    tb = tp.make_binning(edges, n_mu, geo_t, L)
    ob = oracle.Binning(edges, n_mu, geo_o, L)
    dev = torch.device("cuda", 0)
    dm = [{"data": torch.from_numpy(d).to(dev), "randoms": torch.from_numpy(np.concatenate(r)).to(dev),
           "offsets": [0] + list(np.cumsum([len(x) for x in r]))} for d, r in mocks]
    ref = [oracle.count_mock(d, r, ob) for d, r in mocks]
    ctx = tp.Context(0)
    ctx.tpcf_set_option(tp.TPCF_OPT_KERNEL, tp.TPCF_KERNEL_DIRECT)
    used = set()
    for subdiv in (1, 2, 0):
        ctx.tpcf_set_cell_subdiv(subdiv)
        for mode in (tp.TPCF_BATCHED, tp.TPCF_PER_LAUNCH):
            out = ctx.tpcf_count(dm, tb, mode=mode)
            assert ctx.tpcf_sync() == tp.TPCF_OK
            if subdiv != 1:   # periodic cells of a third of the box are left to the general counter
                used.add(ctx.tpcf_last_count_info()["pair_kernel"])
            for i, o in enumerate(ref):
                for k, want in (("dd", o["DD"]), ("dr", o["DR"]), ("rr", o["RR"])):
                    assert np.array_equal(out[k][i].cpu().numpy(), want), (subdiv, mode, i, k)
    assert used == {tp.TPCF_KERNEL_DIRECT}
    ctx.close()
