"""Direct pair counter on geometric (logarithmic) s bins against the brute-force oracle (whole numbers).

The cases are where the logarithm's bins can go wrong: a first edge far below the last (pairs below a chosen bin are all
rechecked) and one close to it (pairs below the first edge are certain misses), one bin, narrow bins, edges that are
nearly but not quite geometric, separations exactly on the edges, coincident points, both geometries, mu bins along x
with each number of histogram copies.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

L = 128.0


@pytest.fixture(scope="module")
def tp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2205_11852_gb300 as tp
    return tp


def _points(seed, n):
    """Clustered points, coincident ones, and a lattice of spacing 1 whose separations fall on powers of two."""
    rng = np.random.default_rng(seed)
    parents = rng.random((6, 3)) * L
    x = np.mod(parents[rng.integers(0, 6, n)] + rng.normal(0.0, 6.0, (n, 3)), L)
    u = rng.random((n, 3)) * L
    lat = np.stack(np.meshgrid(np.arange(6), np.arange(5), np.arange(4), indexing="ij"), -1).reshape(-1, 3) * 1.0 + 64.0
    out = np.concatenate([x, u, x[:40], lat, lat + [4.0, 0.0, 0.0]])
    out[out >= L] = 0.0
    return out


def _edges(kind):
    if kind == "wide":
        return np.geomspace(0.2, 40.0, 25)
    if kind == "powers":
        return 2.0 ** np.arange(-3, 6)
    if kind == "far":
        return np.geomspace(20.0, 40.0, 8)
    if kind == "one":
        return np.array([4.0, 32.0])
    if kind == "narrow":
        return np.geomspace(10.0, 40.0, 121)
    if kind == "tiny":
        return np.geomspace(1e-5, 32.0, 13)
    e = np.geomspace(1.0, 40.0, 17)   # "off": the middle edge off by a part in 10^5
    e[8] *= 1.0 + 1e-5
    return e


@pytest.mark.parametrize("kind", ["wide", "powers", "far", "one", "narrow", "tiny", "off"])
@pytest.mark.parametrize("n_mu,geometry", [(1, "periodic"), (1, "open"), (5, "periodic"), (12, "open"), (25, "periodic")])
def test_direct_geometric_bins(tp, kind, n_mu, geometry):
    edges = _edges(kind)
    mocks = [(_points(3, 400), [_points(4, 300), _points(5, 333)]), (_points(6, 1), [_points(7, 30), _points(8, 20)])]
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
    for subdiv in (1, 3, 0):
        ctx.tpcf_set_cell_subdiv(subdiv)
        for mode in (tp.TPCF_BATCHED, tp.TPCF_PER_LAUNCH):
            out = ctx.tpcf_count(dm, tb, mode=mode)
            assert ctx.tpcf_sync() == tp.TPCF_OK
            if subdiv != 1:   # periodic cells of a third of the box are left to the general counter
                used.add(ctx.tpcf_last_count_info()["pair_kernel"])
            for i, o in enumerate(ref):
                for k, want in (("dd", o["DD"]), ("dr", o["DR"]), ("rr", o["RR"])):
                    assert np.array_equal(out[k][i].cpu().numpy(), want), (subdiv, mode, i, k)
    if kind in ("wide", "powers", "far", "one") and n_mu <= 12:
        assert used == {tp.TPCF_KERNEL_DIRECT}
    ctx.close()
