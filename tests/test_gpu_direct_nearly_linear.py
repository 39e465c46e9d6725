"""Direct pair counter on linear edges whose width no float64 holds exactly, against the brute-force oracle (whole numbers).

Separations on a lattice of the bin width fall on the edges; edges off by a part in 10^8 stay with the direct counter,
edges off by a part in 10^4 go to the general one.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

L = 150.0


@pytest.fixture(scope="module")
def tp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2205_11852_gb300 as tp
    return tp


@pytest.mark.parametrize("n_s,s_max,off,direct", [(23, 40.0, 0.0, True), (7, 47.0, 0.0, True), (37, 33.0, 1e-8, True),
                                                  (11, 49.9, 0.0, True), (13, 40.0, 1e-4, False)])
@pytest.mark.parametrize("n_mu,los", [(1, "x"), (6, "x"), (6, "mid"), (40, "x")])
def test_direct_nearly_linear_bins(tp, n_s, s_max, off, direct, n_mu, los):
    rng = np.random.default_rng(n_s)
    edges = np.linspace(0.0, s_max, n_s + 1)
    edges[n_s // 2] += off * edges[1]
    w = edges[1]
    lat = np.stack(np.meshgrid(np.arange(12), np.arange(4), np.arange(3), indexing="ij"), -1).reshape(-1, 3) * w + 20.0
    d = np.concatenate([rng.random((400, 3)) * L, lat, lat[:50]])
    r = [np.concatenate([rng.random((300, 3)) * L, lat]), rng.random((350, 3)) * L]
    obs = (-30.0, -20.0, -10.0)
    if los == "mid":
        tb = tp.make_binning(edges, n_mu, tp.TPCF_OPEN, L, los=tp.TPCF_LOS_MIDPOINT, observer=obs)
        ob = oracle.Binning(edges, n_mu, oracle.OPEN, L, los=oracle.LOS_MIDPOINT, observer=obs)
    else:
        tb, ob = tp.make_binning(edges, n_mu, tp.TPCF_PERIODIC, L), oracle.Binning(edges, n_mu, oracle.PERIODIC, L)
    dev = torch.device("cuda", 0)
    dm = [{"data": torch.from_numpy(d).to(dev), "randoms": torch.from_numpy(np.concatenate(r)).to(dev),
           "offsets": [0, len(r[0]), len(r[0]) + len(r[1])]}]
    ref = oracle.count_mock(d, r, ob)
    ctx = tp.Context(0)
    ctx.tpcf_set_option(tp.TPCF_OPT_KERNEL, tp.TPCF_KERNEL_DIRECT)
    for subdiv in (2, 3, 0):
        ctx.tpcf_set_cell_subdiv(subdiv)
        out = ctx.tpcf_count(dm, tb)
        assert ctx.tpcf_sync() == tp.TPCF_OK
        assert (ctx.tpcf_last_count_info()["pair_kernel"] == tp.TPCF_KERNEL_DIRECT) == direct
        for k, want in (("dd", ref["DD"]), ("dr", ref["DR"]), ("rr", ref["RR"])):
            assert np.array_equal(out[k][0].cpu().numpy(), want), (subdiv, k)
    ctx.close()
