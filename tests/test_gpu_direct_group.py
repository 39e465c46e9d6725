"""Direct pair counter with units of two cells along x, against the brute-force oracle (whole numbers).

The autotuner picks such units by timing; here they are pinned.  Meshes with odd and even numbers of cells (a short last
group), reaches of one to four cells, boxes at and below the smallest that a group fits (both are left to the general
counter), both geometries, auto and cross terms, each kind of binning.
"""
import numpy as np
import pytest

import oracle

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


def _check(tp, ctx, dm, tb, ref, what):
    for mode in (tp.TPCF_BATCHED, tp.TPCF_PER_LAUNCH):
        out = ctx.tpcf_count(dm, tb, mode=mode)
        assert ctx.tpcf_sync() == tp.TPCF_OK
        for i, o in enumerate(ref):
            for k, want in (("dd", o["DD"]), ("dr", o["DR"]), ("rr", o["RR"])):
                assert np.array_equal(out[k][i].cpu().numpy(), want), (what, mode, i, k)
    return ctx.tpcf_last_count_info()


def _mocks(rng, sizes, L):
    host = [(rng.random((n, 3)) * L, [rng.random((n, 3)) * L, rng.random((max(0, n - 5), 3)) * L]) for n in sizes]
    dev = torch.device("cuda", 0)
    return host, [{"data": torch.from_numpy(d).to(dev), "randoms": torch.from_numpy(np.concatenate(r)).to(dev),
                   "offsets": [0, len(r[0]), len(r[0]) + len(r[1])]} for d, r in host]


def _fits(tp, tb, n_c, group, reach):
    """Every neighbour within half a box of the unit's corner, no cell a neighbour from both sides."""
    last = tp.tpcf_thresholds(tb)[-1]
    span = group * -(-2 ** 32 // n_c) - 1 + int(np.floor(np.sqrt(float(last - 1))))
    return span < 2 ** 31 and group + 2 * reach <= n_c


# box side over last edge: from the smallest allowed to where a group fits at every subdivision
@pytest.mark.parametrize("ratio", [3.0, 3.34, 4.01, 4.5, 5.01, 6.2, 7.03])
@pytest.mark.parametrize("subdiv", [1, 2, 3, 4])
def test_groups_of_two_in_a_box(tp, ratio, subdiv, monkeypatch):
    monkeypatch.setenv("TPCF_TEST_GROUP", "2")
    s_max = 30.0
    L = ratio * s_max
    rng = np.random.default_rng(int(100 * ratio) + subdiv)
    host, dm = _mocks(rng, [700, 1, 64, 0], L)
    ctx = tp.Context(0)
    ctx.tpcf_set_option(tp.TPCF_OPT_KERNEL, tp.TPCF_KERNEL_DIRECT)
    ctx.tpcf_set_cell_subdiv(subdiv)
    for edges, n_mu in ((np.linspace(0.0, s_max, 11), 1), (np.linspace(0.0, s_max, 11), 6),
                        (np.geomspace(1.0, s_max, 9), 1), (np.geomspace(1.0, s_max, 9), 4),
                        (np.linspace(0.0, s_max, 31), 40)):
        tb = tp.make_binning(edges, n_mu, tp.TPCF_PERIODIC, L)
        ob = oracle.Binning(edges, n_mu, oracle.PERIODIC, L)
        info = _check(tp, ctx, dm, tb, [oracle.count_mock(d, r, ob) for d, r in host], (ratio, subdiv, len(edges), n_mu))
        fits = _fits(tp, tb, info["cells_per_axis"], 2, subdiv)
        assert info["pair_kernel"] == (tp.TPCF_KERNEL_DIRECT if fits else tp.TPCF_KERNEL_GENERAL)
    ctx.close()


@pytest.mark.parametrize("los", ["x", "midpoint"])
@pytest.mark.parametrize("subdiv", [1, 2, 3, 4])
def test_groups_of_two_in_the_open(tp, los, subdiv, monkeypatch):
    monkeypatch.setenv("TPCF_TEST_GROUP", "2")
    rng = np.random.default_rng(subdiv)
    ctx = tp.Context(0)
    ctx.tpcf_set_option(tp.TPCF_OPT_KERNEL, tp.TPCF_KERNEL_DIRECT)
    ctx.tpcf_set_cell_subdiv(subdiv)
    edges, obs = np.linspace(0.0, 20.0, 9), (0.0, 5.0, 1.0)
    for L in (41.0, 62.0, 100.0, 141.0):   # two cells per last edge and more, odd and even numbers
        host, dm = _mocks(rng, [500, 2, 33], L)
        tb = tp.make_binning(edges, 4, tp.TPCF_OPEN, L, los=tp.TPCF_LOS_X if los == "x" else tp.TPCF_LOS_MIDPOINT,
                             observer=obs)
        ob = oracle.Binning(edges, 4, oracle.OPEN, L, los=oracle.LOS_X if los == "x" else oracle.LOS_MIDPOINT, observer=obs)
        info = _check(tp, ctx, dm, tb, [oracle.count_mock(d, r, ob) for d, r in host], (L, subdiv, los))
        assert info["pair_kernel"] == tp.TPCF_KERNEL_DIRECT
    ctx.close()


# which counter the half-box rule leaves a mesh to (one cell per unit)
@pytest.mark.parametrize("ratio", [1.0 / 3.0, 0.32, 0.26, 0.25, 0.24])
@pytest.mark.parametrize("subdiv", [1, 2, 3])
def test_counter_at_half_the_box(tp, ratio, subdiv):
    L = 120.0
    host, dm = _mocks(np.random.default_rng(3), [400], L)
    edges = np.arange(9) * (ratio * L / 8.0)
    tb = tp.make_binning(edges, 4, tp.TPCF_PERIODIC, L)
    ctx = tp.Context(0)
    ctx.tpcf_set_option(tp.TPCF_OPT_KERNEL, tp.TPCF_KERNEL_DIRECT)
    ctx.tpcf_set_cell_subdiv(subdiv)
    ob = oracle.Binning(edges, 4, oracle.PERIODIC, L)
    info = _check(tp, ctx, dm, tb, [oracle.count_mock(d, r, ob) for d, r in host], (ratio, subdiv))
    direct = _fits(tp, tb, info["cells_per_axis"], 1, subdiv)
    assert info["pair_kernel"] == (tp.TPCF_KERNEL_DIRECT if direct else tp.TPCF_KERNEL_GENERAL)
    assert direct == (subdiv > 1 or ratio <= 0.25) or ratio > 0.3
    ctx.close()
