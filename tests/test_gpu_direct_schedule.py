"""Direct pair counter: how a block's warps pass from term to term, against the brute-force oracle (whole numbers).

The cases are the edges of the schedule: many terms of fewer units than a block has warps (more terms in flight than
tables), terms without any unit, one long term, and binnings that give four, two and one table per block.
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


def _mocks(sizes, M, L, seed):
    rng = np.random.default_rng(seed)
    out = []
    for n in sizes:
        parents = rng.random((4, 3)) * L
        d = np.mod(parents[rng.integers(0, 4, n)] + rng.normal(0.0, 0.05 * L, (n, 3)), L)
        d[d >= L] = 0.0
        out.append((d, [rng.random((max(0, n - i), 3)) * L for i in range(M)]))
    return out


MANY = [0, 1, 2, 3, 5, 17, 33, 64, 65, 90, 0, 7, 130, 2, 40, 200] * 2
# s bins x mu bins: four tables (s only), two with 16 and 8 copies, one; the largest has few copies of its own
BINNINGS = [(12, 1), (20, 5), (40, 10), (60, 10), (30, 25)]


@pytest.mark.parametrize("n_s,n_mu", BINNINGS)
@pytest.mark.parametrize("sizes,M", [(MANY, 2), ([2500], 1), ([600, 1, 500], 3)])
def test_direct_terms_and_tables(tp, n_s, n_mu, sizes, M):
    L, s_max = 100.0, 24.0
    mocks = _mocks(sizes, M, L, 91 + n_s)
    edges = np.linspace(0.0, s_max, n_s + 1)
    tb = tp.make_binning(edges, n_mu, tp.TPCF_PERIODIC, L)
    ob = oracle.Binning(edges, n_mu, oracle.PERIODIC, L)
    dev = torch.device("cuda", 0)
    dm = [{"data": torch.from_numpy(d).to(dev), "randoms": torch.from_numpy(np.concatenate(r)).to(dev),
           "offsets": [0] + list(np.cumsum([len(x) for x in r]))} for d, r in mocks]
    ref = [oracle.count_mock(d, r, ob) for d, r in mocks]
    ctx = tp.Context(0)
    for kernel, subdiv in ((tp.TPCF_KERNEL_DIRECT, 1), (tp.TPCF_KERNEL_DIRECT, 2), (tp.TPCF_KERNEL_DIRECT, 4),
                           (tp.TPCF_KERNEL_AUTO, 0)):   # 0: tuned (cells wider, or two to a unit, when sparse)
        ctx.tpcf_set_option(tp.TPCF_OPT_KERNEL, kernel)
        ctx.tpcf_set_cell_subdiv(subdiv)
        for mode in (tp.TPCF_BATCHED, tp.TPCF_PER_LAUNCH):
            out = ctx.tpcf_count(dm, tb, mode=mode)
            assert ctx.tpcf_sync() == tp.TPCF_OK
            for i, o in enumerate(ref):
                for k, want in (("dd", o["DD"]), ("dr", o["DR"]), ("rr", o["RR"])):
                    assert np.array_equal(out[k][i].cpu().numpy(), want), (kernel, subdiv, mode, i, k)
            info = ctx.tpcf_last_count_info()
            assert info["n_binned"] == sum(int(o[k].sum()) for o in ref for k in ("DD", "DR", "RR"))
    ctx.close()
