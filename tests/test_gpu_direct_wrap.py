"""Direct pair counter where a unit's neighbourhood reaches half the periodic box, against the brute-force oracle.

Coordinates are differences from the unit's corner modulo the box, so a cell and the last edge must fit in half of it:
at subdivision 1 with last edges beyond a quarter of the box (three cells per axis) they do not.
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


# last edge over box side: a third, just below it, just above, at and below a quarter
@pytest.mark.parametrize("ratio", [1.0 / 3.0, 0.32, 0.26, 0.25, 0.24])
@pytest.mark.parametrize("n_mu", [1, 4])
def test_direct_at_half_the_box(tp, ratio, n_mu):
    L, n = 120.0, 700
    rng = np.random.default_rng(7)
    d, r = rng.random((n, 3)) * L, [rng.random((n, 3)) * L, rng.random((n - 3, 3)) * L]
    edges = np.arange(9) * (ratio * L / 8.0)
    tb = tp.make_binning(edges, n_mu, tp.TPCF_PERIODIC, L)
    ref = oracle.count_mock(d, r, oracle.Binning(edges, n_mu, oracle.PERIODIC, L))
    dev = torch.device("cuda", 0)
    dm = [{"data": torch.from_numpy(d).to(dev), "randoms": torch.from_numpy(np.concatenate(r)).to(dev),
           "offsets": [0, n, 2 * n - 3]}]
    ctx = tp.Context(0)
    for kernel in (tp.TPCF_KERNEL_DIRECT, tp.TPCF_KERNEL_AUTO):
        ctx.tpcf_set_option(tp.TPCF_OPT_KERNEL, kernel)
        for subdiv in (1, 2, 0):   # 0: tuned
            ctx.tpcf_set_cell_subdiv(subdiv)
            out = ctx.tpcf_count(dm, tb)
            assert ctx.tpcf_sync() == tp.TPCF_OK
            for k, want in (("dd", ref["DD"]), ("dr", ref["DR"]), ("rr", ref["RR"])):
                assert np.array_equal(out[k][0].cpu().numpy(), want), (kernel, subdiv, k)
    ctx.close()
