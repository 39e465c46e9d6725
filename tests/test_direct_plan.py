"""The direct pair counter's plan on the host: which catalogues its 32-bit counters admit (no GPU).

A unit may add at most unit_pair_bound pairs to a counter, and a table takes (2^32 - 1) / unit_pair_bound units between
drains: a plan whose bound passes 2^32 - 1 could never take one, and its warps would wait for a table until the wait
gives up.  Such catalogues belong to the general counter.
"""
import ctypes
import pathlib
import subprocess

import numpy as np
import pytest

import __graft_entry__

ROOT = pathlib.Path(__file__).resolve().parent.parent
PKG = ROOT / "paper_2205_11852_gb300"

SHIM = r"""
#include <string>
#include "plan.h"
extern "C" int direct_plan(int geometry, double L, int n_s, int n_mu, const double *edges, int los,
                           unsigned long long max_cat, unsigned long long *bound, int *copies, int *tables)
{
    tpcf_binning b = {};
    b.geometry = geometry;
    b.box_L = L;
    b.n_s = n_s;
    b.n_mu = n_mu;
    b.s_edges = edges;
    b.los = los;
    tpcf::Plan pl;
    std::string err;
    if (tpcf::build_plan(b, 2, 1ull << 24, pl, err)) return -1;
    tpcf::DirectParams d;
    // shared memory per SM and per block of a GB300, and the reservation per block
    if (!tpcf::build_direct(b, pl, 233472, 232448, 1024, max_cat, 1, d)) return 0;
    *bound = d.unit_pair_bound;
    *copies = d.R;
    *tables = d.NT;
    return 1;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    __graft_entry__.build()
    build = __graft_entry__._build_module()
    d = tmp_path_factory.mktemp("plan")
    (d / "shim.cpp").write_text(SHIM)
    cuda = pathlib.Path(build._cuda_lib_dir()).parent / "include"
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{build.INCLUDE}", f"-I{build.CSRC}", f"-I{cuda}",
                    str(d / "shim.cpp"), str(build.LIB), f"-Wl,-rpath,{build.BUILD}", "-o", str(d / "shim.so")],
                   check=True)
    f = ctypes.CDLL(str(d / "shim.so")).direct_plan
    f.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_int,
                  ctypes.c_ulonglong, ctypes.POINTER(ctypes.c_ulonglong), ctypes.POINTER(ctypes.c_int),
                  ctypes.POINTER(ctypes.c_int)]

    def call(edges, n_mu, max_cat, geometry=0, L=1500.0, los=0):
        e = np.ascontiguousarray(edges, dtype=np.float64)
        bound, copies, tables = ctypes.c_ulonglong(), ctypes.c_int(), ctypes.c_int()
        rc = f(geometry, L, len(e) - 1, n_mu, e.ctypes.data, los, max_cat, bound, copies, tables)
        assert rc >= 0
        return (bound.value, copies.value, tables.value) if rc else None

    return call


BINNINGS = {
    "s only": (np.linspace(0.0, 200.0, 41), 1, 32),
    "mu": (np.linspace(0.0, 200.0, 41), 10, 8),
    "geometric": (np.geomspace(1.0, 200.0, 25), 5, None),
    "fine mu": (np.linspace(0.0, 200.0, 201), 100, 1),
}


@pytest.mark.parametrize("name", list(BINNINGS))
@pytest.mark.parametrize("max_cat", [1, 1000, 10 ** 6, 67 * 10 ** 6, 67_108_000, 67_109_000, 68 * 10 ** 6, 10 ** 8, 2 ** 28 - 1])
def test_a_unit_never_passes_a_counter(plan, name, max_cat):
    edges, n_mu, copies = BINNINGS[name]
    got = plan(edges, n_mu, max_cat)
    # one copy of the table: 64 a-points times the whole catalogue reach 2^32 at 67.1 million points
    assert (got is None) == (name == "fine mu" and 64 * (max_cat + 512 + 16) >= 2 ** 32)
    if got:
        assert got[0] < 2 ** 32
        assert copies is None or got[1] == copies


# the tables that the schedule tests count on: four, two and one per block, copied or with a column per |mu| bin
@pytest.mark.parametrize("n_s,n_mu,tables,copies", [(12, 1, 4, 32), (20, 5, 2, 16), (40, 10, 2, 8), (60, 10, 1, 8),
                                                    (30, 25, 2, 1)])
def test_tables_per_block(plan, n_s, n_mu, tables, copies):
    _, r, nt = plan(np.linspace(0.0, 24.0, n_s + 1), n_mu, 3000, L=100.0)
    assert (nt, r) == (tables, copies)
