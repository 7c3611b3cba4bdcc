"""Products of patterns outside the paper's family on grids of more warps than fit at once,
where the FP64 kernel takes its other form, and on both sides of that line; FP32 products
and applies in both directions.  Compared with the oracle: FP64 at the tolerance of that
path, FP32 by the norm at 1e-6 (operators rounded to 24 bits, sums of some 500 terms).
"""
import numpy as np
import pytest

import oracle
from paper_2403_09198_gb300 import inputs
from paper_2403_09198_gb300.binding import StsJacobian
from tests._gpu import TOL64, dev, from_component_major, host, oracle_jac, rel_err, to_component_major

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


# 32 cells a tile, 16 groups of rows or more: 2432 warps are 16 per SM.  One row a group and
# few tiles; just below and above the line; several rows a group; single rows on many tiles
@pytest.mark.parametrize("Lx,Ly,N,density,r", [(24, 20, 30, 0.15, 2), (47, 40, 60, 0.1, 2), (64, 63, 20, 0.5, 1),
                                               (91, 90, 30, 0.1, 2), (100, 61, 10, 0.3, 3), (40, 131, 61, 0.03, 0)])
def test_products_against_the_oracle(Lx, Ly, N, density, r):
    w = inputs.make_workload(Lx, Ly, N=N, r_diag=r, r_off=1, seed=31 + N, random_density=density)
    J = oracle_jac(w)
    F = oracle.bj_setup(J)
    x = np.random.default_rng(6).standard_normal(w.n)
    ref = {t: (oracle.matvec(J, x, trans=t), oracle.bj_apply(F, x, trans=t)) for t in (False, True)}
    for layout in ("cell", "component"):
        jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V), transpose=True, mixed=True, layout=layout)
        jac.bjacobi_setup()
        xi = dev(x if layout == "cell" else to_component_major(x, w.n_cells, w.b))
        back = (lambda v: host(v)) if layout == "cell" else (lambda v: from_component_major(host(v), w.n_cells, w.b))
        for trans in (False, True):
            for f, want in zip((jac.matvec, jac.bjacobi_apply), ref[trans]):
                assert rel_err(back(f(xi, trans=trans)), want) <= TOL64, (layout, trans, f.__name__)
                got = back(f(xi.float(), trans=trans)).astype(np.float64)
                assert np.linalg.norm(got - want) / np.linalg.norm(want) <= 1e-6, (layout, trans, f.__name__)
        jac.close()


@pytest.mark.parametrize("Lx,Ly", [(3, 2), (91, 90)])
def test_absent_neighbours_add_nothing(Lx, Ly):
    """An infinite component of a corner cell reaches its own entry and its two neighbours'
    rows and nothing else, in both precisions."""
    w = inputs.make_workload(Lx, Ly, N=2, r_diag=0, r_off=0, seed=90, random_density=0.3)
    w.d_indptr, w.d_indices = np.arange(w.b + 1, dtype=np.int32), np.arange(w.b, dtype=np.int32)
    w.o_indptr, w.o_indices = np.arange(w.b + 1, dtype=np.int32), np.zeros(w.b, dtype=np.int32)
    w.S = np.ones(w.nnzb * w.b)
    jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V), mixed=True)
    x = np.ones((w.n_cells, w.b))
    x[0, 0] = np.inf
    want = np.zeros((w.n_cells, w.b), bool)
    want[0, 0] = want[1] = want[Lx] = True
    for v in (dev(x.ravel()), dev(x.ravel()).float()):
        y = host(jac.matvec(v)).reshape(w.n_cells, w.b)
        assert np.array_equal(~np.isfinite(y), want)
    jac.close()
