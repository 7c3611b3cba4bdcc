"""Operators on public vectors in place, and the general kernels' programs.

Component-major and small cell-major vectors are read and written in place; larger
cell-major matvecs transpose x, and applies whose working vector lives in y go through
the internal layout.  Either way the arithmetic is the same, so every layout gives the
same bits.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2403_09198_gb300 import inputs
from paper_2403_09198_gb300.binding import StsJacobian
from tests._gpu import TOL64, dev, from_component_major, host, oracle_jac, rel_err, to_component_major

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _calls(jac, x, out):
    """The four operators on views of x, into views from out(x)."""
    got = []
    for v in (x, x.float()):
        for f in (jac.matvec, jac.bjacobi_apply):
            for trans in (False, True):
                got.append(host(f(v, out=out(v), trans=trans)))
    return got


# ragged and full tiles; 130 x 127 x 33 values are more than a cell-major matvec reads
# in place in FP64 (2^18), 60 x 50 x 33 more than in FP32 (2^15); b = 143 keeps the apply's
# working vector in y (FP64)
@pytest.mark.parametrize("Lx,Ly,N,density", [(8, 4, 20, 0.0), (5, 7, 60, 0.0), (60, 50, 30, 0.0), (130, 127, 30, 0.0),
                                             (9, 8, 140, 0.0), (91, 90, 30, 0.1)])
def test_layouts_give_the_same_bits(Lx, Ly, N, density):
    w = inputs.make_workload(Lx, Ly, N=N, w=2, r_diag=2, r_off=1, seed=70, random_density=density)
    x = np.random.default_rng(1).standard_normal(w.n)
    got = {}
    for layout in ("cell", "component"):
        jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V), transpose=True, mixed=True, layout=layout)
        jac.bjacobi_setup()
        xi = dev(x if layout == "cell" else to_component_major(x, w.n_cells, w.b))
        back = (lambda v: v) if layout == "cell" else (lambda v: from_component_major(v, w.n_cells, w.b))
        got[layout] = [back(v) for v in _calls(jac, xi, torch.empty_like)]
        # the same vectors one value off a 16-byte boundary
        pad = torch.empty(w.n + 1, dtype=torch.float64, device="cuda")
        pad[1:] = xi
        off = [back(v) for v in _calls(jac, pad[1:], lambda v: torch.empty(w.n + 1, dtype=v.dtype, device="cuda")[1:])]
        for a, b in zip(off, got[layout]):
            assert np.array_equal(a, b), layout
        # nothing is written outside the result
        y = torch.full((w.n + 64,), 7.0, dtype=torch.float64, device="cuda")
        for f in (jac.matvec, jac.bjacobi_apply):
            f(xi, out=y[32:32 + w.n])
            assert bool((y[:32] == 7.0).all()) and bool((y[32 + w.n:] == 7.0).all())
        jac.close()
    for a, b in zip(got["cell"], got["component"]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("N,density,r", [(1, 0.5, 1), (2, 0.3, 0), (5, 0.9, 3), (6, 0.2, 5), (30, 0.15, 2),
                                         (29, 0.02, 12), (61, 0.1, 16), (200, 0.01, 1)])
@pytest.mark.parametrize("Lx,Ly", [(1, 1), (9, 7)])
def test_general_patterns(N, density, r, Lx, Ly):
    """Blocks of 4 to 203 rows, all remainders of the four warps' dealing, empty
    columns, 0 to 16 pairs, full fill-in."""
    w = inputs.make_workload(Lx, Ly, N=N, r_diag=r, r_off=1, seed=80 + N, random_density=density)
    J = oracle_jac(w)
    F = oracle.bj_setup(J)
    x = np.random.default_rng(2).standard_normal(w.n)
    for layout in ("cell", "component"):
        jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V), transpose=True, mixed=True, layout=layout)
        jac.bjacobi_setup()
        xi = dev(x if layout == "cell" else to_component_major(x, w.n_cells, w.b))
        back = (lambda v: v) if layout == "cell" else (lambda v: from_component_major(v, w.n_cells, w.b))
        for trans in (False, True):
            assert rel_err(back(host(jac.matvec(xi, trans=trans))), oracle.matvec(J, x, trans=trans)) <= TOL64
            assert rel_err(back(host(jac.bjacobi_apply(xi, trans=trans))), oracle.bj_apply(F, x, trans=trans)) <= TOL64
        z = back(host(jac.bjacobi_apply(xi.float())).astype(np.float64))
        ref = oracle.bj_apply(F, x)
        assert np.linalg.norm(z - ref) / np.linalg.norm(ref) <= 1e-6
        jac.close()


def test_absent_neighbours_add_nothing_in_general_patterns():
    """A boundary cell's absent neighbour is not read as its own cell: an infinite
    component that no present block multiplies leaves the product finite."""
    w = inputs.make_workload(3, 1, N=2, r_diag=0, r_off=0, seed=90, random_density=0.3)
    d = np.zeros((w.b, w.b), bool)
    o = np.zeros((w.b, w.b), bool)
    d[np.arange(w.b), np.arange(w.b)] = True
    o[:, 0] = True
    w.d_indptr, w.d_indices = np.arange(w.b + 1, dtype=np.int32), np.arange(w.b, dtype=np.int32)
    w.o_indptr, w.o_indices = np.arange(w.b + 1, dtype=np.int32), np.zeros(w.b, dtype=np.int32)
    w.S = np.ones(3 * w.b + 4 * w.b)
    jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V))
    x = np.ones((3, w.b))
    x[0, 0] = np.inf
    y = host(jac.matvec(dev(x.ravel()))).reshape(3, w.b)
    assert np.isinf(y[0, 0]) and np.isfinite(y[0, 1:]).all() and np.isinf(y[1]).all() and np.isfinite(y[2]).all()
    jac.close()


def test_block_sizes_take_turns():
    """Handles whose launches of one kernel instance need different shared memory, applied
    in turn: the larger one's launches stay possible after the smaller one's.  Applies on
    a pattern of one cell solve with the block itself, so J M b = b; the rounding of a
    block of 63 with entries below 1 on a diagonal above 1000 is far below TOL64."""
    jacs = []
    for N in (60, 10):
        w = inputs.make_workload(1, 1, N=N, w=2, r_diag=2, r_off=0, seed=5)
        jacs.append((StsJacobian(w, dev(w.S), dev(w.U), dev(w.V)), w))
        jacs[-1][0].bjacobi_setup()
    for j, w in jacs + jacs:
        assert rel_err(host(j.matvec(j.bjacobi_apply(dev(w.rhs)))), w.rhs) <= TOL64
    for j, _ in jacs:
        j.close()
