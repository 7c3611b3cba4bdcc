"""Orthogonalisation sweeps at the vector counts and lengths where they change form:
one to a chunk's 31 vectors and past it, cycles of every length below the graph's 64,
vectors shorter than a block, of ragged length, and longer than a grid pass.
"""
import numpy as np
import pytest

import oracle
from paper_2403_09198_gb300 import inputs
from paper_2403_09198_gb300.binding import StsJacobian
from tests._gpu import dev, host, oracle_jac, sol_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _solve_all(w, restart, rtol, precond, tol, max_iters=400):
    """Graph and host-driven cycles against the oracle: iterations within one, solutions
    within tol (bounded by the residual tolerance times the conditioning, see below)."""
    jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V))
    jac.bjacobi_setup()
    xo, io = oracle.gmres(oracle_jac(w), w.rhs, restart=restart, rtol=rtol, precond=precond, max_iters=max_iters)
    assert io["converged"]
    for graph in (True, False):
        x, info = jac.gmres(dev(w.rhs), restart=restart, rtol=rtol, precond=precond, max_iters=max_iters, graph=graph)
        assert info.converged and abs(info.iterations - io["iterations"]) <= 1, (graph, info.iterations)
        assert sol_err(host(x), xo) <= tol, graph
    jac.close()


@pytest.mark.parametrize("restart", [1, 2, 3, 5, 7, 9, 15, 16, 17, 23, 24, 25])
def test_cycle_lengths(restart):
    # both solvers reach a residual of 1e-13; J is within a factor of about 10 of its
    # inverse's scale here (dt = 0.5), so the solutions agree to 1e-11
    w = inputs.make_workload(6, 5, N=4, w=2, r_diag=2, r_off=1, seed=9, dt=0.5)
    _solve_all(w, restart, 1e-13, "bj", 1e-11)


@pytest.mark.parametrize("restart", [31, 32, 33, 64])
def test_cycles_past_one_chunk(restart):
    """63 to 70 unpreconditioned steps (dt = 1), so cycles of more than 31 vectors run."""
    w = inputs.make_workload(8, 6, N=6, w=2, r_diag=2, r_off=1, seed=9, dt=1.0)
    jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V))
    its = {}
    for graph in (True, False):
        x, info = jac.gmres(dev(w.rhs), restart=restart, rtol=1e-12, precond="none", max_iters=400, graph=graph)
        r = w.rhs - oracle.matvec(oracle_jac(w), host(x))
        assert info.converged and np.linalg.norm(r) / np.linalg.norm(w.rhs) <= 1.01e-12
        its[graph] = info.iterations
    _, io = oracle.gmres(oracle_jac(w), w.rhs, restart=restart, rtol=1e-12, precond="none", max_iters=400)
    # rounding moves the end of a slowly converging solve by a few steps
    assert abs(its[True] - io["iterations"]) <= 3 and its[True] == its[False]
    jac.close()


@pytest.mark.parametrize("Lx,Ly,N", [(1, 1, 5), (3, 11, 4), (41, 29, 10), (97, 83, 13)])
def test_vector_lengths(Lx, Ly, N):
    """From one block of 256 elements to several passes of the full grid (304 x 256)."""
    w = inputs.make_workload(Lx, Ly, N=N, w=1, r_diag=2, r_off=1, seed=10, dt=0.02)
    _solve_all(w, 12, 1e-13, "bj", 1e-11)
