"""GMRES on problems that break it down: what the caller's vector, the status and the
counts are afterwards, alike for cycles that run as one graph and host-driven ones.

The Jacobians are one block with a diagonal S and no pairs, whose solves can be followed
by hand.
"""
import types

import numpy as np
import pytest
import torch

from paper_2403_09198_gb300.binding import StsJacobian
from tests._gpu import dev, host

pytestmark = pytest.mark.gpu

STS_ERR_NUMERIC = 6


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _diagonal(vals, layout="cell"):
    """One cell whose block is diag(vals)."""
    b = len(vals)
    w = types.SimpleNamespace(
        b=b, r_diag=0, r_off=0, block_indptr=np.array([0, 1]), block_indices=np.array([0]),
        d_indptr=np.arange(b + 1), d_indices=np.arange(b), o_indptr=np.zeros(b + 1), o_indices=np.zeros(0))
    none = np.zeros((0, b))
    return StsJacobian(w, dev(np.array(vals, dtype=np.float64)), dev(none), dev(none), layout=layout)


def _solve(jac, b, x0, **kw):
    """(status, x, info) of a solve that is allowed to fail."""
    o = {}
    real = jac.lib.sts_gmres_solve
    jac.lib = types.SimpleNamespace(sts_gmres_solve=lambda *a: o.setdefault("status", real(*a)),
                                    sts_jac_destroy=jac.lib.sts_jac_destroy)
    x, info = jac.gmres(b, x0, precond="none", raise_on_fail=False, **kw)
    return o["status"], host(x) if torch.is_tensor(x) else x, info


# the zero block breaks down in the first cycle (w = 0: the rotation is 0 / 0).  With
# diag(1, 0, 0, 0), b = 1 and cycles of one step, x changes in the first cycle (the first
# component's residual drops to rounding) and a later one breaks down
@pytest.mark.parametrize("vals,restart", [([0.0] * 4, 3), ([1.0, 0.0, 0.0, 0.0], 1)])
@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("layout", ["cell", "component"])
@pytest.mark.parametrize("on_host", [False, True])
def test_x_stays_as_it_was_after_a_breakdown(vals, restart, graph, layout, on_host):
    jac = _diagonal(vals, layout)
    b, x0 = np.ones(4), np.array([0.0, 3.0, -2.0, 5.0])
    st, x, _ = _solve(jac, b if on_host else dev(b), x0 if on_host else dev(x0), restart=restart, graph=graph)
    assert st == STS_ERR_NUMERIC
    assert np.array_equal(x, x0)
    jac.close()


# ||w||^2 overflows where w itself is finite; in the first case w is a multiple of v_0, so
# that what is left of it after the update is zero, in the second small
@pytest.mark.parametrize("vals", [[1e200] * 4, [1e155, 1.0000001e155, 1e155, 1e155], [1e200, 2e200, 3e200, 5e200]])
@pytest.mark.parametrize("graph", [True, False])
def test_an_overflowing_norm_is_no_breakdown(vals, graph):
    jac = _diagonal(vals)
    st, x, info = _solve(jac, dev(np.ones(4)), dev(np.zeros(4)), restart=5, graph=graph)
    assert st == STS_ERR_NUMERIC and info.iterations == 0
    assert not x.any()
    jac.close()


def test_a_broken_cycle_counts_no_product():
    """A graph cycle that broke down adds neither steps nor products, the residual queued
    behind it included."""
    jac = _diagonal([1e200, 2e200, 3e200, 5e200])
    st, _, info = _solve(jac, dev(np.ones(4)), dev(np.zeros(4)), restart=5)
    assert st == STS_ERR_NUMERIC and (info.matvecs, info.iterations, info.restarts) == (0, 0, 0)
    jac.close()


@pytest.mark.parametrize("restart,max_iters", [(2, 1), (2, 2), (2, 3), (5, 200)])
@pytest.mark.parametrize("graph", [True, False])
def test_x_is_the_last_iterate_when_the_steps_run_out(restart, max_iters, graph):
    """STS_ERR_NOT_CONVERGED returns the iterate whose residual info reports."""
    vals = np.array([1.0, 2.0, 4.0, 8.0, 16.0, 64.0])
    jac = _diagonal(vals)
    b = np.arange(1.0, 7.0)
    st, x, info = _solve(jac, dev(b), dev(np.zeros(6)), restart=restart, max_iters=max_iters, rtol=1e-12, graph=graph)
    assert st == (0 if max_iters == 200 else 5)
    rel = np.linalg.norm(b - vals * x) / np.linalg.norm(b)
    # the device sums six squares in another order than numpy; 1e-13 is far above that rounding
    assert abs(rel - info.true_rel_residual) <= 1e-13
    jac.close()
