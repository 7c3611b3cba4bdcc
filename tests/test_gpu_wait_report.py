"""How a bounded wait that gave up is reported, with the handle's flag set from the host:
each synchronous call reports it once, and a set-up that reports it sets nothing up.
"""
import numpy as np
import pytest

import oracle
from paper_2403_09198_gb300.binding import StsError, StsJacobian, check
from tests._gpu import TOL64, dev, host, oracle_jac, rel_err, workload

pytestmark = pytest.mark.gpu

STS_ERR_SINGULAR, STS_ERR_TIMEOUT, STS_ERR_NOT_SETUP = 4, 7, 8


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _raises(status, call, *args, **kw):
    with pytest.raises(StsError) as e:
        call(*args, **kw)
    assert e.value.status == status, e.value.message


def _flag(jac):
    check(jac.lib.sts_selftest_wait_flag(jac.h))


@pytest.mark.parametrize("name,dense", [("grid16_N10", False), ("random_pattern", False), ("grid16_N10", True)])
def test_setup_that_reports_a_timeout(name, dense):
    w = workload(name)
    x = np.random.default_rng(4).standard_normal(w.n)
    ref = oracle.bj_apply(oracle.bj_setup(oracle_jac(w)), x)
    jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V), dense=dense)
    _flag(jac)
    _raises(STS_ERR_TIMEOUT, jac.bjacobi_setup)
    _raises(STS_ERR_NOT_SETUP, jac.bjacobi_apply, dev(x))
    _raises(STS_ERR_NOT_SETUP, jac.gmres, dev(w.rhs))
    jac.bjacobi_setup()                                  # reported once
    assert rel_err(host(jac.bjacobi_apply(dev(x))), ref) <= TOL64
    _flag(jac)
    _raises(STS_ERR_TIMEOUT, jac.bjacobi_setup)          # set up before, and still
    assert rel_err(host(jac.bjacobi_apply(dev(x))), ref) <= TOL64
    jac.update_values(dev(w.S), dev(w.U), dev(w.V))
    _flag(jac)
    _raises(STS_ERR_TIMEOUT, jac.bjacobi_setup)
    _raises(STS_ERR_NOT_SETUP, jac.bjacobi_apply, dev(x))
    jac.close()


def test_a_singular_cell_is_not_lost_behind_a_timeout():
    w = workload("grid16_N10")
    offs = w.s_offsets()[:-1][w.is_diag_block()]
    w.S[offs[5]:offs[5] + w.nnz_d] = 0.0
    jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V))
    _flag(jac)
    _raises(STS_ERR_TIMEOUT, jac.bjacobi_setup)
    _raises(STS_ERR_NOT_SETUP, jac.bjacobi_apply, dev(w.rhs))
    _raises(STS_ERR_SINGULAR, jac.bjacobi_setup)
    jac.close()


@pytest.mark.parametrize("graph", [True, False])
def test_solve_reports_a_timeout_once(graph):
    w = workload("grid16_N10")
    jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V))
    jac.bjacobi_setup()
    _flag(jac)
    _raises(STS_ERR_TIMEOUT, jac.gmres, dev(w.rhs), rtol=1e-12, graph=graph)
    x, info = jac.gmres(dev(w.rhs), rtol=1e-12, graph=graph)
    assert info.converged
    jac.close()
