"""Block-Jacobi setup and values load at the sizes where their windows and tiles end.

The paper's pattern family runs its own factorisation and solve kernels for every
level band 0..4, with C^-1 per pair count; each is compared with the oracle's dense
solves, element by element, at the tolerance of the FP64 path.
"""
import numpy as np
import pytest

import oracle
from paper_2403_09198_gb300 import inputs
from paper_2403_09198_gb300.binding import StsError, StsJacobian
from tests._gpu import TOL64, dev, host, oracle_jac, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _check(w, tol=TOL64, mixed=False):
    J = oracle_jac(w)
    F = oracle.bj_setup(J)
    jac = StsJacobian(w, *(np.zeros_like(a) + 1.0 for a in (w.S, w.U, w.V)), transpose=True, mixed=mixed)
    jac.update_values(dev(w.S), dev(w.U), dev(w.V))          # every value is replaced, padding stays zero
    jac.bjacobi_setup()
    x = np.random.default_rng(3).standard_normal(w.n)
    for trans in (False, True):
        assert rel_err(host(jac.matvec(dev(x), trans=trans)), oracle.matvec(J, x, trans=trans)) <= tol
        assert rel_err(host(jac.bjacobi_apply(dev(x), trans=trans)), oracle.bj_apply(F, x, trans=trans)) <= tol
    if mixed:
        x32 = dev(x).float()
        for got, ref in ((jac.matvec(x32), oracle.matvec(J, x)), (jac.bjacobi_apply(x32), oracle.bj_apply(F, x))):
            ref = np.asarray(ref)
            assert np.linalg.norm(host(got) - ref) / np.linalg.norm(ref) <= 1e-6
    jac.close()


@pytest.mark.parametrize("w", range(5))
@pytest.mark.parametrize("N", ["least", 31, 34])
def test_band_and_pairs(w, N):
    """The narrowest block of each band (N = w + 1), and rows past one and two runs
    of 32; pair counts over all C^-1 instances and both forms of the apply's tail."""
    N = w + 1 if N == "least" else N
    for r in {0: (1, 4), 1: (2, 9), 2: (3, 10), 3: (1, 6), 4: (5, 8)}[w]:
        _check(inputs.make_workload(7, 5, N=N, w=w, r_diag=r, r_off=1, seed=50 + r), mixed=r in (1, 9))


def _diag_values(w):
    """Views of the diagonal blocks' S values [nc, nnz_d] positions and pair rows [nc, r]."""
    offs = w.s_offsets()[:-1][w.is_diag_block()]
    pairs = np.asarray(w.pair_indptr)[:-1][w.is_diag_block()]
    return offs, pairs


@pytest.mark.parametrize("r", [2, 4, 9])
def test_capacitance_needs_row_exchanges(r):
    """C = I + V^T S^-1 U made a cyclic permutation (no pivot on its diagonal), a
    different one in every cell: the pivot rows differ from lane to lane."""
    w = inputs.make_workload(6, 6, N=12, w=2, r_diag=r, r_off=1, seed=60)
    J = oracle_jac(w)
    offs, pairs = _diag_values(w)
    p = np.repeat(np.arange(w.b), np.diff(w.d_indptr))
    for c in range(w.n_cells):
        S = np.zeros((w.b, w.b))
        S[p, w.d_indices] = w.S[offs[c]:offs[c] + w.nnz_d]
        k = np.arange(r)
        V = np.zeros((r, w.b))
        V[k, k] = 1.0
        X = np.zeros((r, w.b))                       # S^-1 U: column k is e_sigma(k) - e_k
        X[k, (k + 1 + c % (r - 1 or 1)) % r] += 1.0
        X[k, k] -= 1.0
        w.V[pairs[c]:pairs[c] + r], w.U[pairs[c]:pairs[c] + r] = V, X @ S.T
    del J
    _check(w)


@pytest.mark.parametrize("fault", ["capacitance", "pivot", "nan"])
def test_singular_cells_are_named(fault):
    w = inputs.make_workload(9, 8, N=12, w=2, r_diag=2, r_off=1, seed=61)
    offs, pairs = _diag_values(w)
    c = 37
    p = np.repeat(np.arange(w.b), np.diff(w.d_indptr))
    block = w.S[offs[c]:offs[c] + w.nnz_d]
    if fault == "capacitance":                       # C = diag(0, 1)
        S = np.zeros((w.b, w.b))
        S[p, w.d_indices] = block
        w.U[pairs[c]:pairs[c] + 2], w.V[pairs[c]:pairs[c] + 2] = 0.0, 0.0
        w.V[pairs[c], 0] = 1.0
        w.U[pairs[c]] = -S[:, 0]
    elif fault == "pivot":
        block[p == 5] *= 1e-300                      # the row's pivot and its maximum alike stay sound ...
        block[(p == 7) & (w.d_indices == 7)] = 0.0   # ... a zero pivot does not
        block[(p == 7) & (w.d_indices != 7)] = 0.0
    else:
        block[(p == 4) & (w.d_indices == 4)] = np.nan
    jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V))
    with pytest.raises(StsError) as e:
        jac.bjacobi_setup()
    assert e.value.status == 4 and f"cell {c} " in e.value.message
    jac.close()
