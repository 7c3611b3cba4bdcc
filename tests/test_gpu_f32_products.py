"""FP32 products of the paper's family where an item of pass 2 takes more rows so that every
item has a warp of its own, and beside that range.  Against the FP64 product of the same
handle by the norm: operators, vectors and sums are rounded to 24 bits, 1e-6 is eight times
that unit after sums of a few hundred terms with random signs.
"""
import numpy as np
import pytest

from paper_2403_09198_gb300 import inputs
from paper_2403_09198_gb300.binding import StsJacobian
from tests._gpu import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


# cells, N, pairs: items per resident warp just below one, 1.0 to 1.5, above; a last item of one
# row, and few pairs or many (the instances differ)
@pytest.mark.parametrize("L,N,r_diag,r_off", [(80, 60, 2, 1), (96, 60, 2, 1), (112, 60, 2, 1), (121, 60, 2, 1),
                                              (104, 41, 2, 1), (88, 100, 2, 1), (183, 10, 2, 1), (96, 31, 9, 2)])
def test_items_that_fit(L, N, r_diag, r_off):
    w = inputs.make_workload(L, L - 1, N=N, w=2, r_diag=r_diag, r_off=r_off, seed=12)
    jac = StsJacobian(w, dev(w.S), dev(w.U), dev(w.V), mixed=True, transpose=True, layout="component")
    x = dev(w.rhs)
    for trans in (False, True):
        y, ref = host(jac.matvec(x.float(), trans=trans)).astype(np.float64), host(jac.matvec(x, trans=trans))
        y, ref = (v.reshape(w.b, w.n_cells) for v in (y, ref))
        scale = np.linalg.norm(ref) / np.sqrt(ref.size)
        assert np.linalg.norm(y - ref) / np.linalg.norm(ref) <= 1e-6
        # every row by itself: none is left out
        assert (np.linalg.norm(y - ref, axis=1) / np.sqrt(w.n_cells) <= 1e-4 * scale).all()
    jac.close()
