"""The HLL-flux generator where its kernels' tiles end: cells about the 8 of a face
warp and the 32 of a mixture block, species about the 32 lanes, the largest block
(b = 256), and a uniform state, where every wave-speed candidate ties between the two
sides of a face.  Same oracle, scales and tolerance as tests/test_gpu_flow.py.
"""
import numpy as np
import numpy as np
import pytest

from oracle import flux
from paper_2403_09198_gb300 import inputs
from paper_2403_09198_gb300.binding import StsFlow
from tests._gpu import dev, host
from tests.test_gpu_flow import TOL_RES, _res_err, _scaled_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("Lx,Ly,N,w", [(3, 3, 31, 2), (11, 3, 32, 4), (8, 5, 33, 2), (2, 16, 64, 0), (5, 2, 65, 3),
                                       (2, 2, 253, 2), (1, 33, 7, 1)])
@pytest.mark.parametrize("uniform", [False, True])
def test_edges(Lx, Ly, N, w, uniform):
    c = inputs.make_flow_case(Lx, Ly, N=N, w=w, seed=21, dt=0.3)
    if uniform:
        c.Q[:] = c.Q[0]
    m = flux.model_of(c)
    f = StsFlow(c)
    ref = flux.jacobian_blocks(m, Lx, Ly, c.Q)
    for _ in range(2):                       # the second call finds the first one's scalars in its workspace
        R = host(f.residual(dev(c.Q), dev(c.Qn)))
        for key, got in zip("SUV", f.jacobian(dev(c.Q))):
            assert _scaled_err(host(got), ref[key], ref["scales"][key]) <= TOL_RES, key
        assert _res_err(R, m, c) <= TOL_RES
    f.close()


@pytest.mark.parametrize("T", [-0.7, 0.0])
@pytest.mark.parametrize("Lx,Ly,N", [(6, 5, 7), (5, 4, 40)])
def test_a_cell_without_a_sound_speed(T, Lx, Ly, N):
    """A Newton iterate with T <= 0 in one cell: da/dq is no number there, but the cell gives
    its faces no wave speed, so every entry that the model defines stays finite."""
    c = inputs.make_flow_case(Lx, Ly, N=N, w=1, seed=3, dt=0.3)
    c.Q[Lx + 2, N + 2] = T
    m = flux.model_of(c)
    with np.errstate(invalid="ignore", divide="ignore"):
        ref = flux.jacobian_blocks(m, Lx, Ly, c.Q)
    f = StsFlow(c)
    for key, got in zip("SUV", f.jacobian(dev(c.Q))):
        got, r, scale = host(got).ravel(), np.ravel(ref[key]), np.ravel(ref["scales"][key])
        if key == "S":              # T < 0: the terms of an energy entry may cancel, its scale does not show them
            scale = np.full_like(scale, scale.max())
        on = np.isfinite(r)
        assert on.sum() >= r.size - 1                    # T = 0: the source's kap / T^2 alone
        assert np.array_equal(np.isfinite(got), on), key
        assert _scaled_err(got[on], r[on], scale[on]) <= TOL_RES, key
    f.close()


@pytest.mark.parametrize("Lx,Ly", [(1, 3), (101, 6), (1, 607), (1, 608), (1, 609)])
def test_calls_behind_one_another(Lx, Ly):
    """Kernels that start early, on both sides of the line: calls with two states in turn, each
    of which overwrites the scalars that the one before it used, give what they give alone."""
    c = inputs.make_flow_case(Lx, Ly, N=9, w=1, seed=5, dt=0.3)
    f = StsFlow(c)
    states = [dev(c.Q), dev(c.Qn)]
    alone = []
    for q, qn in (states, states[::-1]):
        alone.append([host(t) for t in (f.residual(q, qn), *f.jacobian(q))])
    got = []
    for i in range(20):
        q, qn = states[i % 2], states[1 - i % 2]
        got.append((f.residual(q, qn), *f.jacobian(q)))
    for i, g in enumerate(got):
        for a, b in zip(g, alone[i % 2]):
            assert np.array_equal(host(a), b)
    f.close()
