"""The FP64 mode on elements far thinner in one direction than in the others, against the oracle (the bars of
test_gpu_parity)."""
import numpy as np
import pytest

from oracle import dg
from paper_2003_08831_gb300 import inputs
from test_gpu_parity import G, assert_rhs_close, solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("p", [3, 5])
@pytest.mark.parametrize("ratio", [1e3, 1e6])
def test_flow_along_the_coarse_direction(p, ratio):
    """Nothing varies in the fine direction: its sums vanish and the coarse direction's are the result (Euler:
    the oracle's gradients of a constant are rounding times the fine metric)."""
    n, lo, hi = (3, 4, 2), (0.0, 0.0, 0.0), (3.0, 4.0, 2.0 / ratio)
    mesh = dg.Mesh(p, n, lo, hi)
    x, y, _ = mesh.coords()
    X, Y = 2 * np.pi * x / hi[0], 2 * np.pi * y / hi[1]
    U = inputs.conserved(1 + 0.02 * np.sin(X) * np.cos(Y), 0.3 * np.sin(Y) + 0.2, 0.3 * np.cos(X), 0 * x,
                         1 + 0.02 * np.cos(X + Y), G)
    # (bit for bit along x3: a vectorised sine rounds the same argument in two ways)
    U = np.ascontiguousarray(np.broadcast_to(U[:, :1, :, :, :1], U.shape))
    phys = dg.Physics(G, diss=1)
    s = solver(p, n, lo, hi)
    dq = s.rhs(s.to_device(U)).cpu().numpy()
    assert s.status() == 0
    s.close()
    assert_rhs_close(dq, dg.rhs(mesh, U, phys), dg.rhs_term_magnitude(mesh, U, phys))
