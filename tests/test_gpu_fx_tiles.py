"""The FP64 mode's fixed-point kernels beyond the small-mesh tile: all tiles of the volume kernel
on meshes of more than 600 elements (a ragged last tile), batches of such groups against contexts of fewer
(one element per block), and tiles that hold elements of every kind side by side: both tiers of the
logarithmic mean, fluxes that need the wider scales, gas at rest and jumps that go to FP64.

The sums are integers and every element chooses its own path, so the tiles agree bit for bit.  Against
the oracle the bars are those of test_gpu_parity.
"""
import numpy as np
import pytest

from oracle import dg, rk
from paper_2003_08831_gb300 import inputs
from test_gpu_parity import G, assert_rhs_close, random_state, solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def mixed_state(mesh, seed):
    """Element e is of kind perm[e] % 5: smooth, wide variation, at rest, a jump, slow and noisy."""
    rng = np.random.default_rng(seed)
    x, y, z = mesh.coords()
    kind = (rng.permutation(mesh.K) % 5).reshape(x.shape[:3])[..., None, None, None]
    k = [2 * np.pi / (mesh.hi[m] - mesh.lo[m]) for m in range(3)]
    w = np.sin(k[0] * x + 0.3) * np.cos(k[1] * y + k[2] * z)
    noise = [rng.uniform(-1, 1, x.shape) for _ in range(2)]
    rho = 1 + np.select([kind == 0, kind == 1, kind == 3], [2e-3 * w, 0.08 * noise[0], 0.0], 0.0)
    rho = np.where((kind == 3) & (noise[0] > 0), 1.8, rho)
    p = 1 + np.select([kind == 0, kind == 1, kind == 4], [2e-3 * w, 0.08 * noise[1], 1e-3 * noise[1]], 0.0)
    speed = np.select([kind == 2, kind == 4], [0.0, 1e-3], 0.3)
    return inputs.conserved(rho, speed * (0.7 + 0.1 * w), speed * np.cos(k[0] * x), speed * np.sin(k[1] * y), p, G)


@pytest.mark.parametrize("p", [2, 3, 4, 5])
@pytest.mark.parametrize("mu", [0.0, 0.02])
def test_tiles_agree_and_match_the_oracle(p, mu):
    n = (13, 7, 7)  # 637 elements: no multiple of any tile but those of 1, and 7 of them
    lo, hi = (0.0, 0.0, 0.0), (1.3, 0.7, 0.7)
    mesh = dg.Mesh(p, n, lo, hi)
    U = mixed_state(mesh, seed=p)
    phys = dg.Physics(G, mu=mu, Pr=0.72, diss=1)
    s = solver(p, n, lo, hi, mu=mu)
    q = s.to_device(U)
    from paper_2003_08831_gb300 import _binding as B
    out = []
    for v in range(3):
        B.es_set_volume_variant(s.ctx, v)
        dq, E = s.rhs(q, want_E=True)
        out.append((dq.cpu().numpy(), E.cpu().numpy()))
    assert s.status() == 0
    s.close()
    for dq, E in out[1:]:
        assert np.array_equal(dq, out[0][0]) and np.array_equal(E, out[0][1])
    assert_rhs_close(out[0][0], dg.rhs(mesh, U, phys), dg.rhs_term_magnitude(mesh, U, phys))


@pytest.mark.parametrize("p", [2, 3, 4, 5])
@pytest.mark.parametrize("mu", [0.0, 0.02])
def test_large_group_equals_small_contexts(p, mu):
    """343 + 273 + 12 elements as one group (tiles) and as contexts (one element per block), the last mesh
    100 times finer in one direction (FP64); two steps, states bit for bit."""
    from paper_2003_08831_gb300.solver import BatchSolver
    shapes = [((7, 7, 7), (0.7, 0.7, 0.7)), ((13, 7, 3), (1.3, 0.7, 0.3)), ((3, 2, 2), (0.3, 0.2, 0.002))]
    insts = [dict(p=p, n=n, lo=(0.0, 0.0, 0.0), hi=hi) for n, hi in shapes]
    meshes = [dg.Mesh(p, i["n"], i["lo"], i["hi"]) for i in insts]
    states = [mixed_state(m, seed=20 + j) if j < 2 else random_state(m, seed=p) for j, m in enumerate(meshes)]
    phys = dg.Physics(G, mu=mu, Pr=0.72, diss=1)
    dts = [0.2 * rk.stable_dt(m, U, phys, 0.5) for m, U in zip(meshes, states)]
    b = BatchSolver(insts, mu=mu)
    for i, (m, U) in enumerate(zip(meshes, states)):
        b.set_state(i, m.flat(U))
    b.set_dt(dts)
    b.advance(2)
    t, gamma = b.times()
    for i, (inst, m, U) in enumerate(zip(insts, meshes, states)):
        s = solver(p, inst["n"], inst["lo"], inst["hi"], mu=mu)
        q = s.to_device(U)
        tc, hist, _ = s.advance(q, 2, dts[i])
        assert np.array_equal(np.asarray(b.get_state(i)).reshape(-1), q.cpu().numpy().reshape(-1))
        assert gamma[i] == hist.cpu().numpy()[-1] and t[i] == tc.item()
        s.close()
    b.close()


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
