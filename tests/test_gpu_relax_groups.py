"""es_relax_step with elements of every kind side by side in the lane groups of one warp: unchanged,
changed by less than the floor, solved in fixed point, and two kinds that take the FP64 form (large
changes, a root far from one); a ragged last warp.

The root's relative error is that of A = sum P w.d - d_eta, a difference of terms far larger than itself:
every term is rounded a few times and they are summed, 64 units of 2^-52 of sum |P w.d| over |A| at most.
"""
import numpy as np
import pytest

from oracle import dg, gas, relax
from test_gpu_parity import EPS, G, random_state, solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("p", [2, 3, 4, 5])
def test_mixed_elements(p):
    n, lo, hi = (23, 1, 1), (0.0, 0.0, 0.0), (23.0, 1.0, 1.0)
    mesh = dg.Mesh(p, n, lo, hi)
    U = random_state(mesh, seed=p).reshape(5, mesh.K, mesh.Np)
    rng = np.random.default_rng(p)
    kind = rng.permutation(mesh.K) % 5
    size = np.array([0.0, 1e-13, 1e-2, 0.15, 1e-3])[kind]
    target = np.where(kind == 4, 2.5, 1.0 + 0.01 * rng.uniform(-1, 1, mesh.K))
    rho = U[0]
    c = np.sqrt(G * (G - 1) * (U[4] - 0.5 * (U[1:4] ** 2).sum(0) / rho) / rho)
    s = size[:, None] * rng.uniform(-1, 1, (5, mesh.K, mesh.Np))
    d = np.stack([rho * s[0], rho * c * s[1], rho * c * s[2], rho * c * s[3], U[4] * s[4]])
    new = U + d
    d = new - U  # as the library forms it
    P = np.broadcast_to(mesh.mass().reshape(-1), (mesh.K, mesh.Np))
    wd = np.sum(gas.entropy_variables(U, G) * d, axis=0)
    D = np.sum(P * relax.bregman_entropy(U, target[None, :, None] * d, G), axis=-1)
    deta = np.sum(P * wd, axis=-1) + D / target  # r(target) = D - target (sum P w.d - d_eta ...) = 0
    import torch
    sol = solver(p, n, lo, hi)
    gk, g, out = sol.relax_step(sol.to_device(U), sol.to_device(new), torch.from_numpy(deta).cuda())
    assert sol.status() == 0
    gk = gk.cpu().numpy()
    sol.close()
    free = kind < 2
    assert np.all(np.isinf(gk[free])) and np.all(np.isfinite(gk[~free]))
    A = np.sum(P * wd, axis=-1) - deta
    bound = 64 * EPS * np.sum(P * np.sum(np.abs(gas.entropy_variables(U, G) * d), axis=0), axis=-1)[~free] / np.abs(A[~free])
    assert np.all(np.abs(gk[~free] - target[~free]) <= (bound + 1e-12) * target[~free])
    assert g.item() == gk.min()
    expect = U + g.item() * d
    assert np.max(np.abs(out.cpu().numpy() - expect)) <= 4 * EPS * np.max(np.abs(expect))
