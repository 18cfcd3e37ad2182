"""GPU: the reductions behind the moduli gradient, the energy, the Taylor
deformation and the cell strain at the sizes where they can go wrong (warps
that straddle cells, one block and one more, single tets, point sets without
an inside), against the FP64 oracle or a direct evaluation."""
import numpy as np
import pytest

import oracle
from oracle import analysis
from workloads.configs import Cell
from workloads.mesh import perturb, sphere_tet_mesh

pytestmark = pytest.mark.gpu

TOL = 1e-5  # the bound of the other force and gradient tests
MESH_X, MESH_T = sphere_tet_mesh(9.0, 1.5)


@pytest.fixture(scope="module")
def P():
    from paper_2003_03130_gb300 import build

    build.build()
    import paper_2003_03130_gb300 as P

    return P


def part(nt, k=0, mu=1.0, kappa=20.0, w=0.4):
    """The first nt tets of a sphere as a cell of their own, off the rest shape."""
    t = MESH_T[:nt]
    used, t = np.unique(t, return_inverse=True)
    x = MESH_X[used] + np.array([20.0 * k, 3.0, -5.0])
    return Cell(x, t.reshape(-1, 4).astype(np.int32), perturb(x, 0.08, 50 + k), mu * (1 + 0.1 * k), kappa, w)


def load(P, cells):
    ctx = P.cf_create(0)
    ids = P.cf_mesh_init_batch(ctx, [c.x_ref for c in cells], [c.tets for c in cells], [c.y0 for c in cells])
    P.cf_set_materials(ctx, ids, [c.mu for c in cells], [c.kappa for c in cells], [c.w for c in cells])
    return ctx, ids


@pytest.mark.parametrize("sizes", [(1,), (31,), (32, 33), (127, 1, 1, 3, 128), (2000, 1)])
def test_moduli_gradient(P, sizes):
    cells = [part(n, k) for k, n in enumerate(sizes)]
    ctx, _ = load(P, cells)
    m = oracle.Mesh(cells)
    lam = np.random.default_rng(4).normal(size=m.x.shape)
    got = P.cf_force_param_vjp(ctx, lam)
    y = P.cf_get_positions(ctx, P.CF_ALL_CELLS)
    mu, kappa, w = m.mu.copy(), m.kappa.copy(), m.w.copy()

    def dots(a, b, c):  # lambda . f per cell; the forces are linear in the moduli
        m.mu[:], m.kappa[:], m.w[:] = a, b, c
        return np.array([(lam[i:j] * m.forces(y)[i:j]).sum() for i, j in m.vert_ranges])

    g1, g2, gk = dots(1.0, 0.0, 1.0), dots(1.0, 0.0, 0.0), dots(0.0, 1.0, 0.5)
    ref = np.stack([w * g1 + (1 - w) * g2, gk, mu * (g1 - g2)], axis=1)
    assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref)
    P.cf_destroy(ctx)
