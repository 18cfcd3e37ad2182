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


@pytest.mark.parametrize("nt", [40, 255, 256, 257, 1500])
def test_energy_and_taylor(P, nt):
    cell = part(nt)
    ctx, (cid,) = load(P, [cell])
    y = P.cf_get_positions(ctx, cid)
    m = oracle.Mesh([cell])
    assert abs(P.cf_get_energy(ctx, cid) - m.energy(y)) <= TOL * m.energy(y)
    got, ref = P.cf_get_taylor(ctx, cid), analysis.taylor(y, m.tets)
    assert abs(got["D"] - ref["D"]) <= 1e-6 and abs(got["theta1"] - ref["theta"][0]) <= 1e-6 * ref["theta"][0]
    P.cf_destroy(ctx)


@pytest.mark.parametrize("nv", [4, 255, 256, 257, 1023, 1024, 1025, 2600])
@pytest.mark.parametrize("kind", ["ball", "shell", "line", "moved"])
def test_cell_strain(P, nv, kind):
    """Point sets with one tet: all but the kept ones are pruned (ball), none is (shell), two ends (line), far off (moved)."""
    rng = np.random.default_rng(nv)
    x = rng.normal(size=(nv, 3))
    x /= np.linalg.norm(x, axis=1, keepdims=True)
    if kind in ("ball", "moved"):
        x *= rng.uniform(0.0, 1.0, (nv, 1)) ** (1 / 3)
    if kind == "line":
        x = np.array([1.0, 2.0, -1.0]) * rng.uniform(-1.0, 1.0, (nv, 1)) + 1e-3 * x
    x *= 9.0
    x[:4] = 0.1 * np.array([[1, 0, 0], [0, 1, 0], [0, 0, 1], [0, 0, 0]])
    y = x + (np.array([300.0, -200.0, 90.0]) if kind == "moved" else 0.0)
    ctx = P.cf_create(0)
    cid = P.cf_mesh_init(ctx, x, np.array([[0, 1, 2, 3]]), y)
    y = P.cf_get_positions(ctx, cid)
    ref = np.sqrt(((y[:, None] - y[None]) ** 2).sum(-1).max())
    # FP32 positions: a rounding of at most 2^-24 |y| in each coordinate of either end
    assert abs(P.cf_get_cell_strain(ctx, cid, 1.0)["d_max"] - ref) <= 1e-6 * ref + 2 * np.sqrt(3) * 2.0**-24 * np.abs(y).max()
    P.cf_destroy(ctx)
