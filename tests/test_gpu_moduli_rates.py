"""GPU: the moduli gradient and the directional derivative of the forces
against 64 bits where they are hardest (a large rotation, kappa = 500 mu), each
modulus on its own, and over the range of FP32 directions."""
import numpy as np
import pytest

import oracle
from test_gpu_reductions import P, load, part  # noqa: F401 (P: the fixture)
from workloads.configs import Cell
from workloads.mesh import sphere_tet_mesh

pytestmark = pytest.mark.gpu

TOL = 1e-5  # the bound of the other force and gradient tests


def rotation(seed):
    q = np.linalg.qr(np.random.default_rng(seed).normal(size=(3, 3)))[0]
    return q * np.sign(np.linalg.det(q))


def state(kind):
    """A cell, and the part of its deformation that strains it: a direction along which every tet's energies grow."""
    x, t = sphere_tet_mesh(8.0, 1.5)
    rng = np.random.default_rng(5)
    off = 0.1 * rng.uniform(-1.0, 1.0, x.shape)
    A = {"noise": np.eye(3), "rotated": rotation(3), "turned_over": np.diag([-1.0, -1.0, 1.0]),
         "stretched": rotation(4) @ np.diag([1.1, 0.95, 1.02])}[kind]
    x = x + np.array([11.0, 12.0, 13.0])
    y = x.mean(0) + (x - x.mean(0)) @ A.T + off
    return Cell(x, t, y, 1.3, 650.0, 0.35), off


@pytest.mark.parametrize("kind", ["noise", "rotated", "turned_over", "stretched"])
def test_each_modulus_and_the_derivative(P, kind):  # noqa: F811
    cell, lam = state(kind)
    ctx, (cid,) = load(P, [cell])
    y = P.cf_get_positions(ctx, cid)
    m = oracle.Mesh([cell])
    got = P.cf_force_param_vjp(ctx, lam)[0]

    def dot(mu, kappa, w):  # lambda . f; the forces are linear in the moduli
        m.mu[:], m.kappa[:], m.w[:] = mu, kappa, w
        return float((lam * m.forces(y)).sum())

    g1, g2, gk = dot(1.0, 0.0, 1.0), dot(1.0, 0.0, 0.0), dot(0.0, 1.0, 0.5)
    ref = np.array([cell.w * g1 + (1.0 - cell.w) * g2, gk, cell.mu * (g1 - g2)])
    # d/dw is a difference of two nearly equal energies' rates: held to their size
    assert (np.abs(got - ref) <= TOL * np.abs([ref[0], ref[1], cell.mu * g1])).all(), (got, ref)

    m.mu[:], m.kappa[:], m.w[:] = cell.mu, cell.kappa, cell.w
    v = np.random.default_rng(6).normal(size=y.shape)
    e = 1e-3  # five points: an error of e^4 (some 1e-11 here) beside the oracle's rounding over e
    ref = sum(k * m.forces(y + s * e * v) for k, s in ((8.0, 1.0), (-8.0, -1.0), (-1.0, 2.0), (1.0, -2.0))) / (12.0 * e)
    got = P.cf_force_jvp(ctx, v)
    assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref)
    P.cf_destroy(ctx)


@pytest.mark.parametrize("sizes", [(1,), (33, 95), (700, 3)])
def test_the_gradient_scales_with_the_direction(P, sizes):  # noqa: F811
    """Powers of two near both ends of FP32's range change the result by exactly that factor; blocks of one cell and of two."""
    ctx, _ = load(P, [part(n, k) for k, n in enumerate(sizes)])
    nv = len(P.cf_get_positions(ctx, P.CF_ALL_CELLS))
    lam = np.random.default_rng(9).uniform(0.5, 1.0, (nv, 3)).astype(np.float32).astype(np.float64)
    base = P.cf_force_param_vjp(ctx, lam)
    assert np.isfinite(base).all() and (base != 0.0).any()
    for k in (127, 100, -60, -100, -125):
        got = P.cf_force_param_vjp(ctx, lam * 2.0**k)
        # one warp: the same additions; several add their sums to the cell's in any order of the atomics
        assert np.abs(got * 2.0**-k - base).max() <= (0.0 if sum(sizes) <= 32 else 1e-12) * np.abs(base).max()
    P.cf_destroy(ctx)


def test_a_non_finite_direction_stays_in_its_cell(P):  # noqa: F811
    cells = [part(40, 0), part(300, 1), part(500, 2)]
    ctx, _ = load(P, cells)
    n = [len(c.x_ref) for c in cells]
    lam = np.random.default_rng(10).normal(size=(sum(n), 3))
    base = P.cf_force_param_vjp(ctx, lam)
    lam[n[0] + 7, 1] = np.inf
    got = P.cf_force_param_vjp(ctx, lam)
    assert not np.isfinite(got[1]).any()
    assert np.allclose(got[[0, 2]], base[[0, 2]], rtol=1e-12, atol=0.0)
    P.cf_destroy(ctx)


def test_reverse_steps_scale_with_the_loss(P):  # noqa: F811
    """A reverse pass on chip, the plate force's weight near both ends of FP32's range."""
    x, t = sphere_tet_mesh(5.0, 1.4)
    grads = []
    for k in (0, 70, -90):
        ctx = P.cf_create(0)
        (cid,) = P.cf_mesh_init_batch(ctx, [x], [t], [x])
        P.cf_set_materials(ctx, [cid], [1.0], [20.0], [0.5])
        P.cf_plates_set(ctx, 32.0, [x[:, 2].min()], [x[:, 2].max() - 0.3])
        P.cf_tape_clear(ctx)
        P.cf_relax(ctx, 70, 0.02, 0.9, record=True)
        assert P.cf_get_relax_path(ctx)["reverse_blocks"] > 0
        P.cf_relax_adjoint(ctx, [2.0**k])
        grads.append(P.cf_adjoint_gradients(ctx) * 2.0**-k)
        P.cf_destroy(ctx)
    # two launches add their blocks' sums in any order of the atomics
    for g in grads[1:]:
        assert np.abs(g - grads[0]).max() <= 1e-12 * np.abs(grads[0]).max()
