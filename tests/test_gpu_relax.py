"""GPU: relaxation with the cells' state on chip (csrc/relax.cu) against the
general path of three launches a step: the same positions, velocities
(through the following steps) and forces bit for bit, and the same gradients
up to rounding. One vertex with more incidences than the on-chip path takes
sends a context down the general path, so the same cells run both ways."""
import numpy as np
import pytest

from workloads.mesh import perturb, sphere_tet_mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2003_03130_gb300 import build

    build.build()
    import paper_2003_03130_gb300 as P

    return P


def fan(n):
    """n tets around one edge: both of its ends have n incidences."""
    a = 2 * np.pi * np.arange(n) / n
    x = np.concatenate([[[0, 0, -2.0], [0, 0, 2.0]], np.stack([4 * np.cos(a), 4 * np.sin(a), 0 * a], 1)])
    k = np.arange(n)
    return x, np.stack([0 * k, 0 * k + 1, 2 + k, 2 + (k + 1) % n], 1).astype(np.int32)


def sphere_part(nt):
    x, t = sphere_tet_mesh(6.0, 1.5)
    used, t = np.unique(t[:nt], return_inverse=True)
    return x[used], t.reshape(-1, 4).astype(np.int32)


MESHES = {
    "tet": lambda: [(np.eye(4, 3) * 3.0, np.array([[0, 1, 2, 3]], np.int32))],  # fewer vertices than blocks may be
    "small": lambda: [sphere_part(1), sphere_part(513), sphere_tet_mesh(5.0, 1.4)],  # around a round of threads
    "degree_32": lambda: [fan(32), sphere_tet_mesh(4.0, 1.5)],  # the most incidences that fit
    "uneven": lambda: [sphere_tet_mesh(r, 1.4) for r in (3.0, 10.0, 6.5)],  # clusters of several blocks
    "large": lambda: [sphere_tet_mesh(14.0, 1.72)],  # eight blocks
    "too_large": lambda: [sphere_tet_mesh(16.0, 1.4), sphere_tet_mesh(4.0, 1.5)],  # no room on chip: the general path
}


def context(P, meshes, general, seed):
    if general:
        meshes = meshes + [fan(33)]
    rng = np.random.default_rng(seed)
    xs = [x + np.array([40.0 * k, 3.0, 7.0]) for k, (x, _) in enumerate(meshes)]
    ys = [perturb(x, 0.03, 10 * seed + k) for k, x in enumerate(xs)]
    ctx = P.cf_create(0)
    ids = P.cf_mesh_init_batch(ctx, xs, [t for _, t in meshes], ys)
    n = len(meshes)
    P.cf_set_materials(ctx, ids, 1.0 + 0.1 * np.arange(n), 20.0 + np.arange(n), 0.3 + 0.05 * np.arange(n))
    z_lo = np.array([x[:, 2].min() for x in xs])
    z_hi = np.array([x[:, 2].max() for x in xs]) - 0.3
    P.cf_plates_set(ctx, 30.0, z_lo, z_hi)
    P.cf_tape_clear(ctx)
    return ctx, ids


def common(P, ctx, n):
    return [P.cf_get_positions(ctx, k) for k in range(n)], [P.cf_get_forces(ctx, k) for k in range(n)]


@pytest.mark.parametrize("case", list(MESHES))
@pytest.mark.parametrize("stiff", [False, True])
def test_steps_match_the_general_path_bit_for_bit(P, case, stiff):
    meshes = MESHES[case]()
    got = []
    for general in (False, True):
        ctx, ids = context(P, meshes, general, 3)
        if stiff:  # the FP64 volume, and materials per tet
            n = len(meshes[-1][1])
            P.cf_set_material(ctx, ids[0], 0.5, 60.0, 0.4)
            P.cf_set_tet_materials(ctx, ids[len(meshes) - 1], np.arange(n) % 2, [1.0, 0.2], [20.0, 30.0], [0.5, 0.1])
        P.cf_relax(ctx, 1, 0.02, 0.9)
        one = common(P, ctx, len(meshes))
        P.cf_relax(ctx, 37, 0.02, 0.9)
        got.append((one, common(P, ctx, len(meshes))))
        P.cf_destroy(ctx)
    for a, b in zip(got[0], got[1]):
        for x, y in zip(a[0] + a[1], b[0] + b[1]):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("case", list(MESHES))
@pytest.mark.parametrize("steps", [1, 50, 51, 120])
def test_gradients_match_the_general_path(P, case, steps):
    meshes = MESHES[case]()
    n = len(meshes)
    grads = []
    for general in (False, True):
        ctx, _ = context(P, meshes, general, 4)
        P.cf_relax(ctx, steps, 0.02, 0.9, record=True)
        dF = np.zeros(n + general)
        dF[:n] = 1.0 + 0.5 * np.arange(n)
        P.cf_relax_adjoint(ctx, dF)
        grads.append(P.cf_adjoint_gradients(ctx)[:n])
        P.cf_destroy(ctx)
    # FP32 tangents summed in the same order: a few roundings (2^-24) a step
    assert np.linalg.norm(grads[0] - grads[1]) <= 1e-5 * np.linalg.norm(grads[1])
