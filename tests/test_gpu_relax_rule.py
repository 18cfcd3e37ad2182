"""GPU: sets of cells that are slower on chip than in launches of their own
take the launches: cells in many waves, and one large cell that cuts many
small ones into as many blocks. More cells than multiprocessors that stay on
chip take the same steps as the general path, bit for bit."""
import numpy as np
import pytest
from test_gpu_relax import P, common, fan  # noqa: F401 (P: the fixture)
from workloads.mesh import perturb, sphere_tet_mesh

pytestmark = pytest.mark.gpu

TINY, SMALL = (3.0, 1.5), (5.0, 1.4)  # 192 and 1,248 tets
SETS = {  # cells, and whether steps and reverse steps go on chip
    "few": ([(8, SMALL)], True, True),
    "as_many_as_fill": ([(64, SMALL)], True, True),
    "two_waves": ([(160, TINY)], True, True),
    "many_waves": ([(2000, TINY)], False, False),
    "medium_beside_small": ([(1, (10.0, 1.45)), (63, TINY)], False, False),
    "large_beside_small": ([(1, (14.0, 1.72)), (300, TINY)], False, False),
    "large_cells": ([(24, (14.0, 1.72))], None, False),
}


def meshes(name):
    return [m for n, q in SETS[name][0] for m in [sphere_tet_mesh(*q)] * n]


def context(P, meshes, general, seed):
    meshes = meshes + [fan(33)] * general  # a vertex with more incidences than the on-chip steps take
    n = len(meshes)
    xs = [x + np.array([40.0 * (k % 16), 40.0 * (k // 16), 7.0]) for k, (x, _) in enumerate(meshes)]
    ctx = P.cf_create(0)
    ids = P.cf_mesh_init_batch(ctx, xs, [t for _, t in meshes], [perturb(x, 0.03, seed + k) for k, x in enumerate(xs)])
    at = np.arange(n) % 10
    P.cf_set_materials(ctx, ids, 1.0 + 0.1 * at, 20.0 + at, 0.3 + 0.05 * at)
    P.cf_plates_set(ctx, 30.0, np.array([x[:, 2].min() for x in xs]), np.array([x[:, 2].max() for x in xs]) - 0.3)
    P.cf_tape_clear(ctx)
    return ctx


@pytest.mark.parametrize("name", list(SETS))
def test_the_faster_way_is_taken(P, name):  # noqa: F811
    ctx = context(P, meshes(name), False, 6)
    path = P.cf_get_relax_path(ctx)
    for key, want in zip(("step_blocks", "reverse_blocks"), SETS[name][1:]):
        if want is not None:
            assert (path[key] > 0) == want, (key, path)
    P.cf_destroy(ctx)


@pytest.mark.parametrize("name", ["two_waves", "as_many_as_fill"])
def test_more_cells_than_slots_match_the_general_path(P, name):  # noqa: F811
    m = meshes(name)
    n, got, grads = len(m), [], []
    for general in (False, True):
        ctx = context(P, m, general, 7)
        P.cf_relax(ctx, 53, 0.02, 0.9, record=True)
        got.append(common(P, ctx, n))
        dF = np.zeros(n + general)
        dF[:n] = 1.0 + 0.01 * np.arange(n)
        P.cf_relax_adjoint(ctx, dF)
        grads.append(P.cf_adjoint_gradients(ctx)[:n])
        assert (P.cf_get_relax_path(ctx)["reverse_blocks"] == 0) == general
        P.cf_destroy(ctx)
    for x, y in zip(got[0][0] + got[0][1], got[1][0] + got[1][1]):
        assert np.array_equal(x, y)
    # FP32 tangents summed in the same order: a few roundings (2^-24) a step
    assert np.linalg.norm(grads[0] - grads[1]) <= 1e-5 * np.linalg.norm(grads[1])


@pytest.mark.parametrize("name", ["few", "two_waves"])
def test_calls_of_few_steps_take_the_same_steps(P, name):  # noqa: F811
    """The way on chip prepared beforehand, so that single steps take it, and left to the steps that make it worth it."""
    got = []
    for prepare in (True, False):
        ctx = context(P, meshes(name), False, 8)
        if prepare:
            assert P.cf_get_relax_path(ctx)["step_blocks"] > 0
        for n in (1, 1, 2, 27, 1, 40):
            P.cf_relax(ctx, n, 0.02, 0.9)
            got.append(P.cf_get_positions(ctx, P.CF_ALL_CELLS))
        P.cf_destroy(ctx)
    for a, b in zip(got[:6], got[6:]):
        assert np.array_equal(a, b)
