"""GPU: the memory of the on-chip relaxation's plan. Where there is none for it
the steps take launches of their own, the same bits, and the plan is made once
there is; a recorded call that finds no memory for its checkpoints takes the
plan's."""
import numpy as np
import pytest
from test_gpu_relax import P, fan  # noqa: F401 (P: the fixture)
from workloads.mesh import sphere_tet_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


def cells(P, n, general=False):  # noqa: F811
    x, t = sphere_tet_mesh(5.0, 1.4)  # 1,248 tets; 600 of them: a plan of 56 MB, checkpoints of 7
    xs = [x + np.array([20.0 * (k % 25), 20.0 * (k // 25), 3.0]) for k in range(n)]
    ts = [t] * n
    if general:
        xs, ts = xs + [fan(33)[0]], ts + [fan(33)[1]]
    ctx = P.cf_create(0)
    ids = P.cf_mesh_init_batch(ctx, xs, ts)
    P.cf_set_materials(ctx, ids, np.ones(len(xs)), np.full(len(xs), 20.0), np.full(len(xs), 0.5))
    P.cf_plates_set(ctx, 30.0, np.array([x[:, 2].min() for x in xs]), np.array([x[:, 2].max() - 0.4 for x in xs]))
    P.cf_tape_clear(ctx)
    return ctx


def fill(leave):
    """Tensors that take the device's free memory but for `leave` bytes."""
    torch.cuda.empty_cache()
    try:
        held = [torch.empty(torch.cuda.mem_get_info(0)[0] - leave - 64 * MB, dtype=torch.uint8, device="cuda:0")]
        while torch.cuda.mem_get_info(0)[0] > leave + 4 * MB:
            held.append(torch.empty(torch.cuda.mem_get_info(0)[0] - leave - 2 * MB, dtype=torch.uint8, device="cuda:0"))
    except torch.cuda.OutOfMemoryError:
        pytest.skip("the device's free memory is in use elsewhere")
    return held


def test_the_plan_gives_way(P):  # noqa: F811
    n = 600
    for general in (False, True):  # every kernel below is loaded before memory is short
        ctx = cells(P, 2, general)
        P.cf_relax(ctx, 3, 0.02, 0.9, record=True)
        P.cf_relax_adjoint(ctx, np.ones(2 + general))
        P.cf_adjoint_gradients(ctx)
        P.cf_get_positions(ctx, P.CF_ALL_CELLS)
        P.cf_destroy(ctx)
    torch.zeros(1, device="cuda:0")

    ctx = cells(P, n)
    assert P.cf_get_relax_path(ctx)["step_blocks"] > 0
    y0 = P.cf_get_positions(ctx, P.CF_ALL_CELLS)
    P.cf_relax(ctx, 5, 0.02, 0.9)
    on_chip = P.cf_get_positions(ctx, P.CF_ALL_CELLS)
    P.cf_destroy(ctx)

    ctx = cells(P, n)
    held = fill(40 * MB)
    assert P.cf_get_relax_path(ctx)["step_blocks"] == 0
    P.cf_relax(ctx, 5, 0.02, 0.9)
    assert np.array_equal(P.cf_get_positions(ctx, P.CF_ALL_CELLS), on_chip)
    del held
    torch.cuda.empty_cache()
    assert P.cf_get_relax_path(ctx)["step_blocks"] > 0

    P.cf_set_positions(ctx, P.CF_ALL_CELLS, y0)
    P.cf_tape_clear(ctx)
    held = fill(16 * MB)
    P.cf_relax(ctx, 120, 0.02, 0.9, record=True)  # four checkpoints
    assert P.cf_get_relax_path(ctx)["step_blocks"] == 0
    P.cf_relax_adjoint(ctx, np.ones(n))
    short = P.cf_adjoint_gradients(ctx)
    del held
    torch.cuda.empty_cache()

    P.cf_set_positions(ctx, P.CF_ALL_CELLS, y0)
    P.cf_tape_clear(ctx)
    P.cf_relax(ctx, 120, 0.02, 0.9, record=True)
    assert P.cf_get_relax_path(ctx)["reverse_blocks"] > 0
    P.cf_relax_adjoint(ctx, np.ones(n))
    # FP32 tangents summed in the same order: a few roundings (2^-24) a step
    assert np.linalg.norm(P.cf_adjoint_gradients(ctx) - short) <= 1e-5 * np.linalg.norm(short)
    P.cf_destroy(ctx)
