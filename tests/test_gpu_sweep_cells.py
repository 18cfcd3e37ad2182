"""GPU: a cell in a lattice that is swept to and fro (both buffers larger than
L2), the step split into far and near field: rows that follow the sweep and
the list of region tiles that does not, one step a call and several, give the
same bits in every storage format, stochastic rounding included."""
import numpy as np
import pytest
from test_gpu_sweep import P  # noqa: F401 (the fixture)
from workloads.mesh import perturb, sphere_tet_mesh

pytestmark = pytest.mark.gpu

SHAPES = [({}, 1), ({"near_rows": 1}, 7), ({"tile_x": 8, "tile_y": 8, "tile_z": 4, "far_spec": 1}, 7),
          ({"near_rows": 1, "mark_k5": 1, "tile_x": 32, "tile_y": 2, "tile_z": 4}, 2)]


@pytest.mark.parametrize("fmt", ["f32", "f16", "bf16", "f16sr", "bf16sr"])
def test_rows_and_tiles_of_a_swept_lattice_agree(P, fmt):  # noqa: F811
    nx, ny, nz, steps = 140, 131, 130, 7  # 2 x 19 x 2 bytes a node: 181 MB
    x, t = sphere_tet_mesh(8.0, 1.6)
    x = x + np.array([3.0, 66.0, 127.0])  # across the periodic boundaries
    got = []
    for shape, per_call in SHAPES:
        ctx = P.cf_create(0)
        P.cf_set_population_format(ctx, fmt)
        P.cf_set_spread(ctx, "fixed")
        ids = P.cf_mesh_init_batch(ctx, [x], [t], [perturb(x, 0.1, 3)])
        P.cf_set_materials(ctx, ids, [1e-3], [5e-2], [0.4])
        P.cf_set_launch_shape(ctx, {**P.cf_get_launch_shape(ctx), "pop_pairs": 0, **shape})
        P.cf_lbm_init(ctx, nx, ny, nz, 0.8, -0.03, 0.02, (1e-5, 0.0, 2e-6))
        for k in range(0, steps, per_call):
            P.cf_step(ctx, min(per_call, steps - k))
        got.append((P.cf_get_positions(ctx, ids[0]), P.cf_get_density(ctx)))
        P.cf_destroy(ctx)
    for y, rho in got[1:]:
        assert np.array_equal(y, got[0][0]) and np.array_equal(rho, got[0][1])
