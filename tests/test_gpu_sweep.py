"""GPU: lattices swept to and fro (their populations exceed L2) against a
narrow one. A forced channel between moving walls that starts at rest is
uniform along x and z, so every column of a wide lattice equals the column of
a narrow one, bit for bit, whichever way the planes are taken."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2003_03130_gb300 import build

    build.build()
    import paper_2003_03130_gb300 as P

    return P


def channel(P, nx, nz, fmt, steps):
    ctx = P.cf_create(0)
    P.cf_set_population_format(ctx, fmt)
    P.cf_lbm_init(ctx, nx, 40, nz, 0.9, -0.02, 0.03, (1e-5, 0.0, 0.0))
    P.cf_step(ctx, steps)
    u, rho = P.cf_get_velocity(ctx), P.cf_get_density(ctx)
    P.cf_destroy(ctx)
    return u, rho


@pytest.mark.parametrize("fmt", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,nz,steps", [(256, 161, 1), (256, 161, 14), (131, 320, 13), (512, 201, 6)])
def test_wide_channel_equals_a_narrow_one(P, fmt, nx, nz, steps):
    u, rho = channel(P, nx, nz, fmt, steps)
    un, rn = channel(P, 4, 3, fmt, steps)
    assert np.array_equal(u, np.broadcast_to(un[:1, :, :1], u.shape))
    assert np.array_equal(rho, np.broadcast_to(rn[:1, :, :1], rho.shape))
