"""GPU: the cell strain's largest distance on both sides of the size from which
vertices are selected first, for the shapes whose selections differ most."""
import numpy as np
import pytest
from test_gpu_reductions import P  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu


def points(nv, kind):
    rng = np.random.default_rng(nv)
    x = rng.normal(size=(nv, 3))
    x /= np.linalg.norm(x, axis=1, keepdims=True)
    if kind in ("ball", "moved"):
        x *= rng.uniform(0.0, 1.0, (nv, 1)) ** (1 / 3)
    if kind == "line":
        x = np.array([1.0, 2.0, -1.0]) * rng.uniform(-1.0, 1.0, (nv, 1)) + 1e-3 * x
    x *= 9.0
    x[:4] = 0.1 * np.array([[1, 0, 0], [0, 1, 0], [0, 0, 1], [0, 0, 0]])
    return x, x + (np.array([300.0, -200.0, 90.0]) if kind == "moved" else 0.0)


@pytest.mark.parametrize("nv", [8704, 8705, 9000, 20001])
@pytest.mark.parametrize("kind", ["ball", "shell", "line", "moved"])
def test_largest_distance(P, nv, kind):  # noqa: F811
    x, y = points(nv, kind)
    ctx = P.cf_create(0)
    cid = P.cf_mesh_init(ctx, x, np.array([[0, 1, 2, 3]]), y)
    y = P.cf_get_positions(ctx, cid)
    n2 = (y * y).sum(1)
    far = max((n2[i : i + 512, None] + n2[None] - 2.0 * y[i : i + 512] @ y.T).max() for i in range(0, nv, 512))
    # FP32 positions: a rounding of at most 2^-24 |y| in each coordinate of either end
    tol = 1e-6 * np.sqrt(far) + 2 * np.sqrt(3) * 2.0**-24 * np.abs(y).max()
    assert abs(P.cf_get_cell_strain(ctx, cid, 1.0)["d_max"] - np.sqrt(far)) <= tol
    P.cf_destroy(ctx)
