"""GPU: which way relaxation steps go (cf_get_relax_path): the contexts that
the other relaxation tests compare really run differently."""
import pytest
from test_gpu_relax import MESHES, P, context  # noqa: F401 (P: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", list(MESHES))
def test_compared_contexts_take_different_paths(P, case):  # noqa: F811
    ctx, _ = context(P, MESHES[case](), False, 3)
    path = P.cf_get_relax_path(ctx)
    assert (path["step_blocks"] > 0) == (case != "too_large") and path["step_blocks"] <= 8
    P.cf_relax(ctx, 2, 0.02, 0.9)
    assert P.cf_get_relax_path(ctx) == path
    P.cf_destroy(ctx)
    ctx, _ = context(P, MESHES[case](), True, 3)  # a vertex with 33 incidences more
    path = P.cf_get_relax_path(ctx)
    assert path["step_blocks"] == path["reverse_blocks"] == 0 and path["steps_per_launch"] > 0
    P.cf_destroy(ctx)


def test_the_path_needs_cells(P):  # noqa: F811
    ctx = P.cf_create(0)
    with pytest.raises(P.CellFSIError) as e:
        P.cf_get_relax_path(ctx)
    assert e.value.name == "CF_ESTATE"
    P.cf_destroy(ctx)
