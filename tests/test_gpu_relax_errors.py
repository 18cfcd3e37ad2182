"""GPU: a reverse pass whose vector-Jacobian products leave FP32's range ends
in CF_ENONFINITE, on chip and on the general path alike, and the context goes
on."""
import numpy as np
import pytest
from test_gpu_relax import MESHES, P, context  # noqa: F401 (P: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("case", ["tet", "small", "uneven", "large"])
@pytest.mark.parametrize("bad", [np.inf, np.nan, 1e37, 1e300])  # 1e37: lambda is finite, J m is not; 1e300 is inf in FP32
def test_a_reverse_pass_that_overflows_says_so(P, case, general, bad):  # noqa: F811
    meshes = MESHES[case]()
    n = len(meshes) + general
    ctx, _ = context(P, meshes, general, 5)
    P.cf_relax(ctx, 60, 0.02, 0.9, record=True)
    dF = np.zeros(n)
    dF[len(meshes) - 1] = bad
    with pytest.raises(P.CellFSIError) as e:
        P.cf_relax_adjoint(ctx, dF)
    assert e.value.name == "CF_ENONFINITE"
    P.cf_tape_clear(ctx)
    P.cf_relax(ctx, 60, 0.02, 0.9, record=True)
    P.cf_relax_adjoint(ctx, np.ones(n))
    assert np.isfinite(P.cf_adjoint_gradients(ctx)).all()
    P.cf_destroy(ctx)
