"""A phase that overflows is reported as a state that is not finite, also by
the kernels that carry phases as integers (which have no NaN): the potential's
and the kinetic one's, on grids of the short-axis kernel, of the general one's
integer passes and of its FP64 passes."""
import numpy as np
import pytest

from tests import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("what", ["potential", "kinetic"])
@pytest.mark.parametrize("N", [(12, 12, 12), (16, 16, 16, 16), (64, 54, 48), (16, 18, 12)])
def test_an_overflowing_phase_is_reported(N, what, split):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1909_06412_gb300 as mg

    D = len(N)
    k, m = (1e307, 1.0) if what == "potential" else (1.0, 1e307)
    g = mg.Propagator(N, [1.5] * D, minv=[m] * D)
    g.set_potential(mg.MG_POT_HARMONIC, list(k * np.eye(D).ravel()) + [0.0] * D)
    g.set_state(inputs.random_state(N, seed=4), [10.0] * D, [20.0] * D)
    g.propagate(1, 1.0, "strang", split, mg.MG_GRID_FIXED)
    with pytest.raises(mg.MgError) as e:
        g.sync()
    assert e.value.code == mg.MG_ERR_NONFINITE
