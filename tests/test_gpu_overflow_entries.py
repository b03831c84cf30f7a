"""Where single entries of a phase table overflow, or only the cross terms of a
full mass matrix do, the state is reported as not finite, and it stays so: the
kernels that carry phases as integers give no result for it, write no grid
centre from it and end at the next sum, as the FP64 passes do.  Grids of the
short-axis kernel, of the general one's integer passes (with the multipliers in
shared memory and in the workspace) and of its FP64 passes."""
import numpy as np
import pytest

from tests import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LONG = (128, 2048)
GRIDS = [(12, 12, 12), (16, 16, 16, 16), (64, 54, 48), LONG, (16, 18, 12)]


def propagator(N, minv, k, q, p, dq=1.5):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1909_06412_gb300 as mg

    D = len(N)
    g = mg.Propagator(N, [dq] * D, minv=minv)
    g.set_potential(mg.MG_POT_HARMONIC, list(k * np.eye(D).ravel()) + [0.0] * D)
    g.set_state(inputs.random_state(N, seed=4), [q] * D, [p] * D)
    assert (g.tables_in_workspace == 3) == (N == LONG)
    return mg, g


def reported(mg, g, *args):
    g.propagate(*args)
    with pytest.raises(mg.MgError) as e:
        g.sync()
    return e.value.code == mg.MG_ERR_NONFINITE


@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("N", GRIDS)
def test_a_kinetic_phase_that_overflows_on_part_of_an_axis(N, split):
    # |p| goes up to 2.09; (tau / 2) m^-1 p^2 = 1.5e308 p^2 overflows above 1.1
    mg, g = propagator(N, [7.5e307] * len(N), 1.0, 0.5, 0.0)
    assert reported(mg, g, 1, (8.0, 4.0)[split], "strang", split, mg.MG_GRID_FIXED)
    assert not np.isfinite(g.psi.cpu().numpy()).all()


@pytest.mark.parametrize("N", GRIDS)
def test_a_demodulation_phase_that_overflows(N):
    # p c dq crosses 1.8e308 two points from the centre
    mg, g = propagator(N, [1e-305] * len(N), 1.0, 0.5, 8e307)
    q, p = [0.5] * len(N), [8e307] * len(N)
    assert reported(mg, g, 3, 0.01, "strang", 0, mg.MG_GRID_ADAPTIVE)
    _, q1, p1, _ = g.get_state(want_psi=False)
    assert list(q1) == q and list(p1) == p
    # a state that is not finite is reported by every further propagation
    g.set_state(None, q, [0.0] * len(N))
    assert reported(mg, g, 1, 0.01, "strang", 0, mg.MG_GRID_FIXED)


@pytest.mark.parametrize("N", [(64, 54, 48), (16, 18, 12)])
def test_kinetic_cross_terms_that_overflow(N):
    # (tau / 2) m^-1 p^2 stays below 1.3e308 on every axis, the three cross
    # terms tau 0.9 m^-1 p_a p_b add up to 7e308 at the corners
    m = 3e307
    minv = m * (0.1 * np.eye(3) + 0.9 * np.ones((3, 3)))
    mg, g = propagator(N, minv, 1.0, 0.5, 0.0)
    assert reported(mg, g, 1, 4.0, "strang", 0, mg.MG_GRID_FIXED)
