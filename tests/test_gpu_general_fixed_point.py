"""The general kernel's passes on the integer units, taken by FP64 grids with
at least 1024 points per SM.  Grids just above that line, with every radix,
tables in shared memory and in the workspace, two to eight axes, each leading
substep, a full mass matrix and states that are hard to scale.  Element by
element against the oracle.

Tolerance: 1e-12 of the state's norm, the FP64 parity bar.  A pass rounds
every point to a grid of 2^-60 of its chunk's norm once per multiplication:
with at most five a pass (multiplier, three twiddles, phase), 7000 points a
chunk and sixteen passes the worst case is 80 * 84 * 2^-60 = 6e-15, and FP64
itself (oracle and tables) adds 2^-53 per operation, below 1e-14."""
import numpy as np
import pytest

import oracle
from tests import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def mg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1909_06412_gb300 as m

    m.lib()
    return m


def run(mg, N, kind, pot, minv=None, split=0, motion=0, scale=None):
    D = len(N)
    dq = [np.sqrt(2 * np.pi / n) for n in N]
    minv = np.ones(D) if minv is None else np.asarray(minv)
    u = inputs.random_state(N, seed=5)
    if scale == "decades":
        u *= 10.0 ** np.random.default_rng(6).uniform(-200, 0, N)
    elif scale == "empty":
        u[: N[0] // 2] = 0
    elif scale is not None:
        u *= scale
    psi = u / np.sqrt(np.prod(dq))
    q, p = np.full(D, 0.3), np.full(D, -0.2)
    g = mg.Propagator(N, dq, minv=minv)
    o = oracle.Grid(N, dq, minv=minv)
    for x in (g, o):
        x.set_potential(kind, pot)
        x.set_state(psi, q, p)
    assert g.path == 0
    g.propagate(2, 0.02, "strang", split, motion)
    o.propagate(2, 0.02, "strang", split, motion)
    a, qa, pa, _ = g.get_state()
    b, qb, pb, _ = o.get_state()
    norm = np.linalg.norm(psi.ravel())
    assert np.linalg.norm(((a - b) / norm).ravel()) < TOL
    assert np.abs(qa - qb).max() < TOL * max(1.0, np.abs(qb).max())
    assert np.abs(pa - pb).max() < TOL * max(1.0, np.abs(pb).max())


@pytest.mark.parametrize("split", [0, 1, 2])
@pytest.mark.parametrize("N", [(54, 54, 54), (162, 972), (8, 162, 162), (64, 64, 64), (128, 2048),
                               (96, 1728), (24,) * 4, (6, 8, 6, 8, 6, 12), (4,) * 7 + (12,)])
def test_grids_above_the_line(mg, N, split):
    run(mg, N, mg.MG_POT_HENON_HEILES, [0.111803], split=split)


@pytest.mark.parametrize("scale", ["decades", "empty", 1e-120, 1e120])
def test_states_of_uneven_magnitude(mg, scale):
    run(mg, (54, 64, 48), mg.MG_POT_HENON_HEILES, [0.111803], scale=scale, motion=2)


def test_full_mass_matrix_and_general_harmonic(mg):
    m = [[1.0, 0.25, -0.1], [0.25, 0.8, 0.15], [-0.1, 0.15, 1.2]]
    K = [1.0, 0.1, 0.0, 0.1, 1.44, 0.2, 0.0, 0.2, 2.25, 0.1, -0.2, 0.0]
    run(mg, (64, 54, 48), mg.MG_POT_HARMONIC, K, minv=m)


def test_a_nan_is_reported(mg):
    N = (64, 54, 48)
    g = mg.Propagator(N, [0.5] * 3)
    g.set_potential(mg.MG_POT_HENON_HEILES, [0.111803])
    u = inputs.random_state(N, seed=4)
    u[5, 6, 7] = np.nan
    g.set_state(u, [0.0] * 3, [0.0] * 3)
    g.propagate(1, 0.01, "strang")
    with pytest.raises(mg.MgError) as e:
        g.sync()
    assert e.value.code == mg.MG_ERR_NONFINITE
