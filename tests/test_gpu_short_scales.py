"""The FP64 short-axis kernel carries chunks of the state as 64-bit integers
with a scale per chunk.  States whose chunks are hard to scale: one point, one
flat chunk, magnitudes over hundreds of decades, very small and very large
norms, empty chunks, a NaN.  Element by element against the oracle, on a grid
that stays in place (the sums that move it are compared by the parity tests).

Tolerance.  A pass rounds every point to the integer grid, at most 2^-50 of
its chunk's norm over the chunk's points, and FP64 differs from exact
arithmetic by as much; one Strang step is two kinetic units of at most six
passes: 24 * 2^-50 = 2.1e-14, stated as 1e-13 of the state's norm."""
import numpy as np
import pytest

import oracle
from tests import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1909_06412_gb300 as m

    m.lib()
    return m


def make_state(kind, N):
    rng = np.random.default_rng(7)
    u = inputs.random_state(N, seed=3)
    if kind == "point":
        u[:] = 0
        u[tuple(n // 2 for n in N)] = 1 - 0.5j
    elif kind == "flat":
        u[:] = (0.6 - 0.8j) / np.sqrt(u.size)
    elif kind == "decades":
        u *= 10.0 ** rng.uniform(-200, 0, N)
        u[tuple(n // 2 for n in N)] = 1.0
    elif kind == "empty":
        u[: N[0] // 2] = 0
    elif kind == "tiny":
        u *= 1e-120
    elif kind == "huge":
        u *= 1e120
    return u


@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("N", [(8, 8, 8), (8,) * 5, (12, 12, 12), (12,) * 5, (16, 16, 16), (16,) * 4])
@pytest.mark.parametrize("kind", ["point", "flat", "decades", "empty", "tiny", "huge"])
def test_states_of_uneven_magnitude(mg, kind, N, split):
    D = len(N)
    dq = [np.sqrt(2 * np.pi / n) for n in N]
    u = make_state(kind, N)
    psi = u / np.sqrt(np.prod(dq))
    q, p, fixed = np.full(D, 0.3), np.full(D, -0.2), 2
    g = mg.Propagator(N, dq)
    g.set_potential(mg.MG_POT_HENON_HEILES, [0.111803])
    g.set_state(psi, q, p)
    o = oracle.Grid(N, dq)
    o.set_potential(oracle.POT_HENON_HEILES, [0.111803])
    o.set_state(psi, q, p)
    assert g.path == 1
    g.propagate(1, 0.05, "strang", split, fixed)
    o.propagate(1, 0.05, "strang", split, fixed)
    a, b = g.get_state()[0], o.get_state()[0]
    scale = np.linalg.norm(psi.ravel())
    assert np.linalg.norm((a - b).ravel() / scale) < 1e-13


def test_a_nan_is_reported(mg):
    N = (12, 12, 12)
    g = mg.Propagator(N, [0.7] * 3)
    g.set_potential(mg.MG_POT_HENON_HEILES, [0.111803])
    u = inputs.random_state(N, seed=4)
    u[5, 6, 7] = np.nan
    g.set_state(u, [0.0] * 3, [0.0] * 3)
    g.propagate(1, 0.01, "strang")
    with pytest.raises(mg.MgError) as e:
        g.sync()
    assert e.value.code == mg.MG_ERR_NONFINITE
