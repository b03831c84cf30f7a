"""The general kernel's integer passes on grids of four to six axes that take
them (mg_rules.h), element by element against the oracle: axes that are just
long enough on average, uneven ones, each leading substep.

Tolerance: 1e-12 of the state's norm, the FP64 parity bar; a pass rounds every
point a few times to 2^-60 of its chunk's norm."""
import numpy as np
import pytest

import oracle
from tests import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("N", [(18, 18, 18, 36), (6, 6, 96, 96), (12, 12, 12, 12, 18), (6, 6, 8, 54, 18), (8, 6, 8, 12, 8, 16)])
def test_against_the_oracle(N, split):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1909_06412_gb300 as mg

    D = len(N)
    dq = [np.sqrt(2 * np.pi / n) for n in N]
    psi = inputs.random_state(N, seed=5) / np.sqrt(np.prod(dq))
    q, p = np.full(D, 0.3), np.full(D, -0.2)
    g, o = mg.Propagator(N, dq), oracle.Grid(N, dq)
    for x in (g, o):
        x.set_potential(mg.MG_POT_HENON_HEILES, [0.111803])
        x.set_state(psi, q, p)
    g.propagate(1, 0.02, "strang", split)
    o.propagate(1, 0.02, "strang", split)
    a, qa, pa, _ = g.get_state()
    b, qb, pb, _ = o.get_state()
    assert np.linalg.norm((a - b).ravel()) < 1e-12 * np.linalg.norm(psi.ravel())
    assert np.abs(qa - qb).max() < 1e-12 and np.abs(pa - pb).max() < 1e-12
