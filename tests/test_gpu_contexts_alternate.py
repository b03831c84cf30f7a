"""Contexts whose kernels need different amounts of shared memory, alive at the
same time and used in turn: the larger one keeps working after a smaller one was
created.  (The limit on a kernel's dynamic shared memory is one value per kernel
function, shared by all contexts.)"""
import numpy as np
import pytest

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


def propagator(mg, N, precision):
    g = mg.Propagator(N, [np.sqrt(2 * np.pi / n) for n in N], precision=precision)
    g.set_potential(mg.MG_POT_HENON_HEILES, [0.111803])
    g.set_state(inputs.random_state(N, seed=9), [0.3] * len(N), [-0.2] * len(N))
    return g


# the larger need first: FP64 206 and 107 KB, 127 and 65 KB; FP32 198 and 191 KB;
# the general kernel's passes on the integer units and on the FP64 units
@pytest.mark.parametrize("large,small,prec", [
    ((12,) * 6, (12,) * 3, 0), ((8,) * 7, (8,) * 3, 0), ((12,) * 6, (12,) * 3, 1),
    ((128, 128, 64), (64, 54, 48), 0), ((256, 216), (16, 18), 0), ((256, 216), (16, 18), 1)])
def test_a_larger_context_outlives_a_smaller_one(mg, large, small, prec):
    alone = propagator(mg, large, prec)
    alone.propagate(2, 0.01, "strang")
    want = alone.get_state()[0]
    gs = [propagator(mg, large, prec), propagator(mg, small, prec)]
    for _ in range(2):
        for g in gs:
            g.propagate(1, 0.01, "strang")
    got = gs[0].get_state()[0]
    gs[1].sync()
    gs[0].observables()
    # two calls merge no half steps: rounding only (FP32: 6e-8 a pass)
    tol = 1e-12 if prec == 0 else 1e-5
    assert np.linalg.norm((got - want).ravel()) < tol * np.linalg.norm(want.ravel())


def test_batches_alternate(mg):
    def batch(N):
        gs = [propagator(mg, N, mg.MG_FP64) for _ in range(3)]
        return gs, mg.Batch(gs)

    large, small = batch((48, 512)), batch((16, 18))
    for _ in range(2):
        for gs, b in (large, small):
            b.propagate(1, [0.01] * 3, "strang")
            b.sync()
    assert all(np.isfinite(g.psi.cpu().numpy()).all() for g in large[0] + small[0])
