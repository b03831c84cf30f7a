"""The FP64 passes on the integer units are no less accurate than those on the
FP64 units.  Localised packets on moving grids, where a rounding with a mean
error adds up over the passes, against the same substeps in the host's long
double; mg_propagate_noalloc runs the general kernel's passes on the FP64 units.

Bound: the error of the integer passes is at most that of the FP64 units' passes
on the same problem.  What both share (FP64 tables, one rounding per pass where
the state is stored) is in both; the transforms add 2^-53 per operation on the
FP64 units and about 2^-58 of a chunk's norm on the integer units."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
fft = pytest.importorskip("scipy.fft")
pytestmark = pytest.mark.gpu

L, CL = np.longdouble, np.clongdouble
LAM = 0.111803


def cis(t):
    r = np.empty(t.shape, dtype=CL)
    r.real, r.imag = np.cos(t), np.sin(t)
    return r


def along(v, l, D):
    return v.reshape([-1 if a == l else 1 for a in range(D)])


def reference(u, q, p, dq, gam, dt, om2):
    """TVT steps of the moving-grid method; om2: diagonal force constants, or
    None for Henon-Heiles."""
    D, N, dt = u.ndim, u.shape, L(dt)
    sub = []
    for g in gam:
        for kind, t in (("T", L(g) * dt / 2), ("V", L(g) * dt), ("T", L(g) * dt / 2)):
            if sub and sub[-1][0] == kind:
                sub[-1] = (kind, sub[-1][1] + t)
            else:
                sub.append((kind, t))
    c = [np.arange(n).astype(L) - n // 2 for n in N]
    dq = [L(x) for x in dq]
    dp = [L(2.0 * math.pi / (n * float(h))) for n, h in zip(N, dq)]
    u, q, p = u.astype(CL), [L(x) for x in q], [L(x) for x in p]
    for kind, t in sub:
        if kind == "T":
            A = [along((1 - 2 * (np.arange(N[l]) % 2)) * cis(-p[l] * c[l] * dq[l]), l, D) for l in range(D)]
            for l in range(D):
                u = u * A[l]
            u = fft.fftn(u, workers=-1)
            w = u.real ** 2 + u.imag ** 2
            n = w.sum()
            for l in range(D):
                d = t * (p[l] + dp[l] * (w * along(c[l], l, D)).sum() / n)
                pk = p[l] + c[l] * dp[l]
                u = u * along(cis(d * pk - t * pk ** 2 / 2), l, D)
                q[l] = q[l] + d
            u = fft.ifftn(u, workers=-1)
            for l in range(D):
                u = u * np.conj(A[l])
        else:
            x = [along(q[l] + c[l] * dq[l], l, D) for l in range(D)]
            w = u.real ** 2 + u.imag ** 2
            n = w.sum()
            if om2 is not None:
                g = [L(k) * y for k, y in zip(om2, x)]
                for l in range(D):
                    u = u * cis(-t * g[l] * x[l] / 2)
            else:
                lam, g, V = L(LAM), list(x), 0
                for a in range(D):
                    V = V + x[a] ** 2 / 2 - (lam * x[a] ** 3 / 3 if a else 0) + (lam * x[a] ** 2 * x[a + 1] if a + 1 < D else 0)
                    g[a] = g[a] - (lam * x[a] ** 2 if a else 0) + (2 * lam * x[a] * x[a + 1] if a + 1 < D else 0)
                    g[a] = g[a] + (lam * x[a - 1] ** 2 if a else 0)
                u = u * cis(-t * V)
            for l in range(D):
                p[l] = p[l] - t * (w * g[l]).sum() / n
    return u


@pytest.mark.parametrize("N,scheme,steps", [((12,) * 4, "suzuki4", 4), ((16,) * 4, "suzuki4", 2), ((8,) * 5, "suzuki4", 2),
                                            ((54,) * 3, "yoshida6", 1)])
def test_no_less_accurate_than_the_fp64_units(N, scheme, steps):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1909_06412_gb300 as mg

    D = len(N)
    short = N[0] <= 16
    om2 = None if short else [1.0, 1.44, 2.25]
    dq = [math.sqrt(2 * math.pi / n) for n in N]
    q, p = np.array([0.5 - 0.1 * l for l in range(D)]), np.array([0.1 * l for l in range(D)])
    kind, pot = (mg.MG_POT_HENON_HEILES, [LAM]) if short else (mg.MG_POT_HARMONIC, list(np.diag(om2).ravel()) + [0.0] * D)
    g = mg.Propagator(N, dq)
    g.set_potential(kind, pot)
    g.set_separable([("gauss", q[l], p[l], 1.0) for l in range(D)], q, p)
    assert g.path == (1 if short else 0)
    u0 = g.psi.clone()
    gam = [float(x) for x in mg.mg_scheme_coefficients(scheme)] * steps
    want = reference(u0.view(torch.complex128).reshape(N).cpu().numpy(), q, p, dq, gam, 0.01, om2)
    g.propagate(steps, 0.01, scheme)
    g.sync()
    qn, pn = q.copy(), p.copy()
    mg.mg_propagate_noalloc(N, dq, np.ones(D), 1.0, kind, pot, u0, qn, pn, steps, 0.01, scheme)
    err = [float(np.sqrt((np.abs(x.view(torch.complex128).reshape(N).cpu().numpy() - want) ** 2).sum())) for x in (g.psi, u0)]
    assert err[0] <= err[1], err
