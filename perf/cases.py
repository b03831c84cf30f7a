"""Performance cases: the calls that programs make of this package, over the
range of grids, potentials, precisions and compositions it is used with.

Three families, each through the package's public entry points:
 - "propagate": a Propagator with its potential and wavepacket set advances by
   a few time steps and the grid centres are read back (with readout = 1 the
   observables too, as a program that monitors a run does);
 - "batch": many independent grids of uneven sizes advance in one launch;
 - "gradient": a forward propagation and the reversible adjoint behind
   MovingGridPropagate, for the gradient of a final-time objective.

A propagation continues from where the last pass left the state, as the loop
of a user's program does.
"""
import math

import numpy as np
import torch

import paper_1909_06412_gb300 as mg

AMU = 1822.888486  # electron masses per atomic mass unit
MU = (2.67 * AMU, 0.5 * AMU)  # reduced masses of the atom-diatom model
LAM = 0.111803  # Henon-Heiles coupling
OMEGA = (1.0, 1.2, 1.5)  # anisotropic harmonic model
DUSCHINSKY = ((1.997, -0.04, 0.017), (-0.04, 1.015, 0.04), (0.017, 0.04, 2.48))
DUSCHINSKY_OMEGA = (2.0, 1.0, 2.5)
SPLITS = {"tvt": mg.MG_TVT, "vtv": mg.MG_VTV, "tv": mg.MG_TV}
MOTIONS = {"adaptive": mg.MG_GRID_ADAPTIVE, "centre_p": mg.MG_GRID_ADAPTIVE_CENTRE_P, "fixed": mg.MG_GRID_FIXED}
KINDS = {"harmonic": mg.MG_POT_HARMONIC, "duschinsky": mg.MG_POT_HARMONIC, "atom_diatom": mg.MG_POT_ATOM_DIATOM,
         "henon_heiles": mg.MG_POT_HENON_HEILES, "secrest_johnson": mg.MG_POT_SECREST_JOHNSON}
DTS = {"harmonic": 0.01, "duschinsky": 50.0 / 512, "atom_diatom": 1.0, "henon_heiles": 0.01, "secrest_johnson": 0.1}
BATCH_2D = (64, 72, 96, 128, 144, 192, 256)
BATCH_3D = (16, 18, 24, 32, 36, 48)
# even axis lengths with factors 2 and 3
LENGTHS = sorted(2 ** a * 3 ** b for a in range(1, 12) for b in range(0, 7) if 2 ** a * 3 ** b <= 2048)


def _prop(name, kind, N, prec, scheme, steps, split="tvt", motion="adaptive", readout=0):
    return dict(name=name, family="propagate", kind=kind, N="x".join(str(n) for n in N), prec=prec, scheme=scheme,
                steps=steps, split=split, motion=motion, readout=readout)


def listed():
    return [
        # the smallest call: one second-order step of a small 2D run, with its
        # norm, energy and means read after it (a monitored run, step by step)
        _prop("harmonic_64x64_step_readout", "harmonic", (64, 64), "fp64", "strang", 1, readout=1),
        # the 3D anisotropic oscillator of the plain method, second order
        _prop("harmonic_32p3_strang", "harmonic", (32, 32, 32), "fp64", "strang", 20),
        # collinear atom-diatom scattering, fourth order, in both precisions
        _prop("atom_diatom_256x256_yoshida4", "atom_diatom", (256, 256), "fp64", "yoshida4", 10),
        _prop("atom_diatom_256x256_mixed", "atom_diatom", (256, 256), "fp32", "yoshida4", 10),
        # Secrest-Johnson collision on its wide fixed reference grid, VTV split
        _prop("secrest_johnson_128x2048_vtv", "secrest_johnson", (128, 2048), "fp64", "yoshida4", 4, "vtv", "fixed"),
        # displaced, Duschinsky-rotated oscillator (non-diagonal force
        # constants) on its dense fixed comparison grid
        _prop("duschinsky_128p3_fixed", "duschinsky", (128, 128, 128), "fp64", "yoshida4", 2, "tvt", "fixed"),
        # Henon-Heiles: a reduced-dimension run, the full 8D model in FP64 and
        # a 7D one in FP32 storage
        _prop("henon_heiles_12p4_suzuki4", "henon_heiles", (12,) * 4, "fp64", "suzuki4", 4),
        _prop("henon_heiles_12p8_yoshida4", "henon_heiles", (12,) * 8, "fp64", "yoshida4", 1),
        _prop("henon_heiles_16p7_mixed", "henon_heiles", (16,) * 7, "fp32", "suzuki4", 1),
        # 512 uneven 2D and 3D grids in one launch, FP32 storage
        dict(name="batch_512_mixed", family="batch", count=512, prec="fp32", scheme="suzuki4", steps=2),
        # gradients by the reversible adjoint, sixth order: the 2D scattering
        # model (initial state, centres and potential parameters), and 3D
        dict(name="gradient_atom_diatom_128x128", family="gradient", kind="atom_diatom", N="128x128",
             scheme="yoshida6", steps=10),
        dict(name="gradient_harmonic_64p3", family="gradient", kind="harmonic", N="64x64x64", scheme="yoshida6",
             steps=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _length(rng, lo, hi):
    """An even length with factors 2 and 3, spread over the logarithm of lo..hi."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((n for n in LENGTHS if lo <= n <= hi), key=lambda n: abs(math.log(n / x)))


def draw(rng):
    r = rng.random()
    if r < 0.12:
        return dict(family="batch", count=_log_int(rng, 24, 384), prec=rng.choice(("fp32", "fp32", "fp64")),
                    scheme=rng.choice(("strang", "yoshida4", "suzuki4")), steps=rng.randint(1, 2))
    if r < 0.27:
        if rng.random() < 0.5:
            return dict(family="gradient", kind="atom_diatom", N="%dx%d" % (_length(rng, 48, 144), _length(rng, 32, 144)),
                        scheme=rng.choice(("yoshida4", "yoshida6")), steps=rng.randint(2, 8))
        n = _length(rng, 16, 48)
        return dict(family="gradient", kind="harmonic", N="%dx%dx%d" % (n, n, _length(rng, 16, 48)),
                    scheme=rng.choice(("strang", "yoshida4")), steps=rng.randint(2, 6))
    kind = rng.choice(("harmonic", "atom_diatom", "atom_diatom", "henon_heiles", "henon_heiles", "henon_heiles",
                       "secrest_johnson", "duschinsky"))
    prec = rng.choice(("fp64", "fp64", "fp32"))
    scheme = rng.choice(("strang", "yoshida4", "suzuki4", "yoshida6"))
    split = rng.choice(("tvt", "tvt", "vtv", "tv"))
    motion = rng.choice(("adaptive", "adaptive", "adaptive", "centre_p", "fixed"))
    if kind == "harmonic":
        N = tuple(_length(rng, 16, 256) for _ in range(2)) if rng.random() < 0.5 else tuple(
            _length(rng, 12, 96) for _ in range(3))
    elif kind == "atom_diatom":
        N = (_length(rng, 64, 384), _length(rng, 48, 256))
    elif kind == "secrest_johnson":
        N = (_length(rng, 64, 256), _length(rng, 96, 2048))
        motion = "fixed" if N[1] > 512 else motion
    elif kind == "duschinsky":
        N = (_length(rng, 16, 128),) * 3
    elif rng.random() < 0.75:
        n = rng.choice((8, 12, 16))
        most = 3e8 if prec == "fp32" else 1.5e8
        N = (n,) * rng.randint(3, min(8, int(math.log(most) / math.log(n) + 1e-9)))
    else:
        N = tuple(_length(rng, 6, 36) for _ in range(rng.randint(2, 4)))
    npts = math.prod(N)
    stages = len(_coefficients(scheme)) + 1
    steps = max(1, min(_log_int(rng, 1, 24), int(6e8 / (npts * stages))))
    case = _prop("", kind, N, prec, scheme, steps, split, motion, int(rng.random() < 0.2))
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# Problems: grids, potentials and packets, with a seeded spread
# ---------------------------------------------------------------------------


def _shape(case):
    return tuple(int(n) for n in case["N"].split("x"))


def _morse_mean(Dm, a, re, mass):
    """<r> of the Morse ground state: re - (digamma(2 lam - 1) - ln 2 lam) / a."""
    lam = math.sqrt(2.0 * mass * Dm) / a
    return re - (float(torch.digamma(torch.tensor(2.0 * lam - 1.0, dtype=torch.float64))) - math.log(2.0 * lam)) / a


def _problem(kind, N, seed, span=20.48):
    """dict: N, dq, minv (diagonal), kind, pot (what set_potential takes), fac
    (per-axis factors of the packet), q, p (centres), dt.  span: the range of
    the atom-diatom grid in R."""
    g = np.random.default_rng(seed)
    D = len(N)
    out = dict(kind=kind, N=N, dt=DTS[kind])
    if kind == "harmonic":
        om = np.array([OMEGA[l % 3] for l in range(D)]) * g.uniform(0.9, 1.1, D)
        q = np.array([(1.0, -0.5, 0.8)[l % 3] for l in range(D)]) + g.uniform(-0.3, 0.3, D)
        p = np.array([(0.0, 0.5, -0.3)[l % 3] for l in range(D)]) + g.uniform(-0.3, 0.3, D)
        out.update(dq=[9.6 / n for n in N], minv=[1.0] * D, pot=list(np.diag(om ** 2).ravel()) + [0.0] * D,
                   fac=[("gauss", q[l], p[l], om[l] ** -0.5) for l in range(D)], q=q, p=p)
    elif kind == "duschinsky":
        q0 = np.array([-7.0, 7.0, 7.0])
        q = g.uniform(-0.3, 0.3, 3)
        out.update(dq=[14.0 * math.sqrt(n / 32.0) / n for n in N], minv=list(DUSCHINSKY_OMEGA),
                   pot=list(np.array(DUSCHINSKY).ravel()) + list(q0),
                   fac=[("gauss", q[l], 0.0, 1.0) for l in range(3)], q=q + 0.25 * q0, p=np.zeros(3))
    elif kind == "atom_diatom":
        f = g.uniform(0.95, 1.05, 5)
        Dm, a, re, A, be = 0.17 * f[0], 1.0 * f[1], 1.4 * f[2], 5.0 * f[3], 1.8 * f[4]
        R0, P0 = 8.0 + g.uniform(-0.5, 0.5), -10.0 + g.uniform(-1, 1)
        out.update(dq=[span / N[0], 10.24 / N[1]], minv=[1 / MU[0], 1 / MU[1]], pot=[Dm, a, re, A, be],
                   fac=[("gauss", R0, P0, 0.5), ("morse", Dm, a, re, MU[1])],
                   q=np.array([R0, _morse_mean(Dm, a, re, MU[1])]), p=np.array([P0, 0.0]))
    elif kind == "henon_heiles":
        # displaced Gaussians: q = 2 on the large grids, well inside the
        # barrier on the small ones, whose runs are long
        q = (2.0 if math.prod(N) > 1e6 else 0.5) + g.uniform(-0.1, 0.1, D)
        out.update(dq=[math.sqrt(2 * math.pi / n) for n in N], minv=[1.0] * D, pot=[LAM],
                   fac=[("gauss", q[l], 0.0, 1.0) for l in range(D)], q=q, p=np.zeros(D))
    else:
        # ranges (-14, 14) x (0, 48), or (-50, 400) for the long reference axis
        lo, hi = (-50.0, 400.0) if N[1] > 512 else (0.0, 48.0)
        q2, p2 = 24.0 + g.uniform(-1, 1), -3.56 + g.uniform(-0.2, 0.2)
        out.update(dq=[28.0 / N[0], (hi - lo) / N[1]], minv=[1.0, 1.5], pot=[20.0, 0.158, 0.3],
                   fac=[("gauss", 0.0, 0.0, 1.0), ("gauss", q2, p2, 8.0 ** 0.5)],
                   q=np.array([0.0, lo + (hi - lo) / 2]), p=np.array([0.0, p2]))
    return out


def _batch_problems(count, seed):
    """Half 2D grids (half of them atom-diatom, half harmonic), half 3D."""
    g = np.random.default_rng(seed)
    sizes = np.random.default_rng(20190913)  # the same uneven sizes for every seed
    out = []
    for i in range(count):
        if i < count // 2:
            kind = "atom_diatom" if i % 2 else "harmonic"
            N = tuple(int(sizes.choice(BATCH_2D)) for _ in range(2))
        else:
            kind, N = "harmonic", tuple(int(sizes.choice(BATCH_3D)) for _ in range(3))
        out.append(_problem(kind, N, int(g.integers(1 << 30))))
    return out


def _propagator(P, prec):
    h = mg.Propagator(P["N"], P["dq"], minv=P["minv"], precision=mg.MG_FP64 if prec == "fp64" else mg.MG_FP32_MIXED)
    h.set_potential(KINDS[P["kind"]], P["pot"])
    h.set_separable(P["fac"], P["q"], P["p"])
    return h


def prepare(case, seed):
    fam = case["family"]
    if fam == "propagate":
        P = _problem(case["kind"], _shape(case), seed)
        return dict(case=case, h=_propagator(P, case["prec"]), dt=P["dt"])
    if fam == "batch":
        Ps = _batch_problems(case["count"], seed)
        hs = [_propagator(P, case["prec"]) for P in Ps]
        return dict(case=case, hs=hs, b=mg.Batch(hs), dt=np.array([P["dt"] for P in Ps]))
    P = _problem(case["kind"], _shape(case), seed, 10.24)
    h = _propagator(P, "fp64")
    u0 = h.psi.view(torch.complex128).clone().reshape(P["N"])
    # the target of the overlap term: the same packet, moved and turned
    target = torch.roll(u0, 1, 0) * np.exp(0.3j)
    return dict(case=case, h=h, dt=P["dt"], u0=u0.requires_grad_(), target=target,
                q0=torch.tensor(P["q"], dtype=torch.float64, requires_grad=True),
                p0=torch.tensor(P["p"], dtype=torch.float64, requires_grad=True),
                theta=torch.tensor(_theta(P), dtype=torch.float64, requires_grad=True))


def _theta(P):
    if P["kind"] != "atom_diatom":
        return []
    Dm, a, _, A, be = P["pot"]
    return [Dm, a, be, A]


def _stored(x, case):
    """Numbers formed from a state, in the type its values are stored in: those
    of a run with FP32 storage carry no more than its rounding leaves."""
    return np.asarray(x, dtype=np.float64 if case["prec"] == "fp64" else np.float32)


def run(state):
    case = state["case"]
    if case["family"] == "propagate":
        h = state["h"]
        h.propagate(case["steps"], state["dt"], case["scheme"], SPLITS[case["split"]], MOTIONS[case["motion"]])
        _, q, p, _ = h.get_state(want_psi=False)
        out = dict(psi=h.psi, q=_stored(q, case), p=_stored(p, case))
        if case["readout"]:
            norm, energy, mq, mp = h.observables()
            out.update(norm=_stored(norm, case), energy=_stored(energy, case), mean_q=_stored(mq, case),
                       mean_p=_stored(mp, case))
        return out
    if case["family"] == "batch":
        b = state["b"]
        b.propagate(case["steps"], state["dt"], case["scheme"])
        b.sync()
        centres = [h.get_state(want_psi=False)[1:3] for h in state["hs"]]
        return dict(psi=torch.cat([h.psi for h in state["hs"]]), q=_stored(np.concatenate([c[0] for c in centres]), case),
                    p=_stored(np.concatenate([c[1] for c in centres]), case))
    from paper_1909_06412_gb300.autograd import MovingGridPropagate

    u0, q0, p0, theta = state["u0"], state["q0"], state["p0"], state["theta"]
    uT, qT, pT = MovingGridPropagate.apply(u0, q0, p0, theta, state["h"], case["steps"], state["dt"], case["scheme"])
    loss = qT[0] + (torch.vdot(state["target"].reshape(-1), uT.reshape(-1)).abs() ** 2).cpu()
    leaves = [u0, q0, p0] + ([theta] if theta.numel() else [])
    grads = torch.autograd.grad(loss, leaves)
    # the gradient by the state, and the one by all parameters
    return dict(loss=loss.detach(), uT=uT.detach(), qT=qT.detach(), pT=pT.detach(), grad_u=grads[0],
                grad=torch.cat(grads[1:]))


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------


def _stage_flops(N):
    """One kinetic unit with its potential substep: two transforms (5 N log2 N
    each), the phase factors and the two reductions."""
    D, npts = len(N), math.prod(N)
    return npts * (10.0 * math.log2(npts) + 10.0 * D + 2.0 * (D + 2))


def work(case):
    fam = case["family"]
    S = len(_coefficients(case["scheme"])) * case["steps"]
    if fam == "batch":
        shapes = [P["N"] for P in _batch_problems(case["count"], 0)]
        size = 16 if case["prec"] == "fp64" else 8
        return dict(bytes=2.0 * size * sum(math.prod(N) for N in shapes), flops=S * sum(_stage_flops(N) for N in shapes))
    N = _shape(case)
    if fam == "gradient":
        # forward; then state and cotangent backwards
        return dict(bytes=16.0 * math.prod(N) * 4, flops=3.0 * S * _stage_flops(N))
    size = 16 if case["prec"] == "fp64" else 8
    reads = 2 + (1 if case["readout"] else 0)
    return dict(bytes=float(size) * math.prod(N) * reads, flops=S * _stage_flops(N))


# ---------------------------------------------------------------------------
# The same results in plain 64-bit torch
# ---------------------------------------------------------------------------


def _coefficients(scheme):
    """Stage coefficients of a symmetric composition: triple jump or Suzuki fractal."""
    order = int(scheme[7:] if scheme.startswith("yoshida") else scheme[6:]) if scheme != "strang" else 2
    g = [1.0]
    for k in range(1, order // 2):
        e = 1.0 / (2 * k + 1)
        if scheme.startswith("yoshida"):
            a = 1.0 / (2.0 - 2.0 ** e)
            w = [a, 1.0 - 2.0 * a, a]
        else:
            a = 1.0 / (4.0 - 4.0 ** e)
            w = [a, a, 1.0 - 4.0 * a, a, a]
        g = [x * y for x in w for y in g]
    return g


def _substeps(scheme, split, steps, dt):
    out = []
    for _ in range(steps):
        for g in _coefficients(scheme):
            out += {"tvt": [("T", g * dt / 2), ("V", g * dt), ("T", g * dt / 2)],
                    "vtv": [("V", g * dt / 2), ("T", g * dt), ("V", g * dt / 2)],
                    "tv": [("V", g * dt), ("T", g * dt)]}[split]
    merged = []
    for kind, t in out:  # neighbours of a kind commute
        if merged and merged[-1][0] == kind:
            merged[-1] = (kind, merged[-1][1] + t)
        else:
            merged.append((kind, t))
    return merged


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _axis(v, l, D):
    return v.reshape([-1 if a == l else 1 for a in range(D)])


def _initial(P):
    """u on the grid centred at (q, p): the product of the packet's factors."""
    D, dev = len(P["N"]), _device()
    u = None
    for l, f in enumerate(P["fac"]):
        c = torch.arange(P["N"][l], dtype=torch.float64, device=dev) - P["N"][l] // 2
        x = P["q"][l] + c * P["dq"][l]
        if f[0] == "gauss":
            d = x - f[1]
            v = (math.pi * f[3] ** 2) ** -0.25 * torch.exp(-d * d / (2 * f[3] ** 2)) * torch.exp(1j * f[2] * d)
        else:
            Dm, a, re, mass = f[1:]
            lam = math.sqrt(2.0 * mass * Dm) / a
            lz = math.log(2.0 * lam) - a * (x - re)
            lognorm = 0.5 * (math.log(a) - math.lgamma(2.0 * lam - 1.0))
            v = torch.exp(lognorm + (lam - 0.5) * lz - 0.5 * torch.exp(lz)) + 0j
        v = _axis(v * math.sqrt(P["dq"][l]), l, D)
        u = v if u is None else u * v
    return u


def _potential(P, x, theta):
    """V and the list of dV/dx_a, as arrays that broadcast to the grid."""
    D, kind, pot = len(P["N"]), P["kind"], P["pot"]
    x = [_axis(x[a], a, D) for a in range(D)]
    if kind in ("harmonic", "duschinsky"):
        d = [x[a] - pot[D * D + a] for a in range(D)]
        if kind == "harmonic":  # a diagonal force-constant matrix
            g = [pot[a * D + a] * d[a] for a in range(D)]
        else:
            g = [sum(pot[a * D + b] * d[b] for b in range(D)) for a in range(D)]
        return 0.5 * sum(d[a] * g[a] for a in range(D)), g
    if kind == "atom_diatom":
        (Dm, a, be, A), re = theta, pot[2]
        em = torch.exp(-a * (x[1] - re))
        eR, ep, en = torch.exp(-be * x[0]), torch.exp(0.5 * be * x[1]), torch.exp(-0.5 * be * x[1])
        V = Dm * (1 - em) ** 2 + A * eR * (ep + en)
        return V, [-be * A * eR * (ep + en), 2 * Dm * a * (1 - em) * em + 0.5 * be * A * eR * (ep - en)]
    if kind == "henon_heiles":
        V, g = 0.0, []
        for a in range(D):
            V = V + 0.5 * x[a] ** 2 - (LAM * x[a] ** 3 / 3 if a >= 1 else 0.0)
            if a + 1 < D:
                V = V + LAM * x[a] ** 2 * x[a + 1]
            g.append(x[a] - (LAM * x[a] ** 2 if a >= 1 else 0.0) + (2 * LAM * x[a] * x[a + 1] if a + 1 < D else 0.0)
                     + (LAM * x[a - 1] ** 2 if a >= 1 else 0.0))
        return V, g
    Dm, be, al = pot
    e1, c = torch.exp(-be * x[0]), torch.exp(al * x[0]) * torch.exp(-al * x[1])
    return Dm * (1 - e1) ** 2 + c, [2 * Dm * be * (1 - e1) * e1 + al * c, -al * c]


def _propagate(P, u, q, p, theta, substeps, motion):
    """The moving-grid split-operator steps, plainly: (u, q, p) after them."""
    D, N, dev = len(P["N"]), P["N"], u.device
    c = [torch.arange(n, dtype=torch.float64, device=dev) - n // 2 for n in N]
    dp = [2 * math.pi / (N[l] * P["dq"][l]) for l in range(D)]
    sign = [1.0 - 2.0 * (torch.arange(n, device=dev) % 2) for n in N]
    q, p = list(q), list(p)
    for kind, t in substeps:
        if kind == "T":
            A = [_axis(sign[l] * torch.exp(-1j * p[l] * c[l] * P["dq"][l]), l, D) for l in range(D)]
            for l in range(D):
                u = u * A[l]
            u = torch.fft.fftn(u)
            w = u.real ** 2 + u.imag ** 2
            n = w.sum()
            for l in range(D):
                mean = p[l] + dp[l] * (w * _axis(c[l], l, D)).sum() / n
                d = 0.0 if motion == "fixed" else t * P["minv"][l] * (mean if motion == "adaptive" else p[l])
                pk = p[l] + c[l] * dp[l]
                u = u * _axis(torch.exp(1j * (d * pk - 0.5 * t * P["minv"][l] * pk ** 2)), l, D)
                q[l] = q[l] + d
            del w
            u = torch.fft.ifftn(u)
            for l in range(D):
                u = u * A[l].conj()
        else:
            V, g = _potential(P, [q[l] + c[l] * P["dq"][l] for l in range(D)], theta)
            if motion != "fixed":
                w = u.real ** 2 + u.imag ** 2
                n = w.sum()
                for l in range(D):
                    p[l] = p[l] - t * (w * g[l]).sum() / n
                del w
            u = u * torch.exp(-1j * t * V)
    return u, q, p


def _observables(P, u, q, p):
    D, N, dev = len(P["N"]), P["N"], u.device
    c = [torch.arange(n, dtype=torch.float64, device=dev) - n // 2 for n in N]
    x = [q[l] + c[l] * P["dq"][l] for l in range(D)]
    w = u.real ** 2 + u.imag ** 2
    norm = w.sum()
    V, _ = _potential(P, x, P["theta"])
    phi = u
    for l in range(D):
        phi = phi * _axis((1.0 - 2.0 * (torch.arange(N[l], device=dev) % 2)) * torch.exp(-1j * p[l] * c[l] * P["dq"][l]), l, D)
    phi = torch.fft.fftn(phi)
    k = phi.real ** 2 + phi.imag ** 2
    pk = [p[l] + c[l] * 2 * math.pi / (N[l] * P["dq"][l]) for l in range(D)]
    kin = sum((k * _axis(0.5 * P["minv"][l] * pk[l] ** 2, l, D)).sum() for l in range(D)) / k.sum()
    return dict(norm=np.array(float(norm)), energy=np.array(float(kin + (w * V).sum() / norm)),
                mean_q=np.array([float((w * _axis(x[l], l, D)).sum() / norm) for l in range(D)]),
                mean_p=np.array([float((k * _axis(pk[l], l, D)).sum() / k.sum()) for l in range(D)]))


def _reals(u):
    return torch.view_as_real(u.contiguous()).reshape(-1)


def _scalars(v):
    return [torch.tensor(float(x), dtype=torch.float64, device=_device()) for x in v]


def exact(case, seed):
    if case["family"] == "propagate":
        P = _problem(case["kind"], _shape(case), seed)
        P["theta"] = _theta(P)
        sub = _substeps(case["scheme"], case["split"], case["steps"], P["dt"])
        with torch.no_grad():
            u, q, p = _propagate(P, _initial(P), _scalars(P["q"]), _scalars(P["p"]), P["theta"], sub, case["motion"])
            out = dict(psi=_reals(u), q=np.array([float(v) for v in q]), p=np.array([float(v) for v in p]))
            if case["readout"]:
                out.update(_observables(P, u, q, p))
        return out
    if case["family"] == "batch":
        psi, qs, ps = [], [], []
        with torch.no_grad():
            for P in _batch_problems(case["count"], seed):
                sub = _substeps(case["scheme"], "tvt", case["steps"], P["dt"])
                u, q, p = _propagate(P, _initial(P), _scalars(P["q"]), _scalars(P["p"]), _theta(P), sub, "adaptive")
                psi.append(_reals(u))
                qs += [float(v) for v in q]
                ps += [float(v) for v in p]
        return dict(psi=torch.cat(psi), q=np.array(qs), p=np.array(ps))
    P = _problem(case["kind"], _shape(case), seed, 10.24)
    u0 = _initial(P)
    target = torch.roll(u0, 1, 0) * np.exp(0.3j)
    u0 = u0.detach().requires_grad_()
    q0 = [x.requires_grad_() for x in _scalars(P["q"])]
    p0 = [x.requires_grad_() for x in _scalars(P["p"])]
    theta = [x.requires_grad_() for x in _scalars(_theta(P))]
    sub = _substeps(case["scheme"], "tvt", case["steps"], P["dt"])
    uT, qT, pT = _propagate(P, u0, q0, p0, theta, sub, "adaptive")
    loss = qT[0] + torch.vdot(target.reshape(-1), uT.reshape(-1)).abs() ** 2
    gr = torch.autograd.grad(loss, [u0] + q0 + p0 + theta)
    return dict(loss=loss.detach().cpu(), uT=uT.detach(), qT=torch.stack([x.detach().cpu() for x in qT]),
                pT=torch.stack([x.detach().cpu() for x in pT]), grad_u=gr[0],
                grad=torch.stack([g.detach().cpu() for g in gr[1:]]))
