"""What the speed of this framework is measured on.

Twelve listed cases, and drawn ones over the same ranges: time steps of one
lifted bilayer (1D boxes of every size, 2D boxes, complex64 and complex128, the
deterministic and the stochastic schemes), the batched runner, the gradient of
a final overlap, the wave function at real-space points, and the observables.
Sizes are those of ``workloads.py``, of the tests and of ``bench.py``.

Every case goes through the public entry points (``Context``, ``Batch``,
``overlap_loss``).  Problems are described here, so that ``exact`` (the same
quantities by plain torch in 64 bits) shares no code with the framework.
"""
import math

import numpy as np
import torch

import paper_2103_14897_gb300 as P
from paper_2103_14897_gb300.autograd import overlap_loss

GOLDEN = (math.sqrt(5.0) - 1.0) / 2.0
MASK64 = (1 << 64) - 1
DOF_STEPS = 2049 * 2049 * 20          # lifted elements x time steps of the largest 1D complex64 call


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the small complex128 bilayer (the paper's scale of box): 100 Strang steps per
        # call; the whole state is 68 KB, so latency and launches count
        dict(name="step-65-c128", kind="step", n1=32, n2=32, dtype="c128", scheme="strang", steps=100, tau=1e-3),
        # an uneven complex64 box of ordinary size (a batch instance run alone), Lie steps
        dict(name="step-401x129-c64", kind="step", n1=200, n2=64, dtype="c64", scheme="lie", steps=50, tau=1e-3),
        # the bilayer at scale: 2049 x 2049, complex64, second order
        dict(name="step-2049-c64", kind="step", n1=1024, n2=1024, dtype="c64", scheme="strang", steps=20, tau=5e-4),
        # the same box with the stochastic scheme (1/8 of the slices per sub-step)
        dict(name="step-2049-c64-stoch", kind="step", n1=1024, n2=1024, dtype="c64", scheme="strang_stoch",
             steps=20, tau=5e-4),
        # the same box in complex128: the reference run that the complex64 one is compared with
        dict(name="step-2049-c128", kind="step", n1=1024, n2=1024, dtype="c128", scheme="strang", steps=4, tau=5e-4),
        # the twisted 2D bilayer on its 64^4 box
        dict(name="twisted-64-c64", kind="twisted", q=64, dtype="c64", scheme="strang", steps=5, tau=1e-3),
        # the twisted bilayer on a smaller box: slices of 32 x 32
        dict(name="twisted-32-c64", kind="twisted", q=32, dtype="c64", scheme="strang", steps=10, tau=1e-3),
        # 256 uneven bilayers in one call (parameter studies over L2 and the amplitudes)
        dict(name="batch-256-c64", kind="batch", count=256, nmin=16, nmax=512, shapes=4, dtype="c64",
             scheme="strang", steps=10, tau=1e-3),
        # a smaller batch with the stochastic scheme
        dict(name="batch-64-c64-stoch", kind="batch", count=64, nmin=16, nmax=512, shapes=4, dtype="c64",
             scheme="strang_stoch", steps=10, tau=1e-3),
        # fitting the layer potentials: loss and gradient of a final overlap with respect to
        # 8 cosine coefficients per layer (forward and reverse sweep)
        dict(name="gradient-513-c64", kind="gradient", n=256, harmonics=8, dtype="c64", steps=100, tau=1e-3),
        # the wave function on a line of 4096 points (the localisation plots)
        dict(name="density-2049-c64", kind="density", n1=1024, n2=1024, dtype="c64", points=4096),
        # mass, energy and mean momentum between calls of the stepper
        dict(name="observables-2049-c64", kind="observables", n1=1024, n2=1024, dtype="c64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "twisted", "batch", "gradient", "density", "observables"])
    if kind == "step":
        c = dict(kind=kind, n1=_log_int(rng, 16, 1024), n2=_log_int(rng, 16, 1024),
                 dtype=rng.choice(["c64", "c64", "c64", "c128"]),
                 scheme=rng.choice(["strang", "strang", "lie", "strang_kp", "strang_stoch"]),
                 steps=_log_int(rng, 4, 100), tau=rng.choice([5e-4, 1e-3]))
        cap = DOF_STEPS if c["dtype"] == "c64" else DOF_STEPS // 5
        c["steps"] = max(1, min(c["steps"], cap // ((2 * c["n1"] + 1) * (2 * c["n2"] + 1))))
        return c
    if kind == "twisted":
        q = rng.choice([8, 16, 32, 64])
        dtype = rng.choice(["c64", "c64", "c64", "c128"])
        cap = DOF_STEPS if dtype == "c64" else DOF_STEPS // 5
        return dict(kind=kind, q=q, dtype=dtype, scheme=rng.choice(["strang", "lie", "strang_kp"]),
                    steps=max(1, min(_log_int(rng, 4, 40), cap // q ** 4)), tau=1e-3)
    if kind == "batch":
        return dict(kind=kind, count=_log_int(rng, 8, 256), nmin=16, nmax=_log_int(rng, 64, 512),
                    shapes=rng.randrange(1 << 20), dtype="c64",
                    scheme=rng.choice(["strang", "lie", "strang_stoch"]), steps=_log_int(rng, 4, 10), tau=1e-3)
    if kind == "gradient":
        return dict(kind=kind, n=_log_int(rng, 32, 256), harmonics=rng.randrange(1, 9), dtype="c64",
                    steps=_log_int(rng, 10, 100), tau=1e-3)
    if kind == "density":
        return dict(kind=kind, n1=_log_int(rng, 64, 1024), n2=_log_int(rng, 64, 1024), dtype="c64",
                    points=_log_int(rng, 64, 4096))
    return dict(kind=kind, n1=_log_int(rng, 32, 1024), n2=_log_int(rng, 32, 1024),
                dtype=rng.choice(["c64", "c64", "c128"]))


# ------------------------------------------------------------------ problems
class Problem:
    """A lifted bilayer as ``Context`` takes it (the fields of workloads.Problem)."""

    def __init__(self, d, B1, B2, lo1, q1, lo2, q2, ecut, v1, v2):
        self.d, self.B1, self.B2 = d, np.asarray(B1, dtype=np.float64), np.asarray(B2, dtype=np.float64)
        self.lo1, self.q1, self.lo2, self.q2 = tuple(lo1), tuple(q1), tuple(lo2), tuple(q2)
        self.ecut, self.shared = float(ecut), 0
        (self.v1_h, self.v1_c), (self.v2_h, self.v2_c) = v1, v2

    M1 = property(lambda self: math.prod(self.q1))
    M2 = property(lambda self: math.prod(self.q2))

    def with_potentials(self, v1_c=None, v2_c=None, v1_h=None, v2_h=None):
        return Problem(self.d, self.B1, self.B2, self.lo1, self.q1, self.lo2, self.q2, self.ecut,
                       (np.asarray(v1_h, dtype=np.int64).reshape(-1, 1), np.asarray(v1_c, dtype=np.complex128)),
                       (np.asarray(v2_h, dtype=np.int64).reshape(-1, 1), np.asarray(v2_c, dtype=np.complex128)))


def _cos(amps):
    """sum_h amps[h - 1] cos(2 pi h x / L) as harmonics and coefficients."""
    h, c = [], []
    for k, a in enumerate(amps, start=1):
        h += [[k], [-k]]
        c += [a / 2.0, a / 2.0]
    return np.array(h, dtype=np.int64), np.array(c, dtype=np.complex128)


def _bilayer(n1, n2, a1, a2, L2=GOLDEN):
    return Problem(1, [[2 * math.pi]], [[2 * math.pi / L2]], (-n1,), (2 * n1 + 1,), (-n2,), (2 * n2 + 1,),
                   200.0 * (n1 / 32.0) ** 2, _cos([a1]), _cos([a2]))


def _wells(rng, hmax=8, sigma=0.15):
    """Three Gaussian wells per cell, truncated to |h_i| <= hmax."""
    depth, centre = rng.uniform(1.0, 3.0, 3), rng.uniform(0.0, 1.0, (3, 2))
    h = np.array([[i, j] for i in range(-hmax, hmax + 1) for j in range(-hmax, hmax + 1)], dtype=np.int64)
    env = 2 * math.pi * sigma ** 2 * np.exp(-sigma ** 2 * (2 * math.pi) ** 2 * (h ** 2).sum(1) / 2)
    return h, -(depth[None, :] * np.exp(-2j * math.pi * (h @ centre.T))).sum(1) * env


def _twisted(q, seed):
    rng = np.random.default_rng(seed)
    c, s = math.cos(math.radians(5.0)), math.sin(math.radians(5.0))
    lo, hmax = -(q // 2), min(8, q // 2 - 1)
    return Problem(2, 2 * math.pi * np.eye(2), 2 * math.pi * np.array([[c, -s], [s, c]]),
                   (lo, lo), (q, q), (lo, lo), (q, q), 200.0, _wells(rng, hmax), _wells(rng, hmax))


def _problems(case, seed):
    """The problem (or the batch's problems) of a case; the seed draws the amplitudes."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "twisted":
        return [_twisted(case["q"], seed)]
    if kind == "batch":
        shapes = np.random.default_rng(case["shapes"])
        out = []
        for _ in range(case["count"]):
            L2 = float(shapes.uniform(0.3, 0.9))
            n1, n2 = (int(x) for x in shapes.integers(case["nmin"], case["nmax"] + 1, size=2))
            a1, a2 = rng.uniform(0.5, 2.0, size=2)
            out.append(_bilayer(n1, n2, a1, a2, L2))
        return out
    a1, a2 = rng.uniform(0.5, 2.0, size=2)
    n1, n2 = (case["n"], case["n"]) if kind == "gradient" else (case["n1"], case["n2"])
    return [_bilayer(n1, n2, a1, a2)]


def _k(p):
    """Components of k = B1 m + B2 n, each (M2, M1), float64 on the GPU."""
    def index(lo, q):
        if p.d == 1:
            return (np.arange(q[0]) + lo[0]).reshape(1, -1)
        b, a = np.meshgrid(np.arange(q[1]) + lo[1], np.arange(q[0]) + lo[0], indexing="ij")
        return np.stack([a.reshape(-1), b.reshape(-1)])
    k1 = torch.from_numpy(p.B1 @ index(p.lo1, p.q1)).cuda()
    k2 = torch.from_numpy(p.B2 @ index(p.lo2, p.q2)).cuda()
    return [k1[i][None, :] + k2[i][:, None] for i in range(p.d)]


def _kinetic(p):
    return 0.5 * sum(x * x for x in _k(p))


def _states(p, dtype, seed, count=1):
    """Normalised states as the stepper meets them: a Gaussian packet on the joint cutoff with
    seeded width, place and momentum, and over the whole box a tail, as an evolved state has."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed + 1)
    k = _k(p)
    inside = sum(x * x for x in k) * 0.5 <= p.ecut
    out = []
    for _ in range(count):
        w = rng.uniform(0.5, 2.0) * 3.0 / math.sqrt(2.0 * p.ecut)
        x0, k0 = rng.uniform(-0.5, 0.5, p.d), rng.uniform(-1.0, 1.0, p.d)
        amp = torch.exp(-0.5 * w * w * sum((x - c) ** 2 for x, c in zip(k, k0))) * inside
        phase = -sum(x * c for x, c in zip(k, x0))
        z = torch.polar(amp, phase)
        z /= torch.linalg.vector_norm(z)
        tail = torch.randn(z.shape, generator=gen, device="cuda", dtype=torch.complex128)
        z += 0.1 * tail / torch.linalg.vector_norm(tail)
        z /= torch.linalg.vector_norm(z)
        out.append(z.to(torch.complex64 if dtype == "c64" else torch.complex128))
    return out


def _pitch(p):
    return (p.M1 + 15) // 16 * 16


def _padded(p, z):
    out = torch.zeros((p.M2, _pitch(p)), dtype=z.dtype, device=z.device)
    out[:, :p.M1] = z
    return out


def _points(case, seed):
    return np.random.default_rng(seed + 2).uniform(-20.0, 20.0, case["points"])


def _thetas(case, seed):
    th = np.random.default_rng(seed + 3).normal(0.0, 0.5, size=(2, case["harmonics"]))
    return torch.from_numpy(th[0].copy()), torch.from_numpy(th[1].copy())


# ------------------------------------------------------------------ a user's program
def prepare(case, seed):
    probs = _problems(case, seed)
    p, dtype, kind = probs[0], case["dtype"], case["kind"]
    st = dict(case=case, seed=seed + 7)
    if kind == "batch":
        st["batch"] = P.Batch(probs, dtype)
        st["psi"] = st["batch"].empty()
        for i, q in enumerate(probs):
            st["batch"].view(st["psi"], i).copy_(_states(q, dtype, seed + 11 * i)[0])
        return st
    if kind == "gradient":
        phi0, chi = _states(p, dtype, seed, 2)
        th1, th2 = _thetas(case, seed)
        st.update(base=p, phi0=_padded(p, phi0), chi=_padded(p, chi),
                  theta=(th1.requires_grad_(), th2.requires_grad_()))
        return st
    st["ctx"] = P.Context(p, dtype)
    if kind == "observables":
        psi, chi = _states(p, dtype, seed, 2)
        st["chi"] = _padded(p, chi)
    else:
        psi = _states(p, dtype, seed)[0]
    st["psi"] = _padded(p, psi)
    if kind == "density":
        st["x"] = _points(case, seed)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind in ("step", "twisted"):
        st["ctx"].step(st["psi"], case["steps"], case["tau"], case["scheme"], seed=st["seed"])
        return st["psi"]
    if kind == "batch":
        st["batch"].step(st["psi"], case["steps"], case["tau"], case["scheme"], seed=st["seed"])
        return st["psi"]
    if kind == "gradient":
        loss = overlap_loss(*st["theta"], st["base"], st["phi0"], st["chi"], case["tau"], case["steps"], "strang",
                            case["dtype"])
        g1, g2 = torch.autograd.grad(loss, st["theta"])
        return [loss.detach(), g1, g2]
    if kind == "density":
        return st["ctx"].density(st["psi"], st["x"])
    o = st["ctx"].observables(st["psi"], st["chi"])
    return [o["norm"], o["ekin"], o["epot1"], o["epot2"], o["energy"], o["kmean"][0], o["overlap"].real,
            o["overlap"].imag]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind, es = case["kind"], 8 if case["dtype"] == "c64" else 16
    if kind == "twisted":
        dof = case["q"] ** 4
        # two 2D transforms of q x q points per factor, the potential and the kinetic product
        per = 2 * 5 * 2 * math.log2(case["q"]) + 12
    elif kind == "batch":
        dof = sum(p.M1 * p.M2 for p in _problems(case, 0))
    elif kind == "gradient":
        dof = (2 * case["n"] + 1) ** 2
    else:
        dof = (2 * case["n1"] + 1) * (2 * case["n2"] + 1)
    if kind in ("step", "batch"):
        # a five-point complex kernel and a complex phase per factor
        per = 46
    if kind in ("step", "twisted", "batch"):
        factors = 3 if case["scheme"].startswith("strang") and case["scheme"] != "strang_kp" else 2
        part = 1 / 8 if case["scheme"].endswith("_stoch") else 1
        return {"bytes": 2 * es * dof, "flops": int(dof * case["steps"] * factors * per * part)}
    if kind == "gradient":
        # forward: 2 h + 1 taps and a phase per factor; reverse: the same on two states
        # and the gradient's products
        return {"bytes": 2 * es * dof, "flops": dof * case["steps"] * 3 * 3 * (8 * (2 * case["harmonics"] + 1) + 6)}
    if kind == "density":
        return {"bytes": es * dof + 24 * case["points"], "flops": 8 * dof * case["points"]}
    return {"bytes": 2 * es * dof, "flops": dof * 46}


# ------------------------------------------------------------------ the same in plain 64-bit torch
def _grid_potential(h, c, q):
    d = len(q)
    v = np.zeros(q[::-1], dtype=np.complex128)
    for hh, cc in zip(np.asarray(h), c):
        ph = np.exp(2j * math.pi * ((hh[0] * np.arange(q[0])) % q[0]) / q[0])
        if d > 1:
            ph = np.exp(2j * math.pi * ((hh[1] * np.arange(q[1])) % q[1]) / q[1])[:, None] * ph[None, :]
        v += cc * ph
    return torch.from_numpy(v.real.copy()).cuda()


def _potential_factor(x, p, layer, s, v):
    """exp(-i s v_j) on layer j's grid, every slice (x: (M2, M1))."""
    T = torch.exp(-1j * s * v)
    if p.d == 1:
        dim = 1 if layer == 1 else 0
        return torch.fft.fft(torch.fft.ifft(x, dim=dim) * (T if layer == 1 else T[:, None]), dim=dim)
    y = x.reshape(p.q2[1], p.q2[0], p.q1[1], p.q1[0])
    dims = (2, 3) if layer == 1 else (0, 1)
    T = T if layer == 1 else T[:, :, None, None]
    return torch.fft.fftn(torch.fft.ifftn(y, dim=dims) * T, dim=dims).reshape(x.shape)


def _factors(scheme, t):
    if scheme.startswith("lie"):
        return [("K", t), (1, t), (2, t)]
    if scheme == "strang_kp":
        return [("K", t / 2), (1, t), (2, t), ("K", t / 2)]
    out = []
    for layer, s in ((1, t / 2), (2, t), (1, t / 2)):
        out += [("K", s / 4), (layer, s), ("K", s / 4)]
    return out


def _sample(S, count, seed, g):
    """``count`` of S slices: partial Fisher-Yates shuffle driven by SplitMix64."""
    state = (seed ^ (g * 0xD1B54A32D192ED03)) & MASK64
    perm = list(range(S))
    for i in range(count):
        state = (state + 0x9E3779B97F4A7C15) & MASK64
        z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & MASK64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & MASK64
        j = i + (z ^ (z >> 31)) % (S - i)
        perm[i], perm[j] = perm[j], perm[i]
    return torch.tensor(sorted(perm[:count]), device="cuda")


def _evolve(p, phi, case, seed=0, v=None):
    x = phi.to(torch.complex128)
    scheme = case.get("scheme", "strang")
    v1, v2 = v or (_grid_potential(p.v1_h, p.v1_c, p.q1), _grid_potential(p.v2_h, p.v2_c, p.q2))
    kin = _kinetic(p)
    factors = _factors(scheme, case["tau"])
    phases = {s: torch.exp(-1j * s * kin) for kind, s in factors if kind == "K"}
    g = 0
    for _ in range(case["steps"]):
        for kind, s in factors:
            if kind == "K":
                x = x * phases[s]
                continue
            vj = v1 if kind == 1 else v2
            if scheme.endswith("_stoch"):
                S = p.M2 if kind == 1 else p.M1
                m = max(1, S // 8)
                rows = _sample(S, m, seed, g)
                g += 1
                x = x.clone()
                if kind == 1:
                    x[rows] = _potential_factor(x[rows], p, 1, s * S / m, vj)
                else:
                    x[:, rows] = _potential_factor(x[:, rows], p, 2, s * S / m, vj)
            else:
                x = _potential_factor(x, p, kind, s, vj)
    return x


def exact(case, seed):
    probs = _problems(case, seed)
    p, dtype, kind = probs[0], case["dtype"], case["kind"]
    if kind in ("step", "twisted"):
        return _padded(p, _evolve(p, _states(p, dtype, seed)[0], case, seed + 7))
    if kind == "batch":
        parts = []
        for i, q in enumerate(probs):
            z = _evolve(q, _states(q, dtype, seed + 11 * i)[0], case, seed + 7 + i)
            flat = _padded(q, z).reshape(-1)
            parts.append(torch.nn.functional.pad(flat, (0, -flat.numel() % 32)))
        return torch.cat(parts)
    if kind == "gradient":
        phi0, chi = (z.to(torch.complex128) for z in _states(p, dtype, seed, 2))
        theta = [t.cuda().requires_grad_() for t in _thetas(case, seed)]
        v = []
        for t, q in zip(theta, (p.q1[0], p.q2[0])):
            grid = torch.arange(q, device="cuda", dtype=torch.float64)
            v.append(sum(t[h - 1] * torch.cos(2 * math.pi * torch.remainder(h * grid, q) / q)
                         for h in range(1, len(t) + 1)))
        loss = torch.sum(chi.conj() * _evolve(p, phi0, case, v=v)).abs() ** 2
        g1, g2 = torch.autograd.grad(loss, theta)
        return [loss.detach().cpu(), g1.cpu(), g2.cpu()]
    if kind == "density":
        phi = _states(p, dtype, seed)[0].to(torch.complex128)
        x = torch.from_numpy(_points(case, seed)).cuda()
        m = torch.arange(p.q1[0], device="cuda") + p.lo1[0]
        n = torch.arange(p.q2[0], device="cuda") + p.lo2[0]
        e1 = torch.exp(1j * (x * p.B1[0, 0])[:, None] * m)
        e2 = torch.exp(1j * (x * p.B2[0, 0])[:, None] * n)
        return ((e1 @ phi.T) * e2).sum(1).cpu().numpy()
    psi, chi = (z.to(torch.complex128) for z in _states(p, dtype, seed, 2))
    k = _k(p)[0]
    a2 = psi.real ** 2 + psi.imag ** 2
    pot = []
    for layer, (h, c, q) in ((1, (p.v1_h, p.v1_c, p.q1)), (2, (p.v2_h, p.v2_c, p.q2))):
        y = torch.fft.ifft(psi, dim=2 - layer, norm="ortho")
        v = _grid_potential(h, c, q)
        pot.append(((y.real ** 2 + y.imag ** 2) * (v if layer == 1 else v[:, None])).sum())
    ekin, ovl = (0.5 * k * k * a2).sum(), (chi.conj() * psi).sum()
    return [float(t) for t in (a2.sum(), ekin, pot[0], pot[1], ekin + pot[0] + pot[1], (k * a2).sum(), ovl.real,
                               ovl.imag)]
