"""The work that is timed for this library: lattice runs, an ensemble, a gradient and spectra,
each through the package's public calls, at the sizes of the workloads in `bench.py` and of the
tests, and at sizes in between.

A lattice case is what a run's inner loop does between two rows of its output: advance the lattice
by some steps of the integrator, then read the volume averages (`step`, `energies`).  The state lives in
two torch tensors bound with `bind_buffers`, so the evolved fields are the caller's own memory.
Values are what the runs meet: homogeneous fields of order one with small vacuum-shaped fluctuations,
link variables near the identity, and momenta that satisfy the Gauss laws.
"""
import ctypes
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_2102_01031_gb300 as P
from paper_2102_01031_gb300.autograd import RunSpec, evolved_objective

MODELS = {"lphi4": P.MODEL_LPHI4, "lphi4_chi": P.MODEL_LPHI4_CHI, "u1": P.MODEL_U1_HIGGS,
          "su2u1": P.MODEL_SU2U1_HIGGS, "lphi4su2u1": P.MODEL_LPHI4_SU2U1}
ARRAYS = {"lphi4": 2, "lphi4_chi": 4, "u1": 10, "su2u1": 35, "lphi4su2u1": 41}
INTEGRATORS = {"LF": P.LF, "VV2": P.VV2, "VV4": P.VV4, "VV6": P.VV6}
STAGES = {"LF": 1, "VV2": 1, "VV4": 3, "VV6": 9}
EXPANSIONS = {"off": P.EXP_OFF, "self": P.EXP_SELF, "fixed": P.EXP_FIXED}
DTYPES = {"fp32": torch.float32, "fp64": torch.float64}
# operations per site and pass, counted from the lattice equations (7-point Laplacians and potential
# terms; for the gauge models the covariant hops, plaquettes and staples)
SITE_FLOPS = {"lphi4": 25, "lphi4_chi": 50, "u1": 400, "su2u1": 1900, "lphi4su2u1": 2150}
SIZES = [8 * 2 ** i * 3 ** j for i in range(7) for j in range(4) if 8 * 2 ** i * 3 ** j <= 512]


def listed():
    return [
        # the single-field lambda phi^4 run on a small box in double precision: every pass is short,
        # so latency between passes is what a user waits for
        _evolve("phi4_32_fp64", "lphi4", 32, "fp64", "VV2", "self", 50),
        # the two-field model on the box of a parameter scan
        _evolve("two_field_64_fp32", "lphi4_chi", 64, "fp32", "VV4", "self", 20),
        # the two-field preheating run at its usual size, fields stored in single precision
        _evolve("two_field_256_fp32", "lphi4_chi", 256, "fp32", "VV4", "self", 10),
        # the same at the largest lattice the library takes
        _evolve("two_field_512_fp32", "lphi4_chi", 512, "fp32", "VV4", "self", 4),
        # the same in double precision, at a size that is no power of two
        _evolve("two_field_216_fp64", "lphi4_chi", 216, "fp64", "VV4", "self", 5),
        # the U(1) Abelian-Higgs run in a static background
        _evolve("u1_256_fp32", "u1", 256, "fp32", "LF", "off", 20),
        # the U(1) model with the scale factor evolved along, at a size that is no power of two
        _evolve("u1_144_fp32_self", "u1", 144, "fp32", "VV2", "self", 20),
        # the SU(2) x U(1) doublet in a static background
        _evolve("su2u1_256_fp32", "su2u1", 256, "fp32", "LF", "off", 10),
        # the manual's lphi4SU2U1 example in its expanding background
        _evolve("lphi4su2u1_192_fp32_self", "lphi4su2u1", 192, "fp32", "VV2", "self", 5),
        # an ensemble of independent seeds of the two-field model at mixed sizes
        {"name": "ensemble_64_fp32", "kind": "ensemble", "sizes": "32,64,96,128", "each": 16, "precision": "fp32",
         "integrator": "VV4", "expansion": "self", "alpha": 1.0, "steps": 10},
        # the gradient of the final chi energy fraction, as an optimisation over initial states takes it
        {"name": "gradient_128_fp32", "kind": "gradient", "N": 128, "precision": "fp32", "integrator": "VV4",
         "expansion": "self", "alpha": 1.0, "steps": 60, "every": 30},
        # the power spectra of both fields and both momenta at an output time
        {"name": "spectra_256_fp32", "kind": "spectra", "N": 256, "precision": "fp32", "bin": 1.0},
    ]


def _evolve(name, model, N, precision, integrator, expansion, steps, alpha=1.0):
    return {"name": name, "kind": "evolve", "model": model, "N": N, "precision": precision, "integrator": integrator,
            "expansion": expansion, "alpha": alpha, "steps": steps}


def draw(rng):
    """One more case: the kinds in about the proportions of the listed ones, sizes spread over the
    admissible lattice sizes in their logarithm, each bounded so that it stays below the largest listed case."""
    def size(lo, hi, multiple=8):
        x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return min((n for n in SIZES if lo <= n <= hi and n % multiple == 0), key=lambda n: abs(math.log(n / x)))

    kind = rng.choice(["scalar"] * 5 + ["u1"] * 2 + ["doublet"] * 2 + ["ensemble", "gradient", "spectra"])
    expansion = rng.choice(["self", "self", "off", "fixed"])
    if kind == "scalar":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        N = size(16, 384 if precision == "fp32" else 216)
        integ = rng.choice(["LF", "VV2", "VV4", "VV4", "VV6"])
        most = 30 if N < 200 else 15 if precision == "fp32" else 9
        steps = max(1, rng.randint(most // 3, most) // STAGES[integ])
        return _drawn(_evolve("", rng.choice(["lphi4", "lphi4_chi", "lphi4_chi"]), N, precision, integ, expansion,
                              steps, rng.choice([1.0, 1.0, 0.0])))
    if kind == "u1":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        N = size(16, 256 if precision == "fp32" else 96)
        return _drawn(_evolve("", "u1", N, precision, rng.choice(["LF", "VV2"]), expansion, rng.randint(5, 20)))
    if kind == "doublet":
        precision = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        N = size(16, 192 if precision == "fp32" else 64, 16)
        return _drawn(_evolve("", rng.choice(["su2u1", "lphi4su2u1"]), N, precision, rng.choice(["LF", "VV2"]),
                              expansion, rng.randint(3, 6)))
    if kind == "ensemble":
        sizes = sorted({size(16, 128) for _ in range(rng.randint(2, 4))})
        return {"kind": "ensemble", "sizes": ",".join(map(str, sizes)), "each": rng.randint(2, 12), "precision": "fp32",
                "integrator": rng.choice(["VV2", "VV4"]), "expansion": expansion, "alpha": 1.0,
                "steps": rng.randint(4, 10)}
    if kind == "gradient":
        steps = rng.randint(10, 60)
        return {"kind": "gradient", "N": size(16, 128), "precision": rng.choice(["fp32", "fp32", "fp64"]),
                "integrator": rng.choice(["VV2", "VV4"]), "expansion": expansion, "alpha": 1.0, "steps": steps,
                "every": rng.randint(5, steps)}
    return {"kind": "spectra", "N": size(24, 256), "precision": rng.choice(["fp32", "fp64"]),
            "bin": rng.choice([1.0, 1.0, 0.5, 2.0])}


def _drawn(case):
    del case["name"]
    return case


# ---- inputs -----------------------------------------------------------------------------------------


def _params(case):
    """Keywords of make_params for a case (the run parameters of the library's workloads)."""
    model = case.get("model", "lphi4_chi")
    kw = dict(dt=0.005 if STAGES[case.get("integrator", "VV2")] > 1 else 0.01,
              integrator=INTEGRATORS[case.get("integrator", "VV2")],
              expansion=EXPANSIONS[case.get("expansion", "self")], fstar_over_mp=0.5,
              precision=P.FP32 if case["precision"] == "fp32" else P.FP64)
    if kw["expansion"] == P.EXP_FIXED:
        kw.update(omega_eos=1.0 / 3.0, H0=0.4)
    if model in ("lphi4", "lphi4_chi"):
        kw.update(q=100.0, phi0=[1.0, 0.0])
    elif model == "u1":
        # a massive field's frequency grows with the scale factor, so the vacuum value is for static backgrounds
        kw.update(lam=1.0, v=1.0 if case["expansion"] == "off" else 0.0, gQ=0.5, fstar_over_omegastar=1.0,
                  phi0=[1.0, 1.0])
    else:
        kw.update(lam=1.0, v=0.5 if model == "su2u1" and case["expansion"] == "off" else 0.0, gQ=0.6, gQB=0.8,
                  fstar_over_omegastar=1.3, phi0=[0.5] * 4, dphi0=[0.1] * 4)
        if model == "lphi4su2u1":
            kw.update(qG=1.5, qH=0.8, Qc=0.7)
    return kw


def _kIR(N):
    """The box that keeps the lattice spacing of 256^3 at kIR = 0.1."""
    return 25.6 / N


def _waves(gen, N, rms):
    """A random field with the vacuum's spectrum (amplitude ~ k^-1/2) and the given rms."""
    w = torch.fft.rfftn(torch.randn((N, N, N), generator=gen, device="cuda", dtype=torch.float64))
    k = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, : N // 2 + 1] ** 2
    k2[0, 0, 0] = 1.0
    w *= k2 ** -0.25
    w[0, 0, 0] = 0.0
    f = torch.fft.irfftn(w, s=(N, N, N))
    return f * (rms / f.square().mean().sqrt())


def _shift(f, i, n):
    """f at the site n steps along direction i (0 = x, the fastest index)."""
    return torch.roll(f, -n, -1 - i)


def _state(model, N, dtype, seed):
    """The arrays of one lattice in the library's storage order, [array][z][y][x]."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    out = torch.empty((ARRAYS[model], N, N, N), dtype=dtype, device="cuda")
    if model in ("lphi4", "lphi4_chi"):
        for f in range(ARRAYS[model] // 2):
            out[2 * f] = (1.0 if f == 0 else 0.0) + _waves(gen, N, 0.02)
            out[2 * f + 1] = _waves(gen, N, 0.05)
        return out
    nc = 2 if model == "u1" else 4
    phi0, dphi = (1.0, 0.0) if model == "u1" else (0.5, 0.1)
    rate = dphi / phi0 + _waves(gen, N, 0.1)  # momenta along the fields carry no charge
    phi = [phi0 + _waves(gen, N, 0.03) for _ in range(nc)]
    A = [_waves(gen, N, 0.05) for _ in range(3)]
    N3 = [_waves(gen, N, 0.05) for _ in range(3)]  # link momenta as a curl: no divergence, as the Gauss law asks
    E = []
    for i in range(3):
        j, k = (i + 1) % 3, (i + 2) % 3
        E.append((N3[k] - _shift(N3[k], j, -1)) - (N3[j] - _shift(N3[j], k, -1)))
    if model == "u1":
        for c in range(2):
            out[2 * c], out[2 * c + 1] = phi[c], rate * phi[c]
        for i in range(3):
            out[4 + 2 * i], out[5 + 2 * i] = A[i], E[i]
        return out
    for c in range(4):
        out[c], out[4 + c] = phi[c], rate * phi[c]
    for i in range(3):
        out[8 + i], out[11 + i] = A[i], E[i]
        u = torch.stack([_waves(gen, N, 0.05) for _ in range(4)])
        u[0] += 1.0
        out[14 + 4 * i:18 + 4 * i] = u / u.square().sum(0).sqrt()
        out[26 + 3 * i:29 + 3 * i] = 0.0
    if model == "lphi4su2u1":
        out[35], out[36] = _waves(gen, N, 0.03), _waves(gen, N, 0.05)
        out[37], out[38] = _waves(gen, N, 0.03), _waves(gen, N, 0.03)
        out[39], out[40] = rate * out[37], rate * out[38]
    return out


def _members(case):
    return [int(n) for n in case["sizes"].split(",") for _ in range(case["each"])]


def prepare(case, seed):
    kw = dict(_params(case), stream=P.torch_stream())
    dtype = DTYPES[case["precision"]]
    kind = case["kind"]
    if kind == "gradient":
        N = case["N"]
        kw.pop("stream")
        q = torch.tensor(kw.pop("q"), dtype=torch.float64, device="cuda", requires_grad=True)
        state = _state("lphi4_chi", N, dtype, seed).view(2, 2, N, N, N).requires_grad_()
        scale = torch.tensor([1.0, _b0(case)], dtype=torch.float64, requires_grad=True)
        spec = RunSpec.make(P.MODEL_LPHI4_CHI, N, _kIR(N), case["alpha"], 1, case["steps"], ckpt_every=case["every"],
                            **kw)
        return {"case": case, "q": q, "state": state, "scale": scale, "spec": spec}
    if kind == "ensemble":
        Ns = _members(case)
        lat = P.Ensemble(P.MODEL_LPHI4_CHI, Ns, [_kIR(n) for n in Ns], case["alpha"], list(range(1, len(Ns) + 1)),
                         P.make_params(**kw))
        total = 4 * sum(n ** 3 for n in Ns)
        bufs = [torch.empty(total, dtype=dtype, device="cuda") for _ in range(2)]
        at = 0
        for l, n in enumerate(Ns):
            size = 4 * n ** 3
            lat.bind_buffers(bufs[0][at:at + size], bufs[1][at:at + size], lat=l)
            at += size
            arrays = _state("lphi4_chi", n, dtype, seed * 1000003 + l).double()
            for a in range(4):
                ptr = ctypes.cast(ctypes.c_void_p(arrays[a].data_ptr()), ctypes.POINTER(ctypes.c_double))
                if lat.L.cl_lattice_set_state(lat.h, l, a // 2, a % 2, ptr) != P.CL_OK:
                    raise RuntimeError("cl_lattice_set_state")
        return {"case": case, "lat": lat, "bufs": bufs}
    model, N = case.get("model", "lphi4_chi"), case["N"]
    lat = P.Lattice(MODELS[model], N, _kIR(N), case.get("alpha", 1.0), 1, P.make_params(**kw))
    state = _state(model, N, dtype, seed)
    if kind == "spectra":
        lat.upload(state.data_ptr(), state.numel() * state.element_size())
        return {"case": case, "lat": lat}
    bufs = [torch.empty_like(state) for _ in range(2)]
    lat.bind_buffers(*bufs)
    lat.upload(state.data_ptr(), state.numel() * state.element_size())
    return {"case": case, "lat": lat, "bufs": bufs}


# ---- one pass ---------------------------------------------------------------------------------------


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gradient":
        q, x, scale = state["q"], state["state"], state["scale"]
        J = evolved_objective(q, x, state["spec"], scale=scale)
        gq, gx, gs = torch.autograd.grad(J, [q, x, scale])
        # of a run in single precision, J and the two small gradients carry that much
        d = DTYPES[case["precision"]]
        return {"J": J.detach().to(d), "q": gq.to(d), "state": gx, "scale": gs.to(d)}
    lat = state["lat"]
    if kind == "spectra":
        return [lat.spectrum(f, w, case["bin"]) for f in range(2) for w in range(2)]
    lat.step(case["steps"])
    if kind == "ensemble":
        e = [lat.energies(l) for l in range(lat.size())]
        return {"state": state["bufs"][lat.state_buffer()], "averages": _averages(case, *e),
                "background": _background(case, *e)}
    e = lat.energies()
    out = _named(case["model"], state["bufs"][lat.state_buffer()])
    out.update(averages=_averages(case, e), background=_background(case, e))
    return out


def _named(model, x):
    """The arrays of a state by what they are."""
    if model in ("lphi4", "lphi4_chi"):
        return {"phi": x[0::2], "pi": x[1::2]}
    if model == "u1":
        return {"phi": x[0:4:2], "pi": x[1:4:2], "A": x[4::2], "pi_A": x[5::2]}
    out = {"phi": x[0:4], "pi": x[4:8], "A": x[8:11], "pi_A": x[11:14], "U": x[14:26], "pi_B": x[26:35]}
    if model == "lphi4su2u1":
        out.update(phi_s=x[35:36], pi_s=x[36:37], vphi=x[37:39], pi_vphi=x[39:41])
    return out


def _averages(case, *es):
    """Volume averages, at the accuracy of the storage type that the averaged fields have."""
    keys = ("EK", "EG", "EV", "mean_phi", "mean_phi2", "mean_pi", "mean_pi2")
    rows = [[x for k in keys for x in e[k]] + [e["EKA"], e["EGA"], e["EKB"], e["EGB"], e["rho"]] for e in es]
    return np.array(rows, dtype=np.float32 if case["precision"] == "fp32" else np.float64)


def _background(case, *es):
    return np.array([[e["eta"], e["a"], e["b"]] for e in es],
                    dtype=np.float32 if case["precision"] == "fp32" else np.float64)


# ---- what a pass cannot do without ------------------------------------------------------------------


def work(case):
    """A pass of the integrator kicks every momentum and drifts every field, and with an evolved scale
    factor the next one waits for this one's volume averages: each reads and writes the state once.
    The averages at the end close the stream with one more pass."""
    esz = 4 if case["precision"] == "fp32" else 8
    if case["kind"] == "spectra":
        V = case["N"] ** 3
        return {"bytes": 4 * V * esz, "flops": 4 * 2.5 * V * math.log2(V)}
    passes = case["steps"] * STAGES[case["integrator"]]
    if case["kind"] == "gradient":
        # forward once, then back: the state and its adjoint are read and written by each reversed pass
        V = case["N"] ** 3
        return {"bytes": passes * 3 * 2 * 4 * V * esz, "flops": passes * 3 * SITE_FLOPS["lphi4_chi"] * V}
    model = case.get("model", "lphi4_chi")
    V = sum(n ** 3 for n in _members(case)) if case["kind"] == "ensemble" else case["N"] ** 3
    return {"bytes": (passes + 1) * 2 * ARRAYS[model] * V * esz, "flops": (passes + 1) * SITE_FLOPS[model] * V}


# ---- the same in 64 bits, from the lattice equations ------------------------------------------------


def _b0(case):
    """a' at the start, from the Hubble law with the homogeneous values (a = 1)."""
    if case.get("expansion", "self") == "off":
        return 0.0
    kw = _params(case)
    if case["expansion"] == "fixed":
        return kw["H0"]
    model = case.get("model", "lphi4_chi")
    phi0, dphi0 = kw["phi0"], kw.get("dphi0", [0.0] * 4)
    if model in ("lphi4", "lphi4_chi"):
        V = 0.25 * phi0[0] ** 4
    else:
        V = kw["lam"] * (0.5 * sum(x * x for x in phi0) - kw["v"] ** 2) ** 2
    rho = 0.5 * sum(x * x for x in dphi0) + V
    return math.sqrt(kw["fstar_over_mp"] ** 2 / 3.0 * rho)


def _drifts(order, h):
    if order <= 2:
        return [h]
    z = 1.0 / (2.0 - 2.0 ** (1.0 / (order - 1)))
    return _drifts(order - 2, z * h) + _drifts(order - 2, (1.0 - 2.0 * z) * h) + _drifts(order - 2, z * h)


def _lap(f):
    return sum(_shift(f, i, 1) + _shift(f, i, -1) for i in range(3)) - 6.0 * f


def _grad2(f):
    return sum((_shift(f, i, 1) - f).square().mean() for i in range(3))


def _qmul(a, b):
    """Product of SU(2) elements u0 - i u.sigma held as their four real components."""
    return torch.stack([a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3],
                        a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2],
                        a[0] * b[2] + a[2] * b[0] + a[3] * b[1] - a[1] * b[3],
                        a[0] * b[3] + a[3] * b[0] + a[1] * b[2] - a[2] * b[1]])


def _dag(a):
    return torch.stack([a[0], -a[1], -a[2], -a[3]])


def _apply(u, psi):
    """(u0 - i u.sigma) psi for a complex doublet."""
    return torch.stack([torch.complex(u[0], -u[3]) * psi[0] + torch.complex(-u[2], -u[1]) * psi[1],
                        torch.complex(u[2], -u[1]) * psi[0] + torch.complex(u[0], u[3]) * psi[1]])


class _Scalars:
    """The two scalar models: V = phi^4/4 + (q/2) phi^2 chi^2."""

    def __init__(self, case, N, q=None):
        kw = _params(case)
        self.dx = 2.0 * math.pi / (N * _kIR(N))
        self.q = kw["q"] if q is None else q

    def force(self, X):
        phi = X["phi"]
        V = [phi[0] ** 3]
        if len(phi) == 2:
            V = [phi[0] ** 3 + self.q * phi[0] * phi[1] ** 2, self.q * phi[0] ** 2 * phi[1]]
        # kernels of the momenta by their power of the scale factor: a^(1+alpha), a^(3+alpha), a^(alpha-1)
        return {"pi": (torch.stack([_lap(f) for f in phi]) / self.dx ** 2, -torch.stack(V), None)}

    def potential(self, X):
        phi = X["phi"]
        EG = [_grad2(f) / (2.0 * self.dx ** 2) for f in phi]
        EV = [0.25 * (phi[0] ** 4).mean()]
        if len(phi) == 2:
            EV.append(0.5 * self.q * (phi[0] * phi[1]).square().mean())
        return EG, EV, 0.0, 0.0

    def kinetic(self, Y):
        return [0.5 * p.square().mean() for p in Y["pi"]], 0.0, 0.0

    def drift(self, X, Y, c, cA):
        return {"phi": X["phi"] + c * Y["pi"]}


class _U1:
    """Abelian-Higgs: compact U(1) links, V = lam (|phi|^2 - v^2)^2, phi = (phi_0 + i phi_1)/sqrt 2."""

    def __init__(self, case, N):
        kw = _params(case)
        self.dx = 2.0 * math.pi / (N * _kIR(N))
        self.g, self.lam, self.v = kw["gQ"], kw["lam"], kw["v"]
        self.f2 = kw["fstar_over_omegastar"] ** 2

    def _angle(self, A, i, j):
        return self.g * self.dx * (A[i] + _shift(A[j], i, 1) - _shift(A[i], j, 1) - A[j])

    def _curl(self, A):
        s = {(i, j): torch.sin(self._angle(A, i, j)) for i in range(3) for j in range(i + 1, 3)}
        out = []
        for i in range(3):
            c = 0.0
            for j in range(3):
                if j != i:
                    t = s[min(i, j), max(i, j)] if i < j else -s[j, i]
                    c = c + t - _shift(t, j, -1)
            out.append(-c / (self.g * self.dx ** 3))
        return torch.stack(out)

    def _hops(self, A, z, charge=1.0):
        """V_i z(n+i) for each direction; z: (..., complex)."""
        th = charge * self.g * self.dx
        V = [torch.polar(torch.ones_like(A[i]), -th * A[i]) for i in range(3)]
        fwd = [V[i] * _shift(z, i, 1) for i in range(3)]
        bwd = [_shift(V[i].conj() * z, i, -1) for i in range(3)]
        return fwd, bwd

    def force(self, X):
        z = torch.complex(X["phi"][0], X["phi"][1])
        fwd, bwd = self._hops(X["A"], z)
        D = (sum(fwd) + sum(bwd) - 6.0 * z) / self.dx ** 2
        V = 2.0 * self.lam * (0.5 * X["phi"].square().sum(0) - self.v ** 2) * X["phi"]
        J = torch.stack([self.f2 * self.g / self.dx * (z.conj() * u).imag for u in fwd])
        return {"pi": (torch.stack([D.real, D.imag]), -V, None), "pi_A": (J, None, self._curl(X["A"]))}

    def _magnetic(self, A):
        return sum((2.0 * torch.sin(0.5 * self._angle(A, i, j)).square()).mean()
                   for i in range(3) for j in range(i + 1, 3)) / (self.f2 * (self.g * self.dx ** 2) ** 2)

    def potential(self, X):
        z = torch.complex(X["phi"][0], X["phi"][1])
        fwd, _ = self._hops(X["A"], z)
        EG = sum((u - z).abs().square().mean() for u in fwd) / (2.0 * self.dx ** 2)
        EV = self.lam * (0.5 * X["phi"].square().sum(0) - self.v ** 2).square().mean()
        return [EG], [EV], self._magnetic(X["A"]), 0.0

    def kinetic(self, Y):
        return ([0.5 * Y["pi"].square().sum(0).mean()],
                0.5 * Y["pi_A"].square().sum(0).mean() / self.f2, 0.0)

    def drift(self, X, Y, c, cA):
        return {"phi": X["phi"] + c * Y["pi"], "A": X["A"] + cA * Y["pi_A"]}


class _Doublet(_U1):
    """The SU(2) x U(1) doublet, and with `full` the singlet and the U(1)-charged scalar."""

    def __init__(self, case, N):
        super().__init__(case, N)
        kw = _params(case)
        self.gB, self.full = kw["gQB"], case["model"] == "lphi4su2u1"
        self.qG, self.qH, self.Qc = kw.get("qG", 0.0), kw.get("qH", 0.0), kw.get("Qc", 0.0)

    def _doublet_hops(self, X):
        psi = torch.stack([torch.complex(X["phi"][0], X["phi"][1]), torch.complex(X["phi"][2], X["phi"][3])])
        th = self.g * self.dx
        U = [X["U"][4 * i:4 * i + 4] for i in range(3)]
        V = [torch.polar(torch.ones_like(X["A"][i]), -th * X["A"][i]) for i in range(3)]
        fwd = [V[i] * _apply(U[i], _shift(psi, i, 1)) for i in range(3)]
        bwd = [_shift(V[i].conj() * _apply(_dag(U[i]), psi), i, -1) for i in range(3)]
        return psi, U, fwd, bwd

    def force(self, X):
        psi, U, fwd, bwd = self._doublet_hops(X)
        D = (sum(fwd) + sum(bwd) - 6.0 * psi) / self.dx ** 2
        P2 = 0.5 * X["phi"].square().sum(0)
        g = 2.0 * self.lam * (P2 - self.v ** 2)
        J, K = [], []
        for i in range(3):
            u = fwd[i]
            J.append(self.f2 * self.g / self.dx * (psi.conj() * u).sum(0).imag)
            s = [(psi[0].conj() * u[1] + psi[1].conj() * u[0]).imag,
                 (-1j * psi[0].conj() * u[1] + 1j * psi[1].conj() * u[0]).imag,
                 (psi[0].conj() * u[0] - psi[1].conj() * u[1]).imag]
            K.append(torch.stack(s) * (self.f2 * self.gB / (2.0 * self.dx)))
        B = []
        for i in range(3):
            S = 0.0
            for j in range(3):
                if j != i:
                    Uij = _shift(U[j], i, 1)
                    up = _qmul(_qmul(Uij, _dag(_shift(U[i], j, 1))), _dag(U[j]))
                    lo = _shift(_qmul(_qmul(_dag(Uij), _dag(U[i])), U[j]), j, -1)
                    S = S + up + lo
            B.append(-2.0 * _qmul(U[i], S)[1:] / (self.gB * self.dx ** 3))
        out = {"pi_A": None, "pi_B": (torch.cat(K), None, torch.cat(B))}
        if self.full:
            s, z = X["phi_s"], torch.complex(X["vphi"][0], X["vphi"][1])
            C2 = 0.5 * X["vphi"].square().sum(0)
            g = g + self.qG * s[0].square() + 2.0 * self.qH * C2
            vf, vb = self._hops(X["A"], z, self.Qc)
            Dz = (sum(vf) + sum(vb) - 6.0 * z) / self.dx ** 2
            J = [J[i] + self.f2 * self.Qc * self.g / self.dx * (z.conj() * vf[i]).imag for i in range(3)]
            out["pi_s"] = (_lap(s[0])[None] / self.dx ** 2, -2.0 * self.qG * P2 * s, None)
            out["pi_vphi"] = (torch.stack([Dz.real, Dz.imag]), -2.0 * self.qH * P2 * X["vphi"], None)
        out["pi"] = (torch.stack([D[0].real, D[0].imag, D[1].real, D[1].imag]), -g * X["phi"], None)
        out["pi_A"] = (torch.stack(J), None, self._curl(X["A"]))
        return out

    def potential(self, X):
        psi, U, fwd, _ = self._doublet_hops(X)
        half = 1.0 / (2.0 * self.dx ** 2)
        EG = [sum((u - psi).abs().square().sum(0).mean() for u in fwd) * half]
        P2 = 0.5 * X["phi"].square().sum(0)
        EV = [self.lam * (P2 - self.v ** 2).square().mean()]
        m = 0.0
        for i in range(3):
            for j in range(i + 1, 3):
                p = _qmul(_qmul(U[i], _shift(U[j], i, 1)), _dag(_qmul(U[j], _shift(U[i], j, 1))))
                m = m + 2.0 * (p[1:].square().sum(0) / (1.0 + p[0])).mean()
        EGB = 2.0 * m / (self.f2 * (self.gB * self.dx ** 2) ** 2)
        if self.full:
            s, z = X["phi_s"][0], torch.complex(X["vphi"][0], X["vphi"][1])
            vf, _ = self._hops(X["A"], z, self.Qc)
            EG += [_grad2(s) * half, sum((u - z).abs().square().mean() for u in vf) * half]
            EV += [self.qG * (P2 * s.square()).mean(), self.qH * (P2 * X["vphi"].square().sum(0)).mean()]
        return EG, EV, self._magnetic(X["A"]), EGB

    def kinetic(self, Y):
        EK, EKA, _ = super().kinetic(Y)
        if self.full:
            EK += [0.5 * Y["pi_s"].square().sum(0).mean(), 0.5 * Y["pi_vphi"].square().sum(0).mean()]
        return EK, EKA, 0.5 * Y["pi_B"].square().sum(0).mean() / self.f2

    def drift(self, X, Y, c, cA):
        out = super().drift(X, Y, c, cA)
        U = []
        for i in range(3):
            th = (self.gB * self.dx * cA) * Y["pi_B"][3 * i:3 * i + 3]
            t = th.square().sum(0).sqrt()
            s = 0.5 * torch.sinc(t / (2.0 * math.pi))
            U.append(_qmul(torch.cat([torch.cos(0.5 * t)[None], s * th]), X["U"][4 * i:4 * i + 4]))
        out["U"] = torch.cat(U)
        if self.full:
            out["phi_s"] = X["phi_s"] + c * Y["pi_s"]
            out["vphi"] = X["vphi"] + c * Y["pi_vphi"]
        return out


class _Run:
    """Velocity-Verlet substeps with the scale factor kicked and drifted along; a, b may be tensors."""

    def __init__(self, case, eq):
        kw = _params(case)
        self.eq, self.al, self.fm2 = eq, case["alpha"], kw["fstar_over_mp"] ** 2
        self.mode, self.H = case["expansion"], kw.get("H0", 0.0)
        self.p = 2.0 / (3.0 * (1.0 + kw.get("omega_eos", 0.0)) - 2.0 * self.al)
        self.sub = _drifts(INTEGRATORS[case["integrator"]], kw["dt"])

    def kick(self, Y, F, a, w):
        al, out = self.al, {}
        for k, (f1, f3, fm) in F.items():
            out[k] = Y[k] + w * sum(f * a ** p for f, p in ((f1, 1.0 + al), (f3, 3.0 + al), (fm, al - 1.0))
                                    if f is not None)
        return out

    def energies(self, Y, E, a):
        EK, EKA, EKB = self.eq.kinetic(Y)
        EG, EV, EGA, EGB = E
        return ([e / a ** 6 for e in EK], [e / a ** 2 for e in EG], EV, EKA / a ** 4, EGA / a ** 4, EKB / a ** 4,
                EGB / a ** 4)

    def kick_b(self, Y, E, a, w):
        if self.mode != "self":
            return 0.0
        EK, EG, EV, *gauge = self.energies(Y, E, a)
        al = self.al
        br = (al - 2.0) * sum(EK) + al * sum(EG) + (al - 1.0) * sum(gauge) + (al + 1.0) * sum(EV)
        return w * a ** (2.0 * al + 1.0) / 3.0 * self.fm2 * br

    def step(self, X, Y, eta, a, b):
        F, E = self.eq.force(X), self.eq.potential(X)
        for d in self.sub:
            Y = self.kick(Y, F, a, 0.5 * d)
            b = b + self.kick_b(Y, E, a, 0.5 * d)
            if self.mode == "self":
                a1 = a + d * b
            else:
                a1 = (1.0 + self.H * (eta + d) / self.p) ** self.p if self.mode == "fixed" else a
            mid = 0.5 * (a + a1)
            X = self.eq.drift(X, Y, d * mid ** (self.al - 3.0), d * mid ** (self.al - 1.0))
            a, eta = a1, eta + d
            if self.mode == "fixed":
                b = a * self.H / (1.0 + self.H * eta / self.p)
            F, E = self.eq.force(X), self.eq.potential(X)
            b = b + self.kick_b(Y, E, a, 0.5 * d)
            Y = self.kick(Y, F, a, 0.5 * d)
        return X, Y, eta, a, b

    def observed(self, X, Y, eta, a, b):
        """What _averages and _background return."""
        EK, EG, EV, EKA, EGA, EKB, EGB = self.energies(Y, self.eq.potential(X), a)
        pad = lambda v: [float(x) for x in v] + [0.0] * (4 - len(v))  # noqa: E731
        mean = [pad([m(f).mean() for f in z]) for z in (X["phi"], Y["pi"]) for m in (lambda t: t, torch.square)]
        rho = sum(EK) + sum(EG) + sum(EV) + EKA + EGA + EKB + EGB
        row = pad(EK) + pad(EG) + pad(EV) + sum(mean, []) + [float(x) for x in (EKA, EGA, EKB, EGB, rho)]
        return np.array([row]), np.array([[float(eta), float(a), float(b)]])


def _split(named):
    return ({k: v for k, v in named.items() if not k.startswith("pi")},
            {k: v for k, v in named.items() if k.startswith("pi")})


def _exact_evolve(case, model, x, N):
    eq = {"u1": _U1, "su2u1": _Doublet, "lphi4su2u1": _Doublet}.get(model, _Scalars)(case, N)
    r = _Run(case, eq)
    X, Y = _split(_named(model, x))
    eta, a, b = 0.0, 1.0, _b0(case)
    for _ in range(case["steps"]):
        X, Y, eta, a, b = r.step(X, Y, eta, a, b)
    avg, bg = r.observed(X, Y, eta, a, b)
    return X, Y, avg, bg


def _exact_gradient(case, x):
    N = case["N"]
    q = torch.tensor(_params(case)["q"], dtype=torch.float64, device="cuda", requires_grad=True)
    scale = torch.tensor([1.0, _b0(case)], dtype=torch.float64, device="cuda", requires_grad=True)
    x = x.requires_grad_()
    zero = torch.zeros((), dtype=torch.float64, device="cuda")

    def one(phi, pi, eta, a, b, q):
        r = _Run(case, _Scalars(case, N, q))
        X, Y, eta, a, b = r.step({"phi": phi}, {"pi": pi}, eta, a, b)
        return X["phi"], Y["pi"], zero + eta, zero + a, zero + b

    phi, pi, eta, a, b = x[0::2], x[1::2], zero, scale[0], scale[1]
    for _ in range(case["steps"]):
        phi, pi, eta, a, b = checkpoint(one, phi, pi, eta, a, b, q, use_reentrant=False)
    eq = _Scalars(case, N, q)
    EK, EG, EV, *_ = _Run(case, eq).energies({"pi": pi}, eq.potential({"phi": phi}), a)
    J = (EK[1] + EG[1]) / (sum(EK) + sum(EG) + sum(EV))
    gq, gx, gs = torch.autograd.grad(J, [q, x, scale], allow_unused=True)
    if case["expansion"] != "self":  # the background is given: a and b at the start are no variables
        gs = torch.zeros(2, dtype=torch.float64, device="cuda")
    return {"J": J.detach(), "q": gq, "state": gx.view(2, 2, N, N, N), "scale": gs}


def _exact_spectrum(u, N, dk):
    k = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
    n = (k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2).sqrt().view(-1)[1:]
    nb = int(math.floor(math.sqrt(3.0) * (N // 2) / dk)) + 1
    b = (n / dk).floor().long().clamp_(max=nb - 1)
    power = torch.fft.fftn(u).abs().square().view(-1)[1:]
    add = lambda w: torch.zeros(nb, dtype=torch.float64, device="cuda").index_add_(0, b, w)  # noqa: E731
    count, sn, sp = add(torch.ones_like(n)), add(n), add(power)
    kIR = _kIR(N)
    dx = 2.0 * math.pi / (N * kIR)
    nbar = sn / count.clamp(min=1.0)
    kb = kIR * nbar
    delta = kb ** 3 / (2.0 * math.pi ** 2) * (dx / N) ** 3 * sp / (4.0 * math.pi * nbar.clamp(min=0.1) ** 2)
    return kb, torch.where(count > 0, delta, torch.zeros_like(delta)), None


def exact(case, seed):
    dtype = DTYPES[case["precision"]]
    kind = case["kind"]
    if kind == "ensemble":
        state, avg, bg = [], [], []
        for l, n in enumerate(_members(case)):
            x = _state("lphi4_chi", n, dtype, seed * 1000003 + l).double()
            X, Y, e, g = _exact_evolve(case, "lphi4_chi", x, n)
            state.append(torch.stack([X["phi"], Y["pi"]], 1).reshape(-1))
            avg.append(e)
            bg.append(g)
        return {"state": torch.cat(state), "averages": np.concatenate(avg), "background": np.concatenate(bg)}
    N = case["N"]
    x = _state(case.get("model", "lphi4_chi"), N, dtype, seed).double()
    if kind == "gradient":
        return _exact_gradient(case, x)
    if kind == "spectra":
        return [_exact_spectrum(x[a], N, case["bin"]) for a in range(4)]
    X, Y, avg, bg = _exact_evolve(case, case["model"], x, N)
    return {**X, **Y, "averages": avg, "background": bg}
