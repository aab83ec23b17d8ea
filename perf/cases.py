"""The work that users of this framework have it do, as measurable cases.

Every case goes through the public entry points (``binding``, ``Solver``,
``BatchSolver``, ``TimeStepper``, ``DampingNet``), on inputs made on the GPU
from a seed.  Most are single calls of the damped-gradient iteration; the
whole calls are an iteration of one box, an iteration of a batch of boxes and
a time-dependent step.

Eigenvectors have no phase (and none at all inside a degenerate level), so
the cases that end in a Rayleigh-Ritz step return what does not depend on the
choice: the levels, the densities of the new states, and the mean field and
energy they give.  Where the method fixes the phases (the paper's combined
form) the matrices themselves are returned.
"""
from __future__ import annotations

import math

import torch

from paper_1610_07522_gb300 import binding as B
from paper_1610_07522_gb300 import inputs as IN
from paper_1610_07522_gb300.batched import BatchSolver
from paper_1610_07522_gb300.learned import DampingNet, init_params
from paper_1610_07522_gb300.solver import Solver
from paper_1610_07522_gb300.td import HBARC, TimeStepper

DEV = "cuda:0"
P = IN.SLY4
PREC = {"f64": B.SKY_F64, "f32": B.SKY_F32, "bf16x3": B.SKY_F32_BF16X3, "bf16x6": B.SKY_F32_BF16X6}
X0, E0 = 0.45, 100.0          # step size and damping energy of every workload
AXES = (8, 12, 16, 20, 24, 32)
DT = 0.1                      # fm/c, the time step of the benchmark's evolution


def _case(kind, name=None, n=(16, 16, 16), states=0, protons=0, form="f64", **more):
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "states": states, "protons": protons,
         "form": form, **more}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # h psi of one species with its energies, once per iteration: the small
        # box that convergence studies run thousands of times (launch-bound) ...
        _case("apply_h", "h_f64_16cubed_16", (16, 16, 16), 16, totals=True),
        # ... and the neutrons of the benchmark's 24^3 box in the paper's precision
        _case("apply_h", "h_f64_24cubed_280", (24, 24, 24), 280, totals=True),
        # h phi (no energies asked for) of the 32^3 precision workload's neutrons
        _case("apply_h", "h_f32_32cubed_700", (32, 32, 32), 700, form="f32", totals=False),
        # the damped step: the 24^3 neutrons in FP64, the plain step ...
        _case("damped_step", "step_f64_24cubed_280", (24, 24, 24), 280, weight=False),
        # ... and the 32^3 protons in FP32 with a per-voxel weight (learned form)
        _case("damped_step", "step_f32_32cubed_300_weight", (32, 32, 32), 300, form="f32", weight=True),
        # S = <phi|phi> and H = <phi|h phi> of the 24^3 neutrons
        _case("matrices", "matrices_f64_24cubed_280", (24, 24, 24), 280),
        # the recombination of the 32^3 neutrons in the split-BF16 form
        _case("rotate", "rotate_bf16x3_32cubed_700", (32, 32, 32), 700, form="bf16x3"),
        # Loewdin factors and diagonalisation of both species of the 32^3 workload,
        # in the paper's combined form (its phases are fixed)
        _case("eigen", "eigen_700_300", (8, 8, 8), 700, 300),
        # one whole iteration of the benchmark's box, replayed as a CUDA graph
        _case("iteration", "iteration_f64_24cubed_280_120", (24, 24, 24), 280, 120, coulomb=True),
        # one iteration of six uneven twisted boxes (16^3, 20^3, 24^3) together
        _case("batch", "batch_f64_6_boxes", (16, 16, 16), boxes=6),
        # one predictor-corrector time step of a 20^3 box in FP32
        _case("td_step", "td_f32_20cubed_168_72", (20, 20, 20), 168, 72, form="f32"),
        # one training step of the damping network: two samples (species) of a 24^3 box
        _case("train", "train_24cubed", (24, 24, 24)),
    ]


def draw(rng):
    """A case of the same ranges: any call, any box, any number of states."""
    kind = rng.choice(("apply_h", "apply_h", "damped_step", "damped_step", "matrices", "rotate",
                       "eigen", "iteration", "td_step", "train"))
    n = tuple(rng.choice(AXES) for _ in range(3))
    G = n[0] * n[1] * n[2]
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(max(hi, lo + 1))))))
    cap = lambda points: max(5, min(700, G // 8, points // G))
    if kind == "apply_h":
        form = rng.choice(("f64", "f32"))
        return _case(kind, None, n, log(3, cap(8_000_000)), form=form,
                     totals=form == "f64" and rng.random() < 0.5)
    if kind == "damped_step":
        return _case(kind, None, n, log(3, cap(8_000_000)), form=rng.choice(("f64", "f32")),
                     weight=rng.random() < 0.5)
    if kind == "matrices":
        return _case(kind, None, n, log(3, min(400, cap(6_000_000))))
    if kind == "rotate":
        return _case(kind, None, n, log(3, min(500, cap(8_000_000))),
                     form=rng.choice(("f64", "f32", "bf16x3", "bf16x6")))
    if kind == "eigen":
        a, b = log(3, 700), log(2, 300)
        return _case(kind, None, (8, 8, 8), max(a, b), min(a, b))
    if kind == "iteration":
        N = log(6, min(280, cap(4_000_000)))
        return _case(kind, None, n, N, max(2, int(N * rng.uniform(0.3, 1.0))), coulomb=rng.random() < 0.5)
    if kind == "td_step":
        N = log(6, min(280, cap(2_000_000)))
        return _case(kind, None, n, N, max(2, int(N * rng.uniform(0.3, 1.0))), form=rng.choice(("f64", "f32")))
    return _case("train", None, n)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _n(c):
    return c["nx"], c["ny"], c["nz"]


def _shape(n):
    return n[2], n[1], n[0]


def _k(n, j, theta=0.0):
    """Wavenumbers of direction j (dx = 1 fm) shaped against [nz, ny, nx]."""
    k = 2.0 * math.pi * torch.fft.fftfreq(n[j], dtype=torch.float64, device=DEV) + theta / n[j]
    shape = [1, 1, 1]
    shape[2 - j] = n[j]
    return k.reshape(shape)


def _twist(seed, on=True):
    g = torch.Generator().manual_seed(int(seed) + 77)
    t = (torch.rand(3, generator=g, dtype=torch.float64) * 2.0 - 1.0) * math.pi
    return tuple(float(v) if on else 0.0 for v in t)


def _states(n, I, gen):
    """Trial states of the benchmark's recipe: complex-normal combinations of
    the lowest 2 I spin plane waves, of norm about 1."""
    G = n[0] * n[1] * n[2]
    k2 = (_k(n, 0) ** 2 + _k(n, 1) ** 2 + _k(n, 2) ** 2).reshape(-1)
    low = torch.sort(k2, stable=True).indices[:min(I, G)]
    spec = torch.zeros((I, 2, G), dtype=torch.complex128, device=DEV)
    spec[:, :, low] = torch.randn((I, 2, low.numel()), dtype=torch.complex128, device=DEV, generator=gen)
    psi = torch.fft.ifftn(spec.reshape((I, 2) + _shape(n)), dim=(-3, -2, -1))
    return psi * (G / math.sqrt(G * 2.0 * low.numel()))


def _blobs(n, gen, nblob=6, sigma=2.0):
    """Periodic Gaussian blobs at random centres, largest value 1."""
    f = torch.zeros(_shape(n), dtype=torch.float64, device=DEV)
    for _ in range(nblob):
        u = torch.rand(3, generator=gen, device=DEV, dtype=torch.float64)
        d2 = 0.0
        for j in range(3):
            d = torch.arange(n[j], dtype=torch.float64, device=DEV) - u[j] * n[j]
            d = d - n[j] * torch.round(d / n[j])
            s = [1, 1, 1]
            s[2 - j] = n[j]
            d2 = d2 + (d * d).reshape(s)
        f = f + torch.exp(-d2 / (2.0 * sigma ** 2))
    return (f + 1e-3) / (f.max() + 1e-3)


def _dreal(f, j, n):
    return torch.fft.ifftn(1j * _k(n, j) * torch.fft.fftn(f)).real


def _field(n, gen):
    """A mean field as blobs of nuclear matter give: a well of about -60 MeV, an
    effective mass of 0.7 inside, and the spin-orbit vector along the slope."""
    s = _blobs(n, gen)
    W = torch.stack([12.0 * _dreal(s, j, n) for j in range(3)])
    return -60.0 * s, P["hb2m_n"] * (1.0 + 0.4 * s), W


def _unitary(I, gen):
    a = torch.randn((I, I), dtype=torch.complex128, device=DEV, generator=gen)
    return torch.linalg.qr(a)[0].contiguous()


def _matrices(I, gen):
    """S and H of damped states: S near the identity, H with levels over
    [-60, 40] MeV and none degenerate (as in a twisted box)."""
    a = torch.randn((I, I), dtype=torch.complex128, device=DEV, generator=gen) * (0.03 / math.sqrt(I))
    S = torch.eye(I, dtype=torch.complex128, device=DEV) + a + a.mH
    u = torch.rand(I, generator=gen, device=DEV, dtype=torch.float64)
    lam = -60.0 + 100.0 * (torch.arange(I, device=DEV) + 0.8 * u) / I
    Q = _unitary(I, gen)
    H = (Q * lam) @ Q.mH
    return S.contiguous(), (0.5 * (H + H.mH)).contiguous()


def _cast(c, x):
    return x if c["form"] == "f64" else x.to(torch.complex64)


def _single(c, seed):
    """Inputs of the one-species calls: states, their field, h of them, energies."""
    g, n = _gen(seed), _n(c)
    psi = _cast(c, _states(n, c["states"], g))
    d = {"psi": psi, "field": _field(n, g), "theta": _twist(seed)}
    if c["kind"] in ("damped_step", "matrices"):
        d["h"] = _cast(c, _h(psi, d["field"], n, d["theta"]))
        d["eps"] = _dots(psi, d["h"])
        d["w"] = (0.5 + 1.5 * torch.rand(_shape(n), generator=g, device=DEV, dtype=torch.float32))
    elif c["kind"] == "rotate":
        d["M"] = _unitary(c["states"], g)
    return d


def _workload(n, N, Z, coulomb, twist):
    return IN.Workload(name="box", grid=n, dx=(1.0, 1.0, 1.0), N=N, Z=Z, coulomb=coulomb, twist=twist,
                       x0=X0, E0=E0, init="blobs")


def _boxes(c, seed):
    """(workload, initial states, initial densities) of each box of a whole call."""
    out = []
    for i in range(c.get("boxes", 1)):
        if c["kind"] == "batch":
            n = ((16, 20, 24)[i % 3],) * 3
            A = int(round(0.03 * n[0] ** 3))
            Z = int(math.floor(0.3 * A + 0.5))
            N, coulomb, twisted = A - Z, False, True
        else:
            n, N, Z = _n(c), c["states"], c["protons"]
            coulomb, twisted = c.get("coulomb", False), not c.get("coulomb", False)
        g = _gen(seed * 1000 + i)
        psi = [_states(n, N, g), _states(n, Z, g)]
        s = _blobs(n, g)
        s = s / s.sum()
        rho = torch.stack([N * s, Z * s])
        tau = 0.6 * (3.0 * math.pi ** 2) ** (2.0 / 3.0) * rho ** (5.0 / 3.0)
        out.append((_workload(n, N, Z, coulomb, _twist(seed + i, twisted)), psi, rho, tau))
    return out


# ------------------------------------------------------------------ the calls

class _Context:
    """A library context that is given back with the state that holds it."""

    def __init__(self, n, theta, form, states, coulomb=False):
        stream = torch.cuda.current_stream().cuda_stream
        self.ctx = B.sky_init(n, (1.0, 1.0, 1.0), P, coulomb, theta, PREC[form], states, stream)

    def __del__(self):
        try:
            B.sky_destroy(self.ctx)
        except Exception:
            pass


def prepare(case, seed):
    c, kind = case, case["kind"]
    torch.cuda.set_device(0)
    if kind in ("apply_h", "damped_step", "matrices", "rotate"):
        d = _single(c, seed)
        st = {"kind": kind, "c": c, "I": c["states"], "psi": d["psi"],
              "own": _Context(_n(c), d["theta"], c["form"], c["states"])}
        st["U"], st["B"], st["W"] = (x.contiguous() for x in d["field"])
        st["out"] = torch.empty_like(d["psi"])
        f64 = dict(dtype=torch.float64, device=DEV)
        if kind == "apply_h":
            st["eps"], st["hn2"] = torch.zeros(st["I"], **f64), torch.zeros(st["I"], **f64)
        elif kind == "damped_step":
            st["h"], st["eps"], st["w"] = d["h"], d["eps"], d["w"] if c["weight"] else None
        elif kind == "matrices":
            st["h"] = d["h"]
            st["S"], st["H"] = (torch.zeros((st["I"],) * 2, dtype=torch.complex128, device=DEV) for _ in range(2))
        else:
            st["M"] = d["M"]
        return st
    if kind == "eigen":
        g = _gen(seed)
        I = [c["states"], c["protons"]]
        pairs = [_matrices(i, g) for i in I]
        z = lambda i: torch.zeros((i, i), dtype=torch.complex128, device=DEV)
        return {"kind": kind, "I": I, "S": [p[0] for p in pairs], "H": [p[1] for p in pairs],
                "C": [z(i) for i in I], "M": [z(i) for i in I],
                "lam": [torch.zeros(i, dtype=torch.float64, device=DEV) for i in I],
                "own": _Context((8, 8, 8), (0.0,) * 3, "f64", max(I))}
    if kind == "iteration":
        (w, psi, rho, tau), = _boxes(c, seed)
        s = Solver(w, prec=PREC[c["form"]], concurrent_species=True)
        s.load(psi, rho.cpu().numpy(), tau.cpu().numpy())
        s.step()
        s.capture()
        s.load(psi, rho.cpu().numpy(), tau.cpu().numpy())
        return {"kind": kind, "s": s}
    if kind == "batch":
        boxes = _boxes(c, seed)
        bs = BatchSolver([b[0] for b in boxes], prec=PREC[c["form"]])

        def load():
            torch.cuda.synchronize()
            for s, st, (_, psi, rho, tau) in zip(bs.boxes, bs.streams, boxes):
                with torch.cuda.stream(st):
                    s.load(psi, rho.cpu().numpy(), tau.cpu().numpy())
            torch.cuda.synchronize()
        load()
        bs.step_eager()
        bs.capture()
        load()
        return {"kind": kind, "bs": bs}
    if kind == "td_step":
        (w, psi, rho, tau), = _boxes(c, seed)
        s = Solver(w, prec=PREC[c["form"]])
        s.load(psi, rho.cpu().numpy(), tau.cpu().numpy())
        return {"kind": kind, "s": s, "td": TimeStepper(s, order=6)}
    if kind == "train":
        t = _training(c, seed)
        net = DampingNet(DEV, theta=t["theta"].cpu().numpy())
        net.m.copy_(t["m"])
        net.v.copy_(t["v"])
        net.step_count = t["step"]
        G = c["nx"] * c["ny"] * c["nz"]
        w = [torch.zeros(G, dtype=torch.float32, device=DEV) for _ in range(2)]
        net.workspace(G)
        return {"kind": kind, "net": net, "G": G, "w": w, "samples": t["samples"],
                "own": _Context(_n(c), (0.0,) * 3, "f64", 1)}
    raise ValueError(kind)


def _training(c, seed):
    """A network part of the way through its training, and one sample per species."""
    g, n = _gen(seed), _n(c)
    theta = torch.from_numpy(init_params(seed % 1000)).to(DEV)
    theta = theta + 0.05 * torch.randn(theta.shape, generator=g, device=DEV, dtype=torch.float32)
    m = 1e-3 * torch.randn(theta.shape, generator=g, device=DEV, dtype=torch.float64)
    v = 1e-4 * (0.5 + torch.rand(theta.shape, generator=g, device=DEV, dtype=torch.float64))
    samples = []
    for q in range(2):
        U, Bf, W = (x.contiguous() for x in _field(n, g))
        a = _blobs(n, g)
        b = a * (0.3 + 1.5 * _blobs(n, g))
        abc = torch.stack([a, b, a + b]).reshape(3, -1).contiguous()
        samples.append((q, U, Bf, W, abc, abc[2].sum().reshape(1)))
    return {"theta": theta, "m": m, "v": v, "step": 40, "samples": samples}


def run(state):
    st, kind = state, state["kind"]
    if kind == "apply_h":
        ctx, on = st["own"].ctx, st["c"]["totals"]
        B.sky_apply_h(ctx, st["U"], st["B"], st["W"], st["psi"], st["out"], st["I"],
                      st["eps"] if on else None, st["hn2"] if on else None)
        return [st["out"], st["eps"], st["hn2"]] if on else [st["out"]]
    if kind == "damped_step":
        B.sky_damped_step(st["own"].ctx, 0, st["psi"], st["h"], st["eps"], st["out"], st["I"], X0, E0, st["w"])
        return [st["out"]]
    if kind == "matrices":
        B.sky_overlap(st["own"].ctx, st["psi"], st["psi"], st["I"], st["S"])
        B.sky_overlap(st["own"].ctx, st["psi"], st["h"], st["I"], st["H"])
        return [st["S"], st["H"]]
    if kind == "rotate":
        B.sky_rotate(st["own"].ctx, st["psi"], st["M"], st["I"], st["out"])
        return [st["out"]]
    if kind == "eigen":
        B.sky_orthonormalize_batched(st["own"].ctx, st["S"], st["I"], st["C"])
        B.sky_subspace_diag_literal_batched(st["own"].ctx, st["H"], st["C"], st["I"], st["M"], st["lam"])
        return [st["C"], st["M"], st["lam"]]
    if kind == "iteration":
        st["s"].step()
        return _observables(st["s"])
    if kind == "batch":
        st["bs"].step()
        return [_observables(s, few=True) for s in st["bs"].boxes]
    if kind == "td_step":
        st["td"].step(DT)
        return [st["s"].psi[0], st["s"].psi[1]]
    net = st["net"]
    net.loss.zero_()
    for (q, U, Bf, W, abc, norm), w in zip(st["samples"], st["w"]):
        ws, _ = net.workspace(st["G"])
        B.sky_net_forward(st["own"].ctx, q, net.theta, U, Bf, W, ws, w)
        B.sky_net_backward(st["own"].ctx, net.theta, ws, abc, norm, net.grad, net.loss)
    net.step_count += 1
    B.sky_net_adam(st["own"].ctx, net.theta, net.grad, net.m, net.v, net.step_count, 3e-3)
    return [net.theta, st["w"][0], st["w"][1]]


def _observables(s, few=False):
    """Levels, energies, densities and mean field of a solver after an iteration."""
    out = [s.lam, s.eout, s.spread, s.rho, s.tau, s.divJ, s.U]
    return out if few else out + [s.J, s.Bf, s.W]


# ------------------------------------------------------------------ necessary work

def work(case):
    c, kind = case, case["kind"]
    n = _n(c)
    G = n[0] * n[1] * n[2]
    V, I, b = 2 * G, c["states"], 16 if c["form"] == "f64" else 8
    lg = sum(math.log2(v) for v in n)
    h = lambda I: I * G * (40.0 * lg + 150.0)              # FFT derivatives and the pointwise terms
    step = lambda I: I * G * (20.0 * lg + 20.0)
    eig = lambda I: I ** 3 * (16.0 / 3.0 + 8.0 + 4 * 8.0)   # reduction, back-transformation, four products
    if kind == "apply_h":
        return {"bytes": 2 * b * V * I + 40 * G, "flops": h(I)}
    if kind == "damped_step":
        return {"bytes": 3 * b * V * I + 12 * G, "flops": step(I)}
    if kind == "matrices":
        return {"bytes": 2 * b * V * I + 32 * I * I, "flops": 8.0 * V * I * (I + 1)}
    if kind == "rotate":
        return {"bytes": 2 * b * V * I + 16 * I * I, "flops": 8.0 * V * I * I}
    if kind == "eigen":
        both = (c["states"], c["protons"])
        return {"bytes": sum(64 * i * i for i in both), "flops": sum(eig(i) for i in both)}
    if kind in ("iteration", "batch"):
        byts = flops = 0.0
        boxes = [(n, I, c["protons"])]
        if kind == "batch":
            boxes = [((m,) * 3, round(0.03 * m ** 3) * 0.7, round(0.03 * m ** 3) * 0.3)
                     for m in ((16, 20, 24)[i % 3] for i in range(c["boxes"]))]
        for m, *parts in boxes:
            g = m[0] * m[1] * m[2]
            lg_m = sum(math.log2(v) for v in m)
            for i in parts:
                byts += 2 * b * 2 * g * i + 160 * g          # the states in and out, the fields
                flops += 2 * i * g * (40.0 * lg_m + 150.0) + i * g * (40.0 * lg_m + 80.0)
                flops += 8.0 * 2 * g * i * (i + 1) + 8.0 * 2 * g * i * i + eig(i)
        return {"bytes": byts, "flops": flops}
    if kind == "td_step":
        A = I + c["protons"]
        return {"bytes": 2 * b * V * A + 320 * G, "flops": 12 * h(A) + 2 * A * G * (20.0 * lg + 60.0)}
    conv = 2.0 * 27 * (3 * 16 + 16 * 16 + 16)
    return {"bytes": 2 * (64 + 4) * G, "flops": 2 * 3 * conv * G}


# ------------------------------------------------------------------ plain 64-bit values

def _grad(x, j, n, theta):
    """Spectral derivative along one axis of [..., nz, ny, nx]."""
    return torch.fft.ifft(1j * _k(n, j, theta[j]) * torch.fft.fft(x, dim=-1 - j), dim=-1 - j)


def _sxw(j, W, p0, p1):
    """((sigma x W)_j psi) by components."""
    wx, wy, wz = W
    if j == 0:
        return -wy * p0 - 1j * wz * p1, 1j * wz * p0 + wy * p1
    if j == 1:
        return wx * p0 - wz * p1, -wz * p0 - wx * p1
    return (wy + 1j * wx) * p1, (wy - 1j * wx) * p0


def _h(psi, field, n, theta):
    """h psi = U psi - sum_j [d_j B d_j + (i/2)(A_j d_j + d_j A_j)] psi, A = sigma x W."""
    U, Bf, W = (f.reshape((-1,) + _shape(n)) for f in field)
    out = torch.empty(psi.shape, dtype=torch.complex128, device=psi.device)
    for a in range(0, psi.shape[0], 64):
        p = psi[a:a + 64].to(torch.complex128)
        r = U * p
        for j in range(3):
            d = _grad(p, j, n, theta)
            l0, l1 = _sxw(j, W, d[:, 0], d[:, 1])
            f0, f1 = _sxw(j, W, p[:, 0], p[:, 1])
            flux = -Bf * d - 0.5j * torch.stack([f0, f1], 1)
            r = r - 0.5j * torch.stack([l0, l1], 1) + _grad(flux, j, n, theta)
        out[a:a + 64] = r
    return out


def _dots(a, b):
    a, b = (x.reshape(x.shape[0], -1) for x in (a, b))
    return torch.cat([(x.to(torch.complex128).conj() * y.to(torch.complex128)).sum(1).real
                      for x, y in zip(a.split(64), b.split(64))])


def _damped(psi, h, eps, n, theta, hb2m, w=None):
    Pk = X0 / (E0 + hb2m * sum(_k(n, j, theta[j]) ** 2 for j in range(3)))
    out = torch.empty(psi.shape, dtype=torch.complex128, device=psi.device)
    for a in range(0, psi.shape[0], 64):
        p = psi[a:a + 64].to(torch.complex128)
        r = h[a:a + 64].to(torch.complex128) - eps[a:a + 64, None, None, None, None] * p
        u = torch.fft.ifftn(Pk * torch.fft.fftn(r, dim=(-3, -2, -1)), dim=(-3, -2, -1))
        out[a:a + 64] = p - (u if w is None else w.to(torch.float64) * u)
    return out


def _overlap(a, b):
    X = a.reshape(a.shape[0], -1).conj() @ b.reshape(b.shape[0], -1).T
    L = torch.tril(X, -1)
    return L + L.mH + torch.diag(torch.diagonal(X).real.to(X.dtype))


def _isqrt(S):
    s, Xv = torch.linalg.eigh(S)
    return (Xv / torch.sqrt(s)) @ Xv.mH


def _mix(phi, M):
    return (M.T @ phi.reshape(phi.shape[0], -1)).reshape(phi.shape)


def _dens(psi, n, theta):
    shape = _shape(n)
    rho, tau = (torch.zeros(shape, dtype=torch.float64, device=DEV) for _ in range(2))
    J = torch.zeros((3,) + shape, dtype=torch.float64, device=DEV)
    for p in psi.split(64):
        p = p.to(torch.complex128)
        rho += (p.abs() ** 2).sum((0, 1))
        for j in range(3):
            d = _grad(p, j, n, theta)
            tau += (d.abs() ** 2).sum((0, 1))
            c00, c11 = (p[:, 0].conj() * d[:, 0]).sum(0), (p[:, 1].conj() * d[:, 1]).sum(0)
            c01, c10 = (p[:, 0].conj() * d[:, 1]).sum(0), (p[:, 1].conj() * d[:, 0]).sum(0)
            m = (c01.imag + c10.imag, c10.real - c01.real, c00.imag - c11.imag)   # Im psi^+ sigma_k d_j psi
            J[(j + 2) % 3] += m[(j + 1) % 3]           # eps_ijk = 1 for (i, j, k) cyclic
            J[(j + 1) % 3] -= m[(j + 2) % 3]
    return rho, tau, J, sum(_dreal(J[i], i, n) for i in range(3))


def _couplings():
    t0, t1, t2, t3, x0, x1, x2, x3 = (P[k] for k in ("t0", "t1", "t2", "t3", "x0", "x1", "x2", "x3"))
    return {"rho": (3 * t0 / 8, -t0 * (0.5 + x0) / 4), "rhoa": (t3 / 16, -t3 * (0.5 + x3) / 24),
            "tau": (3 * t1 / 16 + t2 * (1.25 + x2) / 4, -t1 * (0.5 + x1) / 8 + t2 * (0.5 + x2) / 8),
            "drho": (-9 * t1 / 64 + t2 * (1.25 + x2) / 16, 3 * t1 * (0.5 + x1) / 32 + t2 * (0.5 + x2) / 32),
            "nJ": (-0.75 * P["W0"], -0.25 * P["W0"])}


def _lap(f, n):
    k2 = sum(_k(n, j) ** 2 for j in range(3))
    return torch.fft.ifftn(-k2 * torch.fft.fftn(f)).real


def _coulomb(rho, n):
    k2 = sum(_k(n, j) ** 2 for j in range(3))
    inv = torch.where(k2 > 0, 1.0 / torch.where(k2 > 0, k2, torch.ones_like(k2)), torch.zeros_like(k2))
    return torch.fft.ifftn(4 * math.pi * P["e2"] * inv * torch.fft.fftn(rho)).real


def _mean(rho, tau, divJ, n, coulomb):
    C, al = _couplings(), P["alpha"]
    iso = lambda f: (f[0] + f[1], f[0] - f[1])
    r, t, d = iso(rho), iso(tau), iso(divJ)
    U, Bf, W = torch.zeros_like(rho), torch.zeros_like(rho), torch.zeros((2, 3) + rho.shape[1:], dtype=rho.dtype, device=DEV)
    for q in range(2):
        for T in range(2):
            s = 1.0 if T == 0 or q == 0 else -1.0
            U[q] += s * (2 * (C["rho"][T] + C["rhoa"][T] * r[0] ** al) * r[T] + C["tau"][T] * t[T]
                         + 2 * C["drho"][T] * _lap(r[T], n) + C["nJ"][T] * d[T])
            U[q] += al * r[0] ** (al - 1) * C["rhoa"][T] * r[T] ** 2
            Bf[q] += s * C["tau"][T] * r[T]
            for j in range(3):
                W[q, j] -= s * C["nJ"][T] * _dreal(r[T], j, n)
        Bf[q] += P["hb2m_n"] if q == 0 else P["hb2m_p"]
    if coulomb:
        U[1] += _coulomb(rho[1], n)
    return U, Bf, W


def _energy(rho, tau, divJ, n, coulomb):
    C = _couplings()
    iso = lambda f: (f[0] + f[1], f[0] - f[1])
    r, t, d = iso(rho), iso(tau), iso(divJ)
    e = [(P["hb2m_n"] * tau[0] + P["hb2m_p"] * tau[1]).sum()]
    e += [sum(((C["rho"][T] + C["rhoa"][T] * r[0] ** P["alpha"]) * r[T] ** 2).sum() for T in range(2)),
          sum((C["tau"][T] * r[T] * t[T]).sum() for T in range(2)),
          sum((C["drho"][T] * r[T] * _lap(r[T], n)).sum() for T in range(2)),
          sum((C["nJ"][T] * r[T] * d[T]).sum() for T in range(2))]
    e.append(0.5 * (rho[1] * _coulomb(rho[1], n)).sum() if coulomb else torch.zeros_like(e[0]))
    return torch.stack([sum(e)] + e + [(rho[0] + rho[1]).sum()])


def _exact_iteration(w, psi0, rho, tau, few):
    n, th, co = w.grid, w.twist, w.coulomb
    U, Bf, W = _mean(rho, tau, torch.zeros_like(rho), n, co)
    lam, eps, hn2, new = [], [], [], []
    for q in range(2):
        p = _mix(psi0[q], _isqrt(_overlap(psi0[q], psi0[q])))
        field = (U[q], Bf[q], W[q])
        h = _h(p, field, n, th)
        eps.append(_dots(p, h))
        hn2.append(_dots(h, h))
        phi = _damped(p, h, eps[q], n, th, P["hb2m_n"] if q == 0 else P["hb2m_p"])
        C = _isqrt(_overlap(phi, phi))
        Hp = C.mH @ _overlap(phi, _h(phi, field, n, th)) @ C
        l, Z = torch.linalg.eigh(0.5 * (Hp + Hp.mH))
        lam.append(l)
        new.append(_dens(_mix(phi, C @ Z), n, th))
    eps, hn2 = torch.cat(eps), torch.cat(hn2)
    spread = torch.stack([torch.sqrt((hn2 - eps ** 2).sum() / eps.numel()), eps.sum()])
    rho, tau, J, dJ = (torch.stack([d[i] for d in new]) for i in range(4))
    U, Bf, W = _mean(rho, tau, dJ, n, co)
    out = [torch.cat(lam), _energy(rho, tau, dJ, n, co), spread]
    out += [x.reshape(2, -1) for x in (rho, tau, dJ, U)]
    return out if few else out + [J.reshape(2, 3, -1), Bf.reshape(2, -1), W.reshape(2, 3, -1)]


def _exact_td(w, psi0, rho, tau):
    n, th, co = w.grid, w.twist, w.coulomb
    fields = _mean(rho, tau, torch.zeros_like(rho), n, co)
    psi = [_mix(p, _isqrt(_overlap(p, p))) for p in psi0]

    def taylor(p, q, t):
        term, s = p, p
        for k in range(1, 7):
            term = (-1j * t / k) * _h(term, tuple(f[q] for f in fields), n, th)
            s = s + term
        return s
    half = [_dens(taylor(psi[q], q, 0.5 * DT / HBARC), n, th) for q in range(2)]
    rho, tau, _, dJ = (torch.stack([d[i] for d in half]) for i in range(4))
    fields = _mean(rho, tau, dJ, n, co)
    return [taylor(psi[q], q, DT / HBARC) for q in range(2)]


def _exact_train(c, seed):
    t, n = _training(c, seed), _n(c)
    th = t["theta"].double().requires_grad_(True)
    conv = lambda x, W, b: torch.nn.functional.conv3d(
        torch.nn.functional.pad(x[None], (1,) * 6, mode="circular"), W.reshape(W.shape[0], W.shape[1], 3, 3, 3), b)[0]
    cuts = torch.split(th, [16 * 3 * 27, 16, 16 * 16 * 27, 16, 16 * 27, 1])
    total, ws = 0.0, []
    for q, U, Bf, W, abc, norm in t["samples"]:
        hb = P["hb2m_n"] if q == 0 else P["hb2m_p"]
        x = torch.stack([U / B.SKY_NET_USCALE, Bf / hb - 1.0, torch.sqrt((W * W).sum(0)) / B.SKY_NET_WSCALE])
        x = torch.tanh(conv(x, cuts[0].reshape(16, 3, 27), cuts[1]))
        x = torch.tanh(conv(x, cuts[2].reshape(16, 16, 27), cuts[3]))
        w = (B.SKY_NET_WMAX * torch.sigmoid(conv(x, cuts[4].reshape(1, 16, 27), cuts[5]))).reshape(-1)
        total = total + (abc[0] * w * w - 2.0 * abc[1] * w + abc[2]).sum() / norm[0]
        ws.append(w.detach())
    g, = torch.autograd.grad(total, th)
    k, b1, b2 = t["step"] + 1, 0.9, 0.999
    m, v = b1 * t["m"] + (1 - b1) * g, b2 * t["v"] + (1 - b2) * g * g
    new = th.detach() - 3e-3 * (m / (1 - b1 ** k)) / (torch.sqrt(v / (1 - b2 ** k)) + 1e-8)
    return [new] + ws


def exact(case, seed):
    c, kind = case, case["kind"]
    n = _n(c)
    if kind in ("apply_h", "damped_step", "matrices", "rotate"):
        d = _single(c, seed)
        if kind == "apply_h":
            h = _h(d["psi"], d["field"], n, d["theta"])
            return [h, _dots(d["psi"], h), _dots(h, h)] if c["totals"] else [h]
        if kind == "damped_step":
            return [_damped(d["psi"], d["h"], d["eps"], n, d["theta"], P["hb2m_n"], d["w"] if c["weight"] else None)]
        if kind == "matrices":
            return [_overlap(d["psi"], d["psi"]), _overlap(d["psi"], d["h"])]
        return [_mix(d["psi"].to(torch.complex128), d["M"])]
    if kind == "eigen":
        g = _gen(seed)
        Cs, Ms, lams = [], [], []
        for S, H in [_matrices(i, g) for i in (c["states"], c["protons"])]:
            Cm = _isqrt(S)
            lam, Z = torch.linalg.eigh(H)
            top = torch.gather(Z, 0, Z.abs().argmax(0, keepdim=True))[0]
            Cs.append(Cm)
            Ms.append((Z * (top.conj() / top.abs())) @ Cm)
            lams.append(lam)
        return [Cs, Ms, lams]
    if kind == "iteration":
        (w, psi, rho, tau), = _boxes(c, seed)
        return _exact_iteration(w, psi, rho, tau, False)
    if kind == "batch":
        return [_exact_iteration(w, psi, rho, tau, True) for w, psi, rho, tau in _boxes(c, seed)]
    if kind == "td_step":
        (w, psi, rho, tau), = _boxes(c, seed)
        return _exact_td(w, psi, rho, tau)
    return _exact_train(c, seed)
