"""Performance cases: what a user of this package has it compute, in the sizes,
precisions and options it is used with.

One case is one call sequence of the public Python API (KSCurve, KSBatch,
CurveCost): load a curve, run descent steps (or evaluate the cost or its
gradient) and read the results back.  Inputs are synthetic: the stored Newton
equilibria as end sections, the tanh combination of them as the curve, plus
seeded smooth perturbations that vanish at both ends.
"""
import math
import types

import numpy as np
import torch

from paper_2301_11704_gb300 import gen
from paper_2301_11704_gb300.autograd import CurveCost
from paper_2301_11704_gb300.batch import KSBatch
from paper_2301_11704_gb300.curve import KSCurve

NPERT = 4          # s-modes of the trial curve's perturbation
DTAU = 0.01        # the published descent step (IMEX)


def _descent(name, N, Ns, steps, precision, **kw):
    c = dict(name=name, kind="descend", N=N, Ns=Ns, steps=steps, precision=precision, adjoint="paper",
             scheme="imex", dtau=DTAU, symmetry=0, lambda_free=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: load a curve and evaluate J and J_arc (a line search, a check of a guess)
        dict(name="cost_fp64_n32_s128", kind="cost", N=32, Ns=128, precision="fp64"),
        # the published E1 -> E2 search: N = 64, M = 550, FP64, tens of thousands of steps
        _descent("descend_fp64_n64_s552", 64, 552, 64, "fp64"),
        # the L = 22 curve of the differentiation workload, descended in FP32
        _descent("descend_fp32_n64_s1024", 64, 1024, 64, "fp32"),
        # differentiation: J^2 and its exact gradient through autograd, FP64 (L near 60)
        dict(name="gradient_fp64_n32_s1024", kind="gradient", N=32, Ns=1024, precision="fp64"),
        # a search in the odd subspace kept in sine storage, exact adjoint, lambda free, ragged N_s
        _descent("descend_fp32_sine_n128_s3001", 128, 3001, 32, "fp32", adjoint="discrete", symmetry=5,
                 lambda_free=True),
        # a single large curve (L = 44)
        _descent("descend_fp32_n128_s4096", 128, 4096, 32, "fp32"),
        # full-linear-implicit stepping at 20x the explicit step (runs to the floor of J_arc)
        _descent("implicit_fp64_n64_s552", 64, 552, 32, "fp64", scheme="implicit", dtau=0.2),
        # the largest curve end to end: state from pinned host memory, one step, state and cost back
        _descent("end_to_end_fp32_n256_s16384", 256, 16384, 1, "fp32", host=True),
        # the largest curve with split-BF16 x-transforms, and with FP32 FFTs
        _descent("descend_bf16x2_n256_s16384", 256, 16384, 16, "bf16x2"),
        _descent("descend_fp32_n256_s16384", 256, 16384, 16, "fp32"),
        # many independent searches at once: the 256-curve workload in FP32, a smaller batch in FP64
        dict(name="batch_fp32_256", kind="batch", curves=256, first=0, steps=96, precision="fp32"),
        dict(name="batch_fp64_24", kind="batch", curves=24, first=0, steps=16, precision="fp64"),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["descend", "descend", "descend", "descend", "cost", "gradient", "batch"])
    N = rng.choice([32, 64, 128, 256])
    if kind == "cost":
        return dict(kind="cost", N=N, Ns=_loguniform(rng, 65, 4096), precision=rng.choice(["fp64", "fp32"]))
    if kind == "gradient":
        return dict(kind="gradient", N=32, Ns=_loguniform(rng, 128, 3000), precision="fp64")
    if kind == "batch":
        curves, prec = _loguniform(rng, 8, 160), rng.choice(["fp64", "fp32", "fp32"])
        if prec == "fp64":
            curves = min(curves, 24)
        return dict(kind="batch", curves=curves, first=rng.randrange(0, 256 - curves), steps=rng.choice([8, 16, 24]),
                    precision=prec)
    prec = rng.choice(["fp32", "fp32", "fp32", "fp64", "fp64", "bf16x2"])
    Ns = _loguniform(rng, 128, 4096 if prec == "fp64" else 16384)
    if prec == "bf16x2":
        N, Ns = max(N, 64), max(Ns, 1024)
    sine = prec != "bf16x2" and rng.random() < 0.25
    steps = max(1, min(64, int(16 * 16384 * 256 / (N * Ns * (8 if prec == "fp64" else 1)) * rng.uniform(0.3, 1.0))))
    c = _descent("", N, Ns, steps, prec, adjoint=rng.choice(["paper", "paper", "discrete"]),
                 symmetry=5 if sine else rng.choice([0, 0, 0, 1]), lambda_free=rng.random() < 0.25)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _ends(N, kind):
    """L and the end sections of a curve with N modes: a stored equilibrium, and u = 0.
    Differentiation takes the batch workload's longest domain with N modes: the raw gradient
    carries the k^8 of the top mode, which at L = 22, N = 64 leaves FP64 seven digits of it."""
    if kind == "gradient":
        sp = max((s for s in gen.workload(3) if s.N == N), key=lambda s: s.L)
        return (sp.L, *gen.end_points(sp))
    sp = {32: gen.workload(0)[0], 64: gen.workload(1)[0], 128: gen.workload(2)[0], 256: gen.workload(4)[0]}[N]
    up, um = gen.end_points(sp)
    return sp.L, up, um


def _fields(N, L, seed, odd):
    """Amplitudes and smooth spatial fields of the perturbation, from the seed."""
    rng = np.random.RandomState(seed % (1 << 32))
    x = np.arange(N) * (L / N)
    v = np.zeros((NPERT, N))
    for p in range(NPERT):
        for j in range(1, 5):
            a, b = rng.standard_normal(2)
            v[p] += b * np.sin(2 * np.pi * j * x / L) + (0.0 if odd else a) * np.cos(2 * np.pi * j * x / L)
        v[p] /= np.abs(v[p]).max()
    return rng.uniform(0.05, 0.2, NPERT), v


def _trial(N, Ns, S, up, um, amps, v):
    """1/2[(1 + tanh s) u_+ + (1 - tanh s) u_-] + sum_p A_p sin(p theta) v_p at s = S cot(theta), FP64."""
    dev = "cuda"
    th = torch.arange(Ns, dtype=torch.float64, device=dev) * (math.pi / (Ns - 1))
    t = torch.tanh(S / torch.tan(th[1:-1]))
    t = torch.cat([t.new_ones(1), t, -t.new_ones(1)])[:, None]
    up, um = (torch.as_tensor(q, device=dev)[None, :] for q in (up, um))
    u = 0.5 * ((1 + t) * up + (1 - t) * um)
    for p in range(len(amps)):
        s = torch.sin((p + 1) * th)
        s[-1] = 0
        u = u + float(amps[p]) * s[:, None] * torch.as_tensor(v[p], device=dev)[None, :]
    return u


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _single(case, seed):
    """The curve of a case that is not a batch, as its user has it: physical, in the storage type."""
    N, Ns = case["N"], case["Ns"]
    L, up, um = _ends(N, case["kind"])
    S = gen.mapping_scale(Ns)
    amps, v = _fields(N, L, seed, odd=case.get("symmetry", 0) & 1)
    return L, S, up, um, _trial(N, Ns, S, up, um, amps, v).to(_dtype(case))


def _batch(case, seed):
    specs = gen.workload(3)[case["first"]:case["first"] + case["curves"]]
    ends = [gen.end_points(s) for s in specs]
    pert = [_fields(s.N, s.L, seed * 1000 + i, odd=False) for i, s in enumerate(specs)]
    return specs, ends, pert


def prepare(case, seed):
    st = types.SimpleNamespace(case=case)
    if case["kind"] == "batch":
        specs, ends, pert = _batch(case, seed)
        st.batch = KSBatch(specs, [e[0] for e in ends], [e[1] for e in ends], precision=case["precision"])
        st.amps, st.v = np.stack([p[0] for p in pert]), [p[1] for p in pert]
        return st
    L, S, up, um, u = _single(case, seed)
    if case["kind"] == "gradient":
        st.cost = CurveCost(L, case["N"], case["Ns"], S, up, um, precision=case["precision"])
        st.u = u[1:-1].clone().requires_grad_()
        st.lam = torch.tensor(1.0, dtype=torch.float64, device="cuda", requires_grad=True)
        return st
    kw = {}
    if case["kind"] == "descend":
        kw = dict(adjoint=case["adjoint"], scheme=case["scheme"], dtau=case["dtau"], symmetry=case["symmetry"],
                  lambda_free=case["lambda_free"], dtau_lambda=1e-5 if case["lambda_free"] else 0.0)
    st.curve = KSCurve(L, case["N"], case["Ns"], S, up, um, precision=case["precision"], **kw)
    st.u = u.cpu().pin_memory() if case.get("host") else u
    return st


def run(st):
    case = st.case
    if case["kind"] == "batch":
        b = st.batch
        b.init_trial(st.amps, st.v)
        out = b.descend(case["steps"])
        # the costs in the precision the curves are computed in
        f = np.float64 if case["precision"] == "fp64" else np.float32
        return {"u": torch.cat([b.get_state(i).reshape(-1) for i in range(b.nb)]),
                "J": out["J"].astype(f), "J_arc": out["J_arc"].astype(f), "steps": out["steps"]}
    if case["kind"] == "gradient":
        J2 = st.cost(st.u, st.lam)
        gu, gl = torch.autograd.grad(J2, (st.u, st.lam))
        return {"J2": J2.detach(), "grad_u": gu, "grad_lambda": gl}
    c = st.curve
    u = st.u.to("cuda", non_blocking=True) if case.get("host") else st.u
    c.set_state(u)
    if case["kind"] == "cost":
        J2, Ja = c.cost()
        return {"J2": J2, "J_arc": Ja}
    out = c.descend(case["steps"])
    r = {"J": out["J"], "J_arc": out["J_arc"], "steps": out["steps"], "u": c.get_state()}
    if case.get("host"):
        r["u"] = r["u"].cpu()
    if case["lambda_free"]:
        r["lambda"] = c.get_lambda_tau()[0]
    return r


# ---------------------------------------------------------------------------
# Work of a pass
# ---------------------------------------------------------------------------

def _step_work(N, Ns, b):
    """Bytes of a state read once and written once, and the operations of one step:
    four x-transforms and the products per section, four s-transforms."""
    pts = Ns - 2
    return 2.0 * N * Ns * b, pts * (12.5 * N * math.log2(N) + 10 * N * math.log2(2 * (Ns - 1)) + 30 * N)


def work(case):
    b = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "batch":
        w = [_step_work(s.N, s.Ns, b) for s in gen.workload(3)[case["first"]:case["first"] + case["curves"]]]
        return {"bytes": sum(x[0] for x in w), "flops": case["steps"] * sum(x[1] for x in w)}
    N, Ns = case["N"], case["Ns"]
    by, fl = _step_work(N, Ns, b)
    if case["kind"] == "cost":
        return {"bytes": by / 2, "flops": fl / 2}
    if case["kind"] == "gradient":
        return {"bytes": by, "flops": fl}
    if case["scheme"] == "implicit":   # and two products with the half-size eigenbases
        fl += 2 * 2 * 2 * (Ns / 2 - 1) ** 2 * N
    return {"bytes": by, "flops": case["steps"] * fl}


# ---------------------------------------------------------------------------
# The same results in 64 bits, with torch
# ---------------------------------------------------------------------------

class _Exact:
    """f, D_t, the residual, the adjoint and the descent of one curve in FP64 /
    complex128: Fourier in x by rfft (Nyquist dropped), d/dtheta by the FFT of
    the even extension over 2 (N_s - 1) points."""

    def __init__(self, N, Ns, L, S, lam=1.0, symmetry=0):
        dev = "cuda"
        self.N, self.P, self.L, self.lam, self.sym = N, Ns - 1, L, lam, symmetry
        th = torch.arange(Ns, dtype=torch.float64, device=dev) * (math.pi / self.P)
        sin2 = torch.sin(th) ** 2
        sin2[0] = sin2[-1] = 0
        self.g = (-sin2 / S)[:, None]                       # dtheta/ds
        self.w = torch.zeros(Ns, dtype=torch.float64, device=dev)
        self.w[1:-1] = (math.pi / self.P) * S / sin2[1:-1]
        k = torch.fft.fftfreq(2 * self.P, 1.0 / (2 * self.P), device=dev, dtype=torch.float64)
        k[self.P] = 0
        self.ik = (1j * k)[:, None]
        kx = torch.arange(N // 2, dtype=torch.float64, device=dev) * (2 * math.pi / L)
        self.kx, self.a = kx[None, :], (kx ** 4 - kx ** 2)[None, :]

    def spec(self, u):
        return torch.fft.rfft(u, dim=1)[:, :-1] / self.N

    def keep(self, h):
        """The part of a spectrum that the symmetric subspace keeps (odd sections)."""
        return torch.complex(torch.zeros_like(h.imag), h.imag) if self.sym & 1 else h

    def phys(self, h):
        return torch.fft.irfft(torch.cat([h * self.N, torch.zeros_like(h[:, :1])], 1), n=self.N, dim=1)

    def dt(self, h):
        e = torch.cat([h, h[1:-1].flip(0)], 0)
        return self.g * torch.fft.ifft(self.ik * torch.fft.fft(e, dim=0), dim=0)[:self.P + 1]

    def dtT(self, h):
        e = torch.zeros(2 * self.P, h.shape[1], dtype=h.dtype, device=h.device)
        e[:self.P + 1] = self.g * h
        x = -torch.fft.ifft(self.ik * torch.fft.fft(e, dim=0), dim=0)
        y = x[:self.P + 1].clone()
        y[1:-1] += x[self.P + 1:].flip(0)
        return y

    def norm2(self, h):
        q = (h.abs() ** 2)
        return self.L * (q[:, 0] + 2 * q[:, 1:].sum(1))

    def dot(self, x, y):
        q = (x * y.conj()).real
        return self.L * (q[:, 0] + 2 * q[:, 1:].sum(1))

    def evaluate(self, h, gradient="paper"):
        """J^2, J_arc, dJ^2/dlambda and G (None without `gradient`)."""
        u = self.phys(h)
        d = self.dt(h)
        r = self.keep(-0.5j * self.kx * self.spec(u * u) - self.a * h - self.lam * d)
        r[0] = 0
        r[-1] = 0
        nr, nd, w = self.norm2(r), abs(self.lam) * self.norm2(d).sqrt(), self.w
        J2 = (w * nr).sum()
        Ja = (w * nr.sqrt() * nd).sum() / (w * nd).sum()
        dl = -2 * (w * self.dot(d, r)).sum()
        if not gradient:
            return J2, Ja, dl, None
        A = self.keep(self.spec(u * self.phys(1j * self.kx * r)) - self.a * r)
        if gradient == "discrete":
            sterm = torch.zeros_like(r)
            sterm[1:-1] = -self.lam * self.dtT(w[:, None] * r)[1:-1] / w[1:-1, None]
        else:
            sterm = self.lam * self.dt(r)
        G = -(A + sterm)
        G[0] = 0
        G[-1] = 0
        return J2, Ja, dl, G

    def interior_dt2(self):
        """The interior block of D_t, squared (dense)."""
        P = self.P
        eye = torch.eye(P + 1, dtype=torch.complex128, device="cuda")
        D = self.dt(eye).real[1:-1, 1:-1]
        return D @ D

    def descend(self, h, steps, dtau, gradient, scheme="imex", dtau_lambda=0.0):
        pre = dtau / (1 + dtau * self.a ** 2)
        inv = None
        if scheme == "implicit":
            D2 = self.interior_dt2()
            eye = torch.eye(self.P - 1, dtype=torch.float64, device="cuda")
            inv = (1 + dtau * self.a[0] ** 2)[:, None, None] * eye - (dtau * self.lam ** 2) * D2
        for _ in range(steps):
            _, _, dl, G = self.evaluate(h, gradient)
            if inv is None:
                h = h + pre * G
            else:
                b = torch.view_as_real(dtau * G[1:-1].T.contiguous())
                h = h.clone()
                h[1:-1] += torch.view_as_complex(torch.linalg.solve(inv, b).contiguous()).T
            self.lam -= dtau_lambda * float(dl)
        return h


def exact(case, seed):
    if case["kind"] == "batch":
        specs, ends, pert = _batch(case, seed)
        us, J, Ja = [], [], []
        for s, (up, um), (amps, v) in zip(specs, ends, pert):
            x = _Exact(s.N, s.Ns, s.L, s.S)
            h = x.descend(x.spec(_trial(s.N, s.Ns, s.S, up, um, amps, v)), case["steps"], s.dtau, "paper")
            j2, ja, _, _ = x.evaluate(h, None)
            us.append(x.phys(h).reshape(-1))
            J.append(float(j2) ** 0.5)
            Ja.append(float(ja))
        return {"u": torch.cat(us), "J": np.array(J), "J_arc": np.array(Ja), "steps": None}
    L, S, up, um, u = _single(case, seed)
    u = u.double()
    x = _Exact(case["N"], case["Ns"], L, S, symmetry=case.get("symmetry", 0))
    h = x.keep(x.spec(u))
    if case["kind"] == "cost":
        j2, ja, _, _ = x.evaluate(h, None)
        return {"J2": float(j2), "J_arc": float(ja)}
    if case["kind"] == "gradient":
        # fixed end sections: the ends the cost holds are u_+ and u_-, the curve's own
        j2, _, dl, G = x.evaluate(h, "discrete")
        g = -2 * (L / case["N"]) * x.w[:, None] * x.phys(G)
        return {"J2": j2, "grad_u": g[1:-1], "grad_lambda": dl}
    h = x.descend(h, case["steps"], case["dtau"], case["adjoint"], case["scheme"],
                  1e-5 if case["lambda_free"] else 0.0)
    lam = x.lam
    j2, ja, _, _ = x.evaluate(h, None)
    r = {"J": float(j2) ** 0.5, "J_arc": float(ja), "steps": None, "u": x.phys(h)}
    if case["lambda_free"]:
        r["lambda"] = lam
    return r
