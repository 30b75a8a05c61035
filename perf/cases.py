"""The work this library is measured on: time stepping (explicit Euler, Heun,
integrating factor; with forcing and with the per-step record), uneven
ensembles, the standalone 2-D real FFTs, the gradient of the final surface
area, and steps on host buffers, each through the calls a user's program
makes.

A case is a dict of plain values.  `kind` names the call:

  step   nsteps steps of `scheme` on one flame (Flame.step, step_heun,
         step_if), optionally with a forcing box and with the device record
         (`record`: "no", "yes", "area")
  batch  flame_step_batch over `flames` flames of uneven grids
  fft    Flame.fft_r2c of each of `fields` fields, then Flame.fft_c2r of its
         spectrum
  grad   FlameArea forward and backward (area after nsteps steps, its gradient
         with respect to the initial state and gamma)
  host   Flame.step_host on pinned host buffers

n1 x n2 is the grid, k1 and k2 the retained harmonics (0: the largest the
grid allows), prec "fp32" or "fp64".

The inputs are wrinkled flames: every retained mode with |k| <= kmax has the
amplitude (1 + |k|)^-2 and a random phase, at radius t0 = 20, where the
quadratic term is at work; the mean mode starts at 2.
"""
import math

import numpy as np
import torch

from paper_0911_2889_gb300 import flame

GAMMA, T0, MEAN0, AMP = 0.5, 20.0, 2.0, 1.0
# The uneven ensemble's grids.
CLASSES = ((256, 512), (512, 1024), (1024, 2048))
# Point updates of the largest listed stepping case; drawn cases stay below.
MOST_UPDATES = 10 * 4096 * 8192


def listed():
    def step(name, prec, n1, n2, nsteps, scheme="euler", k1=0, k2=0, forcing=False, record="no"):
        return {"name": name, "kind": "step", "prec": prec, "n1": n1, "n2": n2, "k1": k1, "k2": k2,
                "nsteps": nsteps, "scheme": scheme, "forcing": forcing, "record": record}
    return [
        # a program that looks at the flame after every step of a small grid:
        # the smallest call
        step("one step 256x512", "fp32", 256, 512, 1),
        # the double precision trajectory on the paper-sized grid
        step("fp64 128x256", "fp64", 128, 256, 100),
        # the single precision trajectory whose drift is watched
        step("fp32 1024x2048", "fp32", 1024, 2048, 100),
        # the large grid, steps back to back
        step("fp32 4096x8192", "fp32", 4096, 8192, 10),
        # a stiff forced run with a truncated box of odd sizes
        step("if forced 512x1024", "fp32", 512, 1024, 25, "if", k1=101, k2=231, forcing=True),
        # a second-order double precision run that records its diagnostics
        step("fp64 heun 512x1024", "fp64", 512, 1024, 5, "heun", record="yes"),
        # a run that records the surface area of every step
        step("area record 1024x2048", "fp32", 1024, 2048, 20, record="area"),
        # an uneven ensemble of flames
        {"name": "ensemble 96", "kind": "batch", "prec": "fp32", "flames": 96, "nsteps": 16, "grids": 1234},
        # the transforms alone, the ends of the sweep over grids
        {"name": "fft 4096x8192", "kind": "fft", "prec": "fp32", "n1": 4096, "n2": 8192, "fields": 1},
        {"name": "fft 256x256", "kind": "fft", "prec": "fp32", "n1": 256, "n2": 256, "fields": 1},
        # gradient of the final area, checkpoints every 20 steps
        {"name": "grad 512x1024", "kind": "grad", "prec": "fp32", "n1": 512, "n2": 1024, "k1": 0, "k2": 0,
         "nsteps": 40, "ckpt": 20},
        # one step end to end from host memory
        {"name": "host 4096x8192", "kind": "host", "prec": "fp32", "n1": 4096, "n2": 8192, "k1": 0, "k2": 0,
         "nsteps": 1},
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "batch", "fft", "grad", "host"])
    prec = "fp32" if rng.random() < 0.7 else "fp64"
    # rows from half as many to four times as many points as columns
    e1 = rng.randint(6, 12 if prec == "fp32" else 10)
    n1 = 2 ** e1
    n2 = 2 ** min(e1 + rng.randint(-1, 2), 13)
    if kind == "fft":
        fields = rng.randint(2, 7)
        return {"kind": kind, "prec": prec, "n1": n1, "n2": n2, "fields": max(1, min(fields, 2 ** 27 // (n1 * n2)))}
    most = MOST_UPDATES // (1 if prec == "fp32" else 16)
    if kind == "batch":
        return {"kind": kind, "prec": prec, "flames": rng.randint(2, 128 if prec == "fp32" else 9),
                "nsteps": rng.randint(1, 16 if prec == "fp32" else 3), "grids": rng.randint(0, 10 ** 6)}

    def harmonics(n):
        top = (n - 1) // 4
        return 0 if rng.random() < 0.6 else rng.randint(max(1, top // 2), top)

    k1, k2 = harmonics(n1), harmonics(n2)
    cap = max(1, most // (n1 * n2))
    if kind == "grad":  # each step costs about three more in the backward sweep
        n1, n2 = min(n1, 1024), min(n2, 2048)
        cap = max(1, most // (4 * n1 * n2))
        k1, k2 = min(k1, (n1 - 1) // 4), min(k2, (n2 - 1) // 4)
        nsteps = rng.randint(1, min(60, cap))
        return {"kind": kind, "prec": prec, "n1": n1, "n2": n2, "k1": k1, "k2": k2, "nsteps": nsteps,
                "ckpt": rng.randint(1, 20)}
    if kind == "host":
        return {"kind": kind, "prec": prec, "n1": n1, "n2": n2, "k1": k1, "k2": k2, "nsteps": rng.randint(1, min(5, cap))}
    scheme = rng.choice(["euler", "euler", "heun", "if"])
    record = rng.choice(["no", "no", "yes", "area"])
    if scheme != "euler":
        cap = max(1, cap // 2)
    if record == "area":
        cap = max(1, cap // 2)
    nsteps = int(round(math.exp(rng.uniform(0.0, math.log(min(100, cap))))))
    return {"kind": kind, "prec": prec, "n1": n1, "n2": n2, "k1": k1, "k2": k2, "nsteps": nsteps, "scheme": scheme,
            "forcing": rng.random() < 0.25, "record": record}


# ------------------------------------------------------------------- inputs
def _box(case):
    n1, n2 = case["n1"], case["n2"]
    return case["k1"] or (n1 - 1) // 4, case["k2"] or (n2 - 1) // 4


def _dt(k1, k2):
    # the explicit step's stability bound on the linear operator, with room
    return min(1e-3, 0.5 * T0 * T0 / (k1 * k1 + k2 * k2))


def _wavenumbers(k1, k2):
    a = torch.arange(-k1, k1 + 1, device="cuda", dtype=torch.float64)[None, :]
    b = torch.arange(0, k2 + 1, device="cuda", dtype=torch.float64)[:, None]
    return a, b


def _spectrum(gen, k1, k2, kmax, amp):
    """Box of shape (k2 + 1, 2 k1 + 1), complex128, real in physical space."""
    a, b = _wavenumbers(k1, k2)
    kn = torch.sqrt(a * a + b * b)
    phase = 2 * math.pi * torch.rand(kn.shape, generator=gen, device="cuda", dtype=torch.float64)
    z = torch.polar(torch.where(kn <= kmax, amp * (1 + kn) ** -2, torch.zeros_like(kn)), phase)
    z[0, :k1] = z[0, k1 + 1:].flip(0).conj()
    z[0, k1] = 0
    return z


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _ctype(case):
    return torch.complex64 if case["prec"] == "fp32" else torch.complex128


def _flame_state(case, gen, k1, k2):
    kmax = max(1, min(256, k1, k2))
    return _spectrum(gen, k1, k2, kmax, AMP).to(_ctype(case)).contiguous()


def _forcing(case, gen, k1, k2):
    return _spectrum(gen, k1, k2, max(1, min(16, k1, k2)), 1e-2).to(_ctype(case)).contiguous()


def _scalar(v):
    return torch.full((1,), v, dtype=torch.float64, device="cuda")


def _grids(case):
    rng = np.random.default_rng(case["grids"])
    return [CLASSES[i] for i in rng.integers(0, len(CLASSES), size=case["flames"])]


def _handle(case, n1, n2, k1, k2):
    return flame.Flame(n1, n2, K1=k1, K2=k2, gamma=GAMMA, t0=T0, dt=_dt(k1, k2), prec=case["prec"])


def _inputs(case, seed):
    """The tensors of a case (what `run` is given), from the seed alone."""
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "fft":
        rt = torch.float32 if case["prec"] == "fp32" else torch.float64
        x = torch.rand((case["fields"], case["n1"], case["n2"]), generator=gen, device="cuda", dtype=torch.float64) * 2 - 1
        return {"x": x.to(rt)}
    if kind == "batch":
        states = []
        for n1, n2 in _grids(case):
            states.append(_flame_state(case, gen, (n1 - 1) // 4, (n2 - 1) // 4))
        return {"states": states}
    k1, k2 = _box(case)
    out = {"state": _flame_state(case, gen, k1, k2)}
    if case.get("forcing"):
        out["forcing"] = _forcing(case, gen, k1, k2)
    return out


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "fft":
        return {"case": case, "flame": _handle(case, case["n1"], case["n2"], 1, 1), "x": x["x"]}
    if kind == "batch":
        fs = [_handle(case, n1, n2, (n1 - 1) // 4, (n2 - 1) // 4) for n1, n2 in _grids(case)]
        return {"case": case, "flames": fs, "states": x["states"], "means": [_scalar(MEAN0) for _ in fs],
                "ts": [_scalar(T0) for _ in fs]}
    k1, k2 = _box(case)
    s = {"case": case, "flame": _handle(case, case["n1"], case["n2"], k1, k2), "state": x["state"],
         "mean": _scalar(MEAN0), "t": _scalar(T0)}
    if kind == "host":
        for k in ("state", "mean", "t"):
            s[k] = s[k].cpu().pin_memory()
    if kind == "grad":
        s["state"].requires_grad_(True)
        s["gamma"] = torch.tensor(GAMMA, requires_grad=True)
    if kind == "step":
        if case["forcing"]:
            s["flame"].set_forcing(x["forcing"], 1e-3)
        if case["record"] != "no":
            s["rec"] = torch.zeros((case["nsteps"], 4), dtype=torch.float64, device="cuda")
            s["flame"].set_record(s["rec"], with_area=case["record"] == "area")
    return s


# -------------------------------------------------------------------- calls
def run(state):
    case, kind = state["case"], state["case"]["kind"]
    n = case.get("nsteps")
    if kind == "fft":
        out = {"spec": [], "field": []}
        for x in state["x"]:
            out["spec"].append(state["flame"].fft_r2c(x))
            out["field"].append(state["flame"].fft_c2r(out["spec"][-1]))
        return out
    if kind == "batch":
        flame.flame_step_batch([f.h for f in state["flames"]], state["states"], state["means"], state["ts"], n)
        # the flames' boxes one after the other, and their scalars
        return {"states": torch.cat([s.reshape(-1) for s in state["states"]]), "means": torch.cat(state["means"]),
                "ts": torch.cat(state["ts"])}
    f = state["flame"]
    if kind == "grad":
        area = flame.FlameArea.apply(state["state"], state["mean"], state["gamma"], f, state["t"], n, case["ckpt"])
        gs, gg = torch.autograd.grad(area, (state["state"], state["gamma"]))
        return {"area": area.detach(), "grad_state": gs, "grad_gamma": gg}
    if kind == "host":
        f.step_host(state["state"], state["mean"], state["t"], n)
    else:
        {"euler": f.step, "heun": f.step_heun, "if": f.step_if}[case["scheme"]](state["state"], state["mean"],
                                                                             state["t"], n)
    out = {"state": state["state"], "mean": state["mean"], "t": state["t"]}
    if "rec" in state:
        out["rec"] = state["rec"]
    return out


def _entry_bytes(case):
    return 8 if case["prec"] == "fp32" else 16


def _rhs_flops(n1, n2, k1, k2):
    """One evaluation of the right-hand side: the transforms of the two
    derivative fields and of their sum of squares (5 n log2 n per complex
    point, real fields half) on a grid of 3 K + 1 points a side, the smallest
    that keeps the quadratic term free of aliases, and the pointwise work."""
    m1, m2 = 3 * k1 + 1, 3 * k2 + 1
    cols = 3 * (k2 + 1) * 5 * m1 * math.log2(m1)
    rows = 3 * m1 * 2.5 * m2 * math.log2(m2)
    return cols + rows + 3 * m1 * m2 + 20 * (2 * k1 + 1) * (k2 + 1)


def work(case):
    e, kind = _entry_bytes(case), case["kind"]
    if kind == "fft":
        n1, n2 = case["n1"], case["n2"]
        field, spec = n1 * n2 * e // 2, n1 * (n2 // 2 + 1) * e
        m = case["fields"]
        return {"bytes": 2 * m * (field + spec), "flops": 2 * 2.5 * m * n1 * n2 * math.log2(n1 * n2)}
    if kind == "batch":
        b = f = 0
        for n1, n2 in _grids(case):
            k1, k2 = (n1 - 1) // 4, (n2 - 1) // 4
            b += 2 * (2 * k1 + 1) * (k2 + 1) * e
            f += case["nsteps"] * _rhs_flops(n1, n2, k1, k2)
        return {"bytes": b, "flops": f}
    k1, k2 = _box(case)
    box = (2 * k1 + 1) * (k2 + 1) * e
    rhs = _rhs_flops(case["n1"], case["n2"], k1, k2)
    n = case["nsteps"]
    if kind == "grad":
        # forward and, in reverse, one transposed step each (two thirds more
        # transforms than a step) from states that have to be there
        area = 2.5 * 5 * case["n1"] * case["n2"] * math.log2(case["n1"] * case["n2"])
        return {"bytes": 2 * box, "flops": n * rhs * (1 + 5 / 3) + 2 * area}
    stages = 1 if case.get("scheme", "euler") == "euler" else 2
    flops = n * stages * rhs
    if case.get("record") == "area":
        n1, n2 = case["n1"], case["n2"]
        flops += n * (2.5 * n1 * n2 * math.log2(n1 * n2) + 10 * n1 * n2)
    return {"bytes": (2 + int(bool(case.get("forcing")))) * box, "flops": flops}


# ------------------------------------------- the same in 64 bits, plain torch
class _Exact:
    """The model on one grid with torch.fft in double precision."""

    def __init__(self, n1, n2, k1, k2, gamma=GAMMA, forcing=None, forcing0=0.0):
        self.n1, self.n2, self.k1, self.k2, self.gamma = n1, n2, k1, k2, gamma
        self.dt = _dt(k1, k2)
        self.a, self.b = _wavenumbers(k1, k2)
        self.kap2 = self.a ** 2 + self.b ** 2
        self.kap = torch.sqrt(self.kap2)
        self.rows = torch.arange(-k1, k1 + 1, device="cuda") % n1
        self.forcing, self.forcing0 = forcing, forcing0

    def synth(self, box):
        full = torch.zeros((self.n2 // 2 + 1, self.n1), dtype=torch.complex128, device="cuda")
        full[: self.k2 + 1, self.rows] = box
        return torch.fft.irfft2(full.T, s=(self.n1, self.n2), norm="forward")

    def grad2(self, box):
        return self.synth(1j * self.a * box) ** 2 + self.synth(1j * self.b * box) ** 2

    def nonstiff(self, box, r0):
        """c [|grad Phi|^2]_k + f_k on the box (k = 0 zeroed) and its mean."""
        ghat = torch.fft.rfft2(self.grad2(box), norm="forward")
        c = 0.5 / (r0 * r0)
        out = c * ghat.T[: self.k2 + 1][:, self.rows]
        mean = (c * ghat[0, 0].real + self.forcing0).detach()
        if self.forcing is not None:
            out = out + self.forcing
        keep = torch.ones(out.shape, device="cuda", dtype=torch.float64)
        keep[0, self.k1] = 0
        return out * keep, mean

    def omega(self, r0):
        return -self.kap2 / (r0 * r0) + self.gamma * self.kap / (2 * r0)

    def area(self, box, mean, t):
        r = t + mean + self.synth(box)
        w = (2 * math.pi) ** 2 / (self.n1 * self.n2)
        return (w * r * torch.sqrt(r * r + self.grad2(box))).sum()

    def step(self, scheme, box, mean, n):
        t, t1, dt = T0 + n * self.dt, T0 + (n + 1) * self.dt, self.dt
        nl, m0 = self.nonstiff(box, t)
        if scheme == "euler":
            return box + dt * (self.omega(t) * box + nl), mean + dt * m0, m0
        if scheme == "heun":
            f0 = self.omega(t) * box + nl
            p = box + dt * f0
            nl1, m1 = self.nonstiff(p, t1)
            return box + 0.5 * dt * (f0 + self.omega(t1) * p + nl1), mean + 0.5 * dt * (m0 + m1), m0
        e = torch.exp(-self.kap2 * (t1 - t) / (t * t1) + 0.5 * self.gamma * self.kap * math.log1p((t1 - t) / t))
        p = e * (box + dt * nl)
        nl1, m1 = self.nonstiff(p, t1)
        return e * (box + 0.5 * dt * nl) + 0.5 * dt * nl1, mean + 0.5 * dt * (m0 + m1), m0


def exact(case, seed):
    x, kind = _inputs(case, seed), case["kind"]
    if kind == "fft":
        fields = [f.double() for f in x["x"]]
        return {"spec": [torch.fft.rfft2(f) for f in fields], "field": [f * (case["n1"] * case["n2"]) for f in fields]}
    if kind == "batch":
        boxes, means, ts = [], [], []
        for (n1, n2), st in zip(_grids(case), x["states"]):
            m = _Exact(n1, n2, (n1 - 1) // 4, (n2 - 1) // 4)
            box, mean = st.to(torch.complex128), _scalar(MEAN0)
            for n in range(case["nsteps"]):
                box, mean, _ = m.step("euler", box, mean, n)
            boxes.append(box.reshape(-1))
            means.append(mean)
            ts.append(_scalar(T0 + case["nsteps"] * m.dt))
        return {"states": torch.cat(boxes), "means": torch.cat(means), "ts": torch.cat(ts)}
    k1, k2 = _box(case)
    box = x["state"].to(torch.complex128)
    if kind == "grad":
        if case["n1"] * case["n2"] * case["nsteps"] > 2 ** 26:
            return None  # the saved fields of the whole sweep would not be small
        box.requires_grad_(True)
        gamma = torch.tensor(GAMMA, dtype=torch.float64, device="cuda", requires_grad=True)
        m = _Exact(case["n1"], case["n2"], k1, k2, gamma=gamma)
        b, mean = box, _scalar(MEAN0)
        # the mean mode takes part in the area, so its own chain is kept
        for n in range(case["nsteps"]):
            t = T0 + n * m.dt
            ghat0 = m.grad2(b).mean()
            new, _, _ = m.step("euler", b, mean.detach(), n)
            mean = mean + m.dt * 0.5 / (t * t) * ghat0
            b = new
        area = m.area(b, mean, T0 + case["nsteps"] * m.dt)
        gs, gg = torch.autograd.grad(area, (box, gamma))
        gs = gs.clone()
        gs[0, k1] = 0
        return {"area": area.detach().reshape(1), "grad_state": gs, "grad_gamma": gg.cpu()}
    forcing = x["forcing"].to(torch.complex128) if case.get("forcing") else None
    m = _Exact(case["n1"], case["n2"], k1, k2, forcing=forcing, forcing0=1e-3 if case.get("forcing") else 0.0)
    mean, rec = _scalar(MEAN0), []
    scheme = case.get("scheme", "euler")
    for n in range(case["nsteps"]):
        area = _scalar(float("nan"))
        if case.get("record") == "area":
            area = m.area(box, mean, T0 + n * m.dt).reshape(1)
        new, mean1, rate = m.step(scheme, box, mean, n)
        rec.append(torch.cat([_scalar(T0 + n * m.dt), mean, rate.reshape(1), area]))
        box, mean = new, mean1
    out = {"state": box, "mean": mean, "t": _scalar(T0 + case["nsteps"] * m.dt)}
    if case.get("record", "no") != "no":
        out["rec"] = torch.stack(rec)
    return out
