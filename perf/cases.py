"""The work that users of this package have it do, as cases that can be timed.

Three kinds of pass, each through the package's public entry points:

  run       one instance from given initial data: set_state_device, step(n),
            waveform; the state level the steps leave and the n + 1 samples
  batch     the same for several uneven instances advanced by one Batch
  gradient  the gradient of a waveform loss: adjoint.gradients (checkpointed,
            taped, or for the source parameters alone) or waveform_fn with
            autograd

Initial data are smooth: several Gaussian pulses in r* of different widths,
times low polynomials in cos(theta) and the lowest harmonic's envelope, over
the whole grid, with the circular-orbit source on.  The number of steps of
an FP32 run is kept to what the FP32 state resolves (its rounding noise grows
by about 40 times per 85 M of time on these problems).
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_0909_4039_gb300 import adjoint, inputs, teuk

GAMMA = 1.0 - 1.0 / math.sqrt(2.0)


def _run(name, prec, Nr, Nth, steps, a, m, r0, rs_min, rs_max, rs_ext, tuned):
    return {"name": name, "kind": "run", "prec": prec, "Nr": Nr, "Nth": Nth, "steps": steps, "a": a, "m": m, "r0": r0,
            "rs_min": rs_min, "rs_max": rs_max, "rs_ext": rs_ext, "tuned": tuned}


def _gradient(name, prec, Nr, Nth, steps, a, m, r0, rs_max, rs_ext, mode):
    return {"name": name, "kind": "gradient", "prec": prec, "Nr": Nr, "Nth": Nth, "steps": steps, "a": a, "m": m,
            "r0": r0, "rs_min": -100.0, "rs_max": rs_max, "rs_ext": rs_ext, "mode": mode}


def listed():
    return [
        # A few steps of a toy grid (the size the smoke entry and the tests
        # use): what a call costs when there is next to nothing to compute.
        _run("small_96x16_fp64", "fp64", 96, 16, 20, 0.9, 2, 6.0, -20.0, 40.0, 30.0, False),
        # The plain FP64 workload, as it comes without any tuning call.
        _run("plain_1024x32_fp64", "fp64", 1024, 32, 200, 0.9, 2, 10.0, -100.0, 600.0, 500.0, False),
        # The same grid with the FP32 state, autotuned.
        _run("plain_1024x32_fp32", "fp32", 1024, 32, 100, 0.9, 2, 10.0, -100.0, 600.0, 500.0, True),
        # A grid whose sizes fit nothing: prime-like row count, theta rows
        # that are no multiple of a lane's segment, odd azimuthal mode.
        _run("ragged_3001x90_fp32", "fp32", 3001, 90, 130, 0.6, 3, 8.0, -100.0, 600.0, 400.0, False),
        # The large single instance of the benchmark, FP32 and FP64 state.
        _run("single_16384x128_fp32", "fp32", 16384, 128, 200, 0.99, 2, 6.0, -200.0, 1000.0, 500.0, True),
        _run("single_16384x128_fp64", "fp64", 16384, 128, 66, 0.99, 2, 6.0, -200.0, 1000.0, 500.0, True),
        # Fine angular resolution: theta rows of the widest class.
        _run("wide_1500x300_fp64", "fp64", 1500, 300, 40, 0.6, 1, 8.0, -60.0, 240.0, 100.0, False),
        # A parameter study: uneven instances (2048 .. 16384 rows, 32 .. 128
        # theta points, every mode) in one autotuned batch.
        {"name": "uneven_batch16_fp32", "kind": "batch", "set": "uneven", "count": 16, "prec": "fp32", "steps": 130,
         "tuned": True},
        # The long-run batch: eight orbits on the largest grid.
        {"name": "long8_65536x256_fp32", "kind": "batch", "set": "long", "count": 8, "prec": "fp32", "steps": 66,
         "tuned": True},
        # Gradients on the adjoint workload's grid (its extraction radius
        # moved in, so that the orbit's waves arrive within the steps taken):
        # autograd with sqrt(N) checkpoints, and the taped sweep.
        _gradient("autograd_4096x64_fp64", "fp64", 4096, 64, 400, 0.7, 2, 10.0, 600.0, 25.0, "autograd"),
        _gradient("taped_4096x64_fp64", "fp64", 4096, 64, 400, 0.7, 2, 10.0, 600.0, 25.0, "tape"),
        # An FP32 gradient with respect to the source parameters alone.
        _gradient("source_grad_4096x64_fp32", "fp32", 4096, 64, 300, 0.7, 2, 10.0, 600.0, 25.0, "source"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    prec = rng.choice(["fp32", "fp32", "fp64"])
    kind = rng.choice(["run", "run", "run", "batch", "gradient"])
    a, m, r0 = round(rng.uniform(0.0, 0.99), 3), rng.randint(1, 4), round(rng.uniform(6.0, 15.0), 3)
    if kind == "batch":
        return {"kind": "batch", "set": "uneven", "count": rng.randint(2, 24), "prec": prec,
                "steps": rng.randint(20, 130 if prec == "fp32" else 40), "tuned": rng.random() < 0.5, "first": rng.randint(1, 999)}
    if kind == "gradient":
        Nr, Nth = int(_log(rng, 500, 6000)), int(_log(rng, 16, 128))
        Nth = Nth if rng.random() < 0.3 else max(16, Nth // 4 * 4)
        rs_max = round(Nr * _log(rng, 0.1, 0.3) - 100.0, 2)
        c = _gradient("", prec, Nr, Nth, rng.randint(60, 300), a, m, r0, max(60.0, rs_max), 25.0,
                      rng.choice(["autograd", "tape", "source", "checkpoint"]))
    else:
        # the product of the sizes spans the toy grid to the benchmark's
        Nth = int(_log(rng, 12, 320))
        Nth = Nth if rng.random() < 0.3 else max(12, Nth // 4 * 4)
        Nr = int(_log(rng, 90, 16384 if Nth <= 128 else 6000))
        dr = _log(rng, 0.07, 0.7)
        length = max(60.0, Nr * dr)
        lo = -round(min(200.0, length / 4.0), 2)
        steps = rng.randint(20, 200)
        if prec == "fp32":
            steps = max(4, min(steps, int(80.0 * (Nr - 1) / length)))
        c = _run("", prec, Nr, Nth, steps, a, m, r0, lo, round(lo + length, 2), round(lo + 0.7 * length, 2), rng.random() < 0.5)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _workload(c):
    return inputs.Workload("case", s=-2, m=c["m"], a=c["a"], Nr=c["Nr"], Ntheta=c["Nth"], rs_min=c["rs_min"],
                           rs_max=c["rs_max"], steps=c["steps"], r0=c["r0"], rs_ext=c["rs_ext"])


def _instances(c):
    """The workloads of a run or a batch."""
    if c["kind"] != "batch":
        return [_workload(c)]
    if c["set"] == "long":
        return inputs.long_run_batch(c["count"])
    return inputs.batched_instances(c["count"], seed=c.get("first", 0))


def _initial(w, seed):
    """Smooth complex initial data [2][Nr][Ntheta] on the GPU."""
    rng = np.random.default_rng(seed)
    dev = "cuda"
    rs = torch.linspace(w.rs_min, w.rs_max, w.Nr, dtype=torch.float64, device=dev)
    th = (torch.arange(w.Ntheta, dtype=torch.float64, device=dev) + 0.5) * (math.pi / w.Ntheta)
    env = torch.sin(0.5 * th) ** abs(w.m + w.s) * torch.cos(0.5 * th) ** abs(w.m - w.s)
    K, length, dr = 16, w.rs_max - w.rs_min, (w.rs_max - w.rs_min) / (w.Nr - 1)
    centre = torch.as_tensor(w.rs_min + length * (np.arange(K) + rng.uniform(0.0, 1.0, K)) / K, device=dev)
    width = torch.as_tensor(np.maximum(6.0 * dr, length * rng.uniform(0.02, 0.08, K)), device=dev)
    radial = torch.exp(-0.5 * ((rs[:, None] - centre) / width) ** 2)
    radial[0] = radial[-1] = 0.0
    poly = torch.stack([torch.cos(th) ** k for k in range(4)])
    amp = torch.as_tensor(rng.standard_normal((2, K, 4)) + 1j * rng.standard_normal((2, K, 4)), device=dev)
    return torch.einsum("ik,pkq,qj->pij", radial.to(torch.complex128), amp, (poly * env).to(torch.complex128)).contiguous()


def _amplitude(seed):
    rng = np.random.default_rng(seed + 77)
    return complex(rng.uniform(0.5, 1.5), rng.uniform(-0.5, 0.5))


def prepare(case, seed):
    if case["kind"] == "gradient":
        w, amp = _workload(case), _amplitude(seed)
        rng = np.random.default_rng(seed)
        n = case["steps"] + 1
        w = w.with_(r0=w.r0 + float(rng.uniform(-0.5, 0.5)))
        params = torch.tensor([amp.real, amp.imag, w.r0, w.a], dtype=torch.float64, device="cuda")
        dt = w.cfl * (w.rs_max - w.rs_min) / (w.Nr - 1)
        target = torch.as_tensor(inputs.adjoint_target(n, dt, seed=seed, omega_max=2.0), device="cuda")
        return {"case": case, "w": w, "params": params, "prm": adjoint.Params(amp, w.r0, w.a), "target": target,
                "u0": None if case["mode"] == "autograd" else _initial(w, seed)}
    sts, ws = [], _instances(case)
    u0 = [_initial(w, seed + k) for k, w in enumerate(ws)]
    torch.cuda.synchronize()   # a Stepper's set-up runs on its own stream
    for k, w in enumerate(ws):
        drs = (w.rs_max - w.rs_min) / (w.Nr - 1)
        st = teuk.Stepper(s=w.s, m=w.m, a=w.a, Nr=w.Nr, Ntheta=w.Ntheta, rstar_min=w.rs_min, rstar_max=w.rs_max,
                          dt=w.cfl * drs, rstar_extract=w.rs_ext, precision=case["prec"], wave_capacity=case["steps"] + 1)
        st.set_source(_amplitude(seed + k), w.r0, w.sig_r, w.sig_th)
        sts.append(st)
    batch = None
    if case["kind"] == "batch":
        batch = teuk.Batch(sts)
        if case["tuned"]:
            batch.autotune(2 if case["set"] == "long" else 4)
    elif case["tuned"]:
        sts[0].autotune(20)
    torch.cuda.synchronize()
    return {"case": case, "sts": sts, "u0": u0, "batch": batch}


# --------------------------------------------------------------------- run

def _samples(h, prec):
    # the samples are FP64 sums over the state: with the FP32 state they carry
    # its precision, and are kept in it
    return h.astype(np.complex64) if prec == "fp32" else h


def _level(st):
    # the state the steps left, where it lies in the stepper's buffer (Stepper.level_view
    # offers the same where a level is a multiple of 256 bytes)
    off = teuk.teuk_state_level(st.ctx)[0]
    dt = torch.complex64 if st.precision == "fp32" else torch.complex128
    n = 2 * st.Nr * st.Ntheta
    return st.d_state[off:off + n * dt.itemsize].view(dt).view(2, st.Nr, st.Ntheta)


def run(state):
    case = state["case"]
    if case["kind"] == "gradient":
        return _run_gradient(state)
    n = case["steps"]
    for st, u in zip(state["sts"], state["u0"]):
        st.set_state_device(u, 0)
    (state["batch"] or state["sts"][0]).step(n)
    return [(_level(st), _samples(st.waveform(0, n + 1), case["prec"])) for st in state["sts"]]


def _run_gradient(state):
    case, w, n, prec = state["case"], state["w"], state["case"]["steps"], state["case"]["prec"]
    if case["mode"] == "autograd":
        p = state["params"].clone().requires_grad_(True)
        h = adjoint.waveform_fn(p, w, n, precision=prec)
        d = h - state["target"]
        (d.real ** 2 + d.imag ** 2).sum().backward()
        h = h.detach()
        g = p.grad
        return {"h": h if prec == "fp64" else h.to(torch.complex64), "grad": g if prec == "fp64" else g.to(torch.float32)}
    r = adjoint.gradients(w, state["prm"], n, state["target"], u0=state["u0"], precision=prec,
                          wrt_a=case["mode"] != "source", tape=case["mode"] == "tape")
    keys = ("dA_re", "dA_im", "dr0") + (() if case["mode"] == "source" else ("da",))
    h = r["h"] if prec == "fp64" else r["h"].to(torch.complex64)
    real = np.float64 if prec == "fp64" else np.float32
    return {"h": h, "du0": r["du0"], **{k: real(r[k]) for k in keys}}


def work(case):
    """Initial data in and state out, once each; 140 operations a point and
    step for the forward step, 250 more for its adjoint with the spin term
    (140 without it)."""
    cb = 8 if case["prec"] == "fp32" else 16
    pts = sum(w.Nr * w.Ntheta for w in _instances(case))
    n = case["steps"]
    per = 140.0
    if case["kind"] == "gradient":
        per += 140.0 if case["mode"] == "source" else 250.0
    return {"bytes": 2.0 * pts * (16 + cb) + 16.0 * n, "flops": per * pts * n}


# ------------------------------------------------------------------- exact
# The same scheme in 64 bits with plain torch operations: theta runs along
# the first axis, so a tridiagonal solve is a loop over theta of operations
# on whole r* rows.

def _thomas(lo, di, up, r):
    """x with lo_j x_{j-1} + di_j x_j + up_j x_{j+1} = r_j along axis 0."""
    N = r.shape[0]
    c, z = [None] * N, [None] * N
    den = di[0]
    for j in range(N):
        if j:
            den = torch.addcmul(di[j], lo[j], c[j - 1], value=-1)
        c[j] = up[j] / den
        z[j] = (r[j] if not j else torch.addcmul(r[j], lo[j], z[j - 1], value=-1)) / den
    for j in range(N - 2, -1, -1):
        z[j] = torch.addcmul(z[j], c[j], z[j + 1], value=-1)
    return torch.stack(z)


def _below(x):
    return torch.cat([torch.zeros_like(x[:1]), x[:-1]])


def _above(x):
    return torch.cat([x[1:], torch.zeros_like(x[:1])])


class _Solve(torch.autograd.Function):
    @staticmethod
    def forward(ctx, lo, di, up, r):
        x = _thomas(lo, di, up, r)
        ctx.save_for_backward(lo, di, up, x)
        return x

    @staticmethod
    def backward(ctx, gx):
        lo, di, up, x = ctx.saved_tensors
        gr = _thomas(_below(up).conj(), di.conj(), _above(lo).conj(), gx)
        return -gr * _below(x).conj(), -gr * x.conj(), -gr * _above(x).conj(), gr


class _Exact:
    """Coefficients of one instance (a and r0: 0-dim tensors, for gradients)."""

    def __init__(self, w, amp, a, r0):
        dev, f8 = "cuda", torch.float64
        self.w, self.amp = w, amp
        s, m, Nr, N = float(w.s), float(w.m), w.Nr, w.Ntheta
        self.drs = (w.rs_max - w.rs_min) / (Nr - 1)
        self.dt = w.cfl * self.drs
        root = torch.sqrt(1.0 - a * a)
        rp, gap = 1.0 + root, 2.0 * root
        rm = 1.0 - root

        def rstar(x):
            return rp + x + 2.0 * rp / gap * torch.log(x / 2.0) - 2.0 * rm / gap * torch.log((x + gap) / 2.0)

        rs = w.rs_min + 0.5 * self.drs * torch.arange(2 * Nr - 1, dtype=f8, device=dev)
        # r(r*): Newton on xi = ln(r - r_+), inside a bracket
        with torch.no_grad():
            lo, hi = torch.full_like(rs, -700.0), torch.full_like(rs, 60.0)
            xi = torch.where(rs > rp + 4.0, torch.log(rs.clamp(min=1.0)), (rs - rp) * gap / (2.0 * rp))
            for _ in range(60):
                x = torch.exp(xi)
                f = rstar(x) - rs
                hi, lo = torch.where(f > 0, xi, hi), torch.where(f > 0, lo, xi)
                nxt = xi - f * (x + gap) / ((rp + x) ** 2 + a * a)
                xi = torch.where((nxt > lo) & (nxt < hi), nxt, torch.where(f.abs() < 1e-12, xi, 0.5 * (lo + hi)))
        x = torch.exp(xi)
        # one more step, differentiable in a (r(r*; a) by implicit differentiation)
        slope = ((rp + x) ** 2 + a * a) / (x + gap)
        x = torch.exp(xi - (rstar(x) - rs) / slope.detach())
        r, D = rp + x, x * (x + gap)
        R = r * r + a * a
        th = ((torch.arange(N, dtype=f8, device=dev) + 0.5) * (math.pi / N))[:, None]
        sn, cs = torch.sin(th), torch.cos(th)
        sig2 = R * R - a * a * D * sn * sn
        sig = torch.sqrt(sig2)
        h = D / R
        self.b = R / sig
        b_rs = h * (2.0 * r / sig - R * (4.0 * R * r - 2.0 * a * a * sn * sn * (r - 1.0)) / (2.0 * sig * sig2))
        ct = torch.complex(2.0 * s * (r * D - (r * r - a * a)) / sig2, (4.0 * a * m * r + 2.0 * s * a * D * cs) / sig2)
        qP = torch.complex((2.0 * r * D + 2.0 * s * (r - 1.0) * R) / sig2, 2.0 * a * m * R / sig2)
        cstar = -self.b ** 2 * 6.0 * h / r - qP
        d3 = h * (6.0 * r * D / R + 6.0 * r * r * (r - 1.0) / R - 6.0 * r ** 3 * D / (R * R))
        c0 = -self.b ** 2 * d3 / r ** 3 - 3.0 * h / r * qP - 1j * (4.0 * s * m * a * (r - 1.0) / sig2)
        self.K = self.b * ct - cstar - self.b * b_rs
        # angular operator with the parity ghosts folded into its diagonal
        d, cot, par = math.pi / N, cs / sn, 1.0 if w.m % 2 == 0 else -1.0
        al, au = -(1.0 - 0.5 * cot * d) / d ** 2, -(1.0 + 0.5 * cot * d) / d ** 2
        a0 = 2.0 / d ** 2 + (m + s * cs) ** 2 / sn ** 2 - s
        a0[0] += par * al[0]
        a0[-1] += par * au[-1]
        al[0] = 0.0
        au[-1] = 0.0
        q = (D / sig2)[:, ::2]
        self.ct, self.wl, self.wu = ct[:, ::2], q * al, q * au
        self.wd = q * a0 + c0[:, ::2]
        # source: prefactor, Gaussian and phase (Eq. 1 after the division that gives Eq. 9)
        self.Om = 1.0 / (r0 ** 1.5 + a)
        rs0 = rstar(r0 - rp)
        self.F = 4.0 * math.pi * (r * r + (a * cs) ** 2) * D / (sig2 * r ** 3) * torch.exp(
            -(rs - rs0) ** 2 / (2.0 * w.sig_r ** 2) - (th - 0.5 * math.pi) ** 2 / (2.0 * w.sig_th ** 2))
        self.inner = torch.ones(Nr, dtype=f8, device=dev)
        self.inner[0] = self.inner[-1] = 0.0
        Y = torch.sin(0.5 * th) ** abs(w.m + w.s) * torch.cos(0.5 * th) ** abs(w.m - w.s)
        self.wt = ((sn * Y) / (sn * Y * Y).sum())[:, 0].to(torch.complex128)
        self.ie = min(Nr - 1, max(0, round((w.rs_ext - w.rs_min) / self.drs)))

    def implicit(self, u, h, cols=slice(None)):
        """The two-stage SDIRK2 step of length h of the algebraic terms."""
        wl, wd, wu, ct, inner = (t[..., cols] for t in (self.wl, self.wd, self.wu, self.ct, self.inner))
        gh = GAMMA * h

        def W(x):
            return wl * _below(x) + wd * x + wu * _above(x)

        lo, di, up = gh * gh * wl, 1.0 + gh * ct + gh * gh * wd, gh * gh * wu
        lo, up = lo.to(di.dtype), up.to(di.dtype)
        f, g = u
        g1 = _Solve.apply(lo, di, up, g - gh * W(f))
        f1 = f + gh * g1
        f2, g2 = f + (1.0 - GAMMA) * h * g1, g - (1.0 - GAMMA) * h * (W(f1) + ct * g1)
        g2 = _Solve.apply(lo, di, up, g2 - gh * W(f2))
        return (f2 + gh * g2) * inner, g2 * inner

    def source(self, t):
        ph = float(self.w.m) * self.Om * t
        return torch.complex(torch.cos(ph), -torch.sin(ph)) * self.amp

    def transport(self, u, n):
        f, g = u
        k, t = self.dt / self.drs, n * self.dt
        b, K, F = self.b, self.K, self.F
        df, dg = f[:, 1:] - f[:, :-1], g[:, 1:] - g[:, :-1]
        mf = 0.5 * (f[:, 1:] + f[:, :-1]) - 0.5 * k * b[:, 1::2] * df
        mg = (0.5 * (g[:, 1:] + g[:, :-1]) + 0.5 * k * (b[:, 1::2] * dg + K[:, 1::2] * df)
              + 0.5 * self.dt * F[:, 1::2] * self.source(t))
        df, dg = mf[:, 1:] - mf[:, :-1], mg[:, 1:] - mg[:, :-1]
        b, K, F = b[:, 2:-1:2], K[:, 2:-1:2], F[:, 2:-1:2]
        nf = f[:, 1:-1] - k * b * df
        ng = g[:, 1:-1] + k * (b * dg + K * df) + self.dt * F * self.source(t + 0.5 * self.dt)
        return torch.nn.functional.pad(nf, (1, 1)), torch.nn.functional.pad(ng, (1, 1))

    def run(self, u0, n):
        """u0: (2, Nr, Ntheta) -> the state after n steps (before the closing
        half implicit step, as the stepper holds it) and the n + 1 samples."""
        u = (u0[0].T.contiguous(), u0[1].T.contiguous())
        c = slice(self.ie, self.ie + 1)
        h = [(self.wt * u[0][:, self.ie]).sum()]
        for k in range(n):
            # (recomputed in a backward pass, which otherwise holds some 60 planes a step)
            u = checkpoint(lambda f, g, k=k: self.transport(self.implicit((f, g), self.dt if k else 0.5 * self.dt), k), *u,
                           use_reentrant=False) if torch.is_grad_enabled() else self.transport(
                               self.implicit(u, self.dt if k else 0.5 * self.dt), k)
            x = self.implicit((u[0][:, c], u[1][:, c]), 0.5 * self.dt, c)[0] if 0 < self.ie < self.w.Nr - 1 else 0.0 * u[0][:, c]
            h.append((self.wt * x[:, 0]).sum())
        return torch.stack((u[0].T, u[1].T)), torch.stack(h)


def exact(case, seed):
    n = case["steps"]
    if case["kind"] != "gradient":
        # the sequential solves of every instance: 20 seconds' worth at most
        if sum(w.Ntheta * n for w in _instances(case)) > 150000:
            return None
        out = []
        with torch.no_grad():
            for k, w in enumerate(_instances(case)):
                a, r0 = (torch.tensor(v, dtype=torch.float64, device="cuda") for v in (w.a, w.r0))
                out.append(_Exact(w, _amplitude(seed + k), a, r0).run(_initial(w, seed + k), n))
        return out
    if case["Nth"] * n > 26000:
        return None
    st = prepare(case, seed)
    w = st["w"]
    p = st["params"].clone().requires_grad_(True)
    u0 = torch.zeros(2, w.Nr, w.Ntheta, dtype=torch.complex128, device="cuda") if st["u0"] is None else st["u0"]
    u0 = u0.clone().requires_grad_(True)
    _, h = _Exact(w, torch.complex(p[0], p[1]), p[3], p[2]).run(u0, n)
    if case["mode"] == "autograd":
        d = h - st["target"]
        (d.real ** 2 + d.imag ** 2).sum().backward()
        return {"h": h.detach(), "grad": p.grad}
    (h.real * st["target"].real + h.imag * st["target"].imag).sum().backward()
    keys = ("dA_re", "dA_im", "dr0") + (() if case["mode"] == "source" else ("da",))
    return {"h": h.detach(), "du0": u0.grad, **{k: p.grad[i].clone() for i, k in enumerate(keys)}}
