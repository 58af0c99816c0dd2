"""The calls a program of this framework makes, at the sizes it makes them: what its speed is
judged by.  Each case is one public entry point on one synthetic model (the seed sets the random
matrices, or for the dimer its drive and interaction):

  goe_build     U_T of a dense random-matrix model (the paper's benchmark model), per precision
  dimer_build   U_T of a Bose-Hubbard dimer (tridiagonal), per precision
  resume        a block of states taken through some of the steps of a period (resuming a chain)
  average       period averages <H(t)>_T of given states (the second propagation round)
  grad          gate-fidelity loss and its gradient in the M piecewise drive amplitudes
  scan          a parameter scan: many dense models of uneven size as one graph launch
  defect        unitarity defect of a finished U_T over sampled columns

Sizes follow the repository's own workloads (GOE N = 64, M = 200; the dimer with M = 2000 steps
per period; GOE N = 4096, M = 512; scans over N = 256..2048 with M = 256; gradients at N = 1024,
M = 256 with checkpoints every 16 steps).  Where a whole period would take seconds, the case runs
the workload's own step length over the first part of the period.
"""
import math

import numpy as np
import torch

import paper_1508_07621_gb300 as fq

PRECISION = {"fp64": fq.FQ_FP64, "fp32": fq.FQ_FP32, "x3": fq.FQ_BF16X3, "x6": fq.FQ_BF16X6, "df32": fq.FQ_DF32,
             "ozaki": fq.FQ_OZAKI}


def listed():
    return [
        # the smallest workload of the repository, where launches and latency count
        _goe("goe64_fp64", 64, 200, "fp64", h=2 * math.pi / 200, amp=1.0, omega=1.0),
        # an ordinary dense build at FP32 level, of a size that is no multiple of a tile
        _goe("goe1000_x3", 1000, 64, "x3", h=2 * math.pi / (2.0 * 512), amp=2.0, omega=2.0),
        # the large dense workload (N = 4096, M = 512), its first 48 steps
        _goe("goe4096_x3", 4096, 48, "x3", h=2 * math.pi / (2.0 * 512), amp=2.0, omega=2.0),
        # a dense build at FP64 level on the tensor cores, ragged
        _goe("goe777_ozaki", 777, 32, "ozaki", h=2 * math.pi / (2.0 * 512), amp=2.0, omega=2.0),
        # the dimer at FP32 level (the default precision), a whole period
        _dimer("dimer1301_fp32", 1300, 2000, 2000, "fp32"),
        # the benchmark dimer's FP64-level kernel, its own step length, a tenth of the period
        _dimer("dimer4001_ozaki", 4000, 2000, 200, "ozaki"),
        # states of a middle-sized dimer resumed in plain FP64
        {"name": "resume501_fp64", "kind": "resume", "nb": 500, "period_steps": 500, "m_begin": 100, "m_end": 260,
         "ncols": 48, "precision": "fp64"},
        # second propagation round over every Floquet state of a dense model
        {"name": "average256_goe", "kind": "average", "model": "goe", "n": 256, "steps": 16, "ncols": 256,
         "h": 2 * math.pi / 200, "amp": 1.0, "omega": 1.0, "precision": "x6"},
        # and of a dimer, with an odd number of steps (trapezoid rule)
        {"name": "average901_dimer", "kind": "average", "model": "dimer", "nb": 900, "period_steps": 2000,
         "steps": 125, "ncols": 901, "precision": "fp32"},
        # gradient workload (N = 1024, checkpoints every 16 steps), an eighth of its period
        {"name": "grad1024_x3", "kind": "grad", "n": 1024, "steps": 32, "h": 2 * math.pi / 256, "precision": "x3",
         "stride": 16},
        # eight instances of the scan workload's recipe as one launch
        {"name": "scan8_x3", "kind": "scan", "count": 8, "n_lo": 256, "n_hi": 1280, "steps": 24, "steps_period": 256,
         "precision": "x3"},
        # the check that follows a large build: 64 columns of U_T
        {"name": "defect4096", "kind": "defect", "n": 4096, "cols": 64},
    ]


def _goe(name, n, steps, precision, h, amp, omega):
    return {"name": name, "kind": "goe_build", "n": n, "steps": steps, "precision": precision, "h": h, "amp": amp,
            "omega": omega}


def _dimer(name, nb, period_steps, steps, precision):
    return {"name": name, "kind": "dimer_build", "nb": nb, "period_steps": period_steps, "steps": steps,
            "precision": precision}


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["goe_build", "goe_build", "dimer_build", "dimer_build", "resume", "average", "grad", "scan",
                       "defect"])
    drive = {"h": 2 * math.pi / rng.choice([200, 400, 1024]), "amp": rng.uniform(0.5, 2.0),
             "omega": rng.uniform(0.5, 4.0)}
    if kind == "goe_build":
        precision = rng.choice(["fp64", "df32", "x3", "x3", "x6", "ozaki"])
        lo, hi = {"fp64": (12, 300), "df32": (12, 128), "x3": (150, 2600), "x6": (150, 2000),
                  "ozaki": (150, 1300)}[precision]
        return {"kind": kind, "n": _log(rng, lo, hi), "steps": rng.randint(20, 48), "precision": precision, **drive}
    if kind == "dimer_build":
        precision = rng.choice(["fp32", "fp32", "ozaki", "ozaki", "df32", "fp64"])
        hi = {"fp32": 6000, "ozaki": 4000, "df32": 1500, "fp64": 800}[precision]
        nb = _log(rng, 30, hi)
        return {"kind": kind, "nb": nb, "period_steps": 2000, "steps": rng.randint(50, 180), "precision": precision}
    if kind == "resume":
        precision = rng.choice(["fp64", "fp32", "df32", "ozaki"])
        m0 = rng.randint(0, 200)
        return {"kind": kind, "nb": _log(rng, 40, 3000), "period_steps": 2000, "m_begin": m0,
                "m_end": m0 + rng.randint(40, 160), "ncols": _log(rng, 1, 160), "precision": precision}
    if kind == "average":
        if rng.random() < 0.5:
            n = _log(rng, 24, 400)
            precision = rng.choice(["fp64", "x6"]) if n <= 200 else rng.choice(["x6", "ozaki"])
            return {"kind": kind, "model": "goe", "n": n, "steps": rng.randint(6, 16), "ncols": _log(rng, 1, n),
                    "precision": precision, **drive}
        nb = _log(rng, 40, 1500)
        return {"kind": kind, "model": "dimer", "nb": nb, "period_steps": 2000, "steps": rng.randint(30, 130),
                "ncols": _log(rng, 1, nb), "precision": rng.choice(["fp32", "fp32", "ozaki"])}
    if kind == "grad":
        return {"kind": kind, "n": _log(rng, 64, 1024), "steps": rng.randint(10, 32), "h": 2 * math.pi / 256,
                "precision": rng.choice(["x3", "x3", "x6", "ozaki"]), "stride": rng.choice([8, 16])}
    if kind == "scan":
        lo = rng.randint(150, 500)
        return {"kind": kind, "count": rng.randint(3, 8), "n_lo": lo, "n_hi": _log(rng, lo + 1, 1300),
                "steps": rng.randint(8, 24), "steps_period": 256, "precision": rng.choice(["x3", "x3", "x6"])}
    n = _log(rng, 200, 4096)
    return {"kind": "defect", "n": n, "cols": _log(rng, 1, min(n, 128))}


# ------------------------------------------------------------------------------- models
def _random_goe(n, rng):
    g = rng.standard_normal((n, n))
    return (g + g.T) / math.sqrt(2.0 * n)


def _dimer_model(case, seed):
    """J = 1, U nb = 2, f = eps1 cos 3t as the repository's dimer, eps1 and U moved a few per cent by the seed."""
    nb = case["nb"]
    rng = np.random.default_rng(seed)
    u = 2.0 / nb * rng.uniform(0.95, 1.05)
    n = np.arange(nb + 1, dtype=np.float64)
    m = nb - n
    k = n[:-1]
    diag = 0.5 * u * (n * (n - 1.0) + m * (m - 1.0))
    off = -np.sqrt((k + 1.0) * (nb - k))
    return diag, off, n - 0.5 * nb, {"omega": 3.0, "f_ac": 1.5 * rng.uniform(0.95, 1.05)}


def _dimer_plan(case, seed, steps):
    diag, off, h1, drive = _dimer_model(case, seed)
    h = 2 * math.pi / 3.0 / case["period_steps"]
    return fq.Plan.tridiag(diag, off, h1, steps=steps, period=steps * h, precision=PRECISION[case["precision"]],
                           **drive)


def _goe_model(case, seed):
    rng = np.random.default_rng(seed)
    return _random_goe(case["n"], rng), _random_goe(case["n"], rng)


def _goe_plan(case, seed):
    h0, h1 = _goe_model(case, seed)
    return fq.Plan.dense(h0, h1, omega=case["omega"], f_ac=case["amp"], steps=case["steps"],
                         period=case["steps"] * case["h"], precision=PRECISION[case["precision"]])


def _scan_models(case, seed):
    """The scan workload's recipe: N uniform in its range, omega in [0.5, 4], amplitude in [0.5, 3]."""
    rng = np.random.default_rng(seed)
    sizes = np.random.default_rng(case["count"] * 10007 + case["n_hi"])  # the work is the case's, not the seed's
    out = []
    for _ in range(case["count"]):
        n = int(sizes.integers(case["n_lo"], case["n_hi"] + 1))
        omega, amp = float(sizes.uniform(0.5, 4.0)), float(sizes.uniform(0.5, 3.0))
        out.append((n, omega, amp, _random_goe(n, rng), _random_goe(n, rng)))
    return out


def _states(n, ncols, seed):
    """Unit states with random complex entries (rows), as the eigenvectors of a U_T are."""
    g = torch.Generator(device="cuda").manual_seed(seed + 101)
    x = torch.randn(ncols, n, 2, dtype=torch.float64, device="cuda", generator=g)
    x = torch.view_as_complex(x)
    return (x / torch.linalg.vector_norm(x, dim=1, keepdim=True)).contiguous()


def _unitary(n, seed):
    """A dense unitary without structure (random phases between Fourier transforms)."""
    g = torch.Generator(device="cuda").manual_seed(seed + 211)

    def phases():
        t = 2 * math.pi * torch.rand(n, dtype=torch.float64, device="cuda", generator=g)
        return torch.polar(torch.ones_like(t), t)

    u = torch.diag(phases())
    for _ in range(2):
        u = torch.fft.fft(u, dim=0, norm="ortho") * phases()[:, None]
    return u.contiguous()


class _Scan:
    """Plans, outputs, workspace and graph of a batched scan; the graph goes before the plans."""

    def __init__(self, plans):
        self.plans = plans
        self.outs = [torch.empty((p.n, p.n), dtype=torch.complex128, device="cuda") for p in plans]
        handles = [p.handle for p in plans]
        self.ws = fq.workspace(fq.floquet_batch_workspace_size(handles))
        self.batch = fq.floquet_batch_create(handles, self.outs, self.ws, 0)

    def __del__(self):
        if getattr(self, "batch", None):
            fq.floquet_batch_destroy(self.batch)
            self.batch = None


# ------------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    if kind == "goe_build":
        plan = _goe_plan(case, seed)
        ws = fq.workspace(plan.workspace_size())
        return {"kind": kind, "plan": plan, "ws": ws,
                "out": torch.empty((plan.n, plan.n), dtype=torch.complex128, device="cuda")}
    if kind == "dimer_build":
        plan = _dimer_plan(case, seed, case["steps"])
        return {"kind": kind, "plan": plan, "ws": fq.workspace(plan.workspace_size()),
                "out": torch.empty((plan.n, plan.n), dtype=torch.complex128, device="cuda")}
    if kind == "resume":
        plan = _dimer_plan(case, seed, case["period_steps"])
        x0 = _states(plan.n, case["ncols"], seed)
        return {"kind": kind, "plan": plan, "x0": x0, "out": torch.empty_like(x0), "m": (case["m_begin"], case["m_end"]),
                "ws": fq.workspace(plan.workspace_size(case["ncols"]))}
    if kind == "average":
        plan = _goe_plan(case, seed) if case["model"] == "goe" else _dimer_plan(case, seed, case["steps"])
        return {"kind": kind, "plan": plan, "x0": _states(plan.n, case["ncols"], seed)}
    if kind == "grad":
        h0, h1 = _goe_model(case, seed)
        f = 1.0 + 0.1 * np.random.default_rng(seed + 7).standard_normal(case["steps"])
        plan = fq.Plan.piecewise(h0, h1, f, period=case["steps"] * case["h"], precision=PRECISION[case["precision"]],
                                 checkpoint_stride=case["stride"], tile_n=64)
        return {"kind": kind, "plan": plan, "f": torch.from_numpy(f).cuda(), "W": _unitary(case["n"], seed),
                "ws": fq.workspace(fq.floquet_grad_workspace_size(plan.handle))}
    if kind == "scan":
        plans = [fq.Plan.dense(h0, h1, omega=omega, f_ac=amp, steps=case["steps"],
                               period=case["steps"] * 2 * math.pi / omega / case["steps_period"],
                               precision=PRECISION[case["precision"]])
                 for _, omega, amp, h0, h1 in _scan_models(case, seed)]
        return {"kind": kind, "scan": _Scan(plans)}
    n, k = case["n"], case["cols"]
    # a U_T as far from unitary as the FP32-level paths leave it after a whole period
    g = torch.Generator(device="cuda").manual_seed(seed + 307)
    noise = torch.randn(n, n, 2, dtype=torch.float64, device="cuda", generator=g)
    u = _unitary(n, seed) + (3e-6 / math.sqrt(n)) * torch.view_as_complex(noise)
    cols = (torch.arange(k, dtype=torch.int64) * n // k).to(torch.int32).cuda()
    return {"kind": "defect", "U": u, "cols": cols}


def run(state):
    kind = state["kind"]
    if kind in ("goe_build", "dimer_build"):
        return state["plan"].build_UT(state["out"], state["ws"])
    if kind == "resume":
        return state["plan"].propagate(state["x0"], *state["m"], out=state["out"], ws=state["ws"])
    if kind == "average":
        return state["plan"].average_observable(state["x0"])
    if kind == "grad":
        return state["plan"].grad(state["f"], state["W"], ws=state["ws"])
    if kind == "scan":
        fq.floquet_batch_launch(state["scan"].batch)
        return state["scan"].outs
    return fq.unitarity_defect(state["U"], state["cols"])


# ------------------------------------------------------------------------------- work
def _bessel(r, kmax):
    """J_0 .. J_kmax at r from the integral (1/pi) int_0^pi cos(k t - r sin t) dt: the midpoint rule
    converges beyond every power here, the integrand being smooth and periodic."""
    q = 2 * (kmax + 40 + int(2 * r))
    t = (np.arange(q) + 0.5) * (2 * math.pi / q)
    k = np.arange(kmax + 1)[:, None]
    return np.cos(k * t[None, :] - r * np.sin(t)[None, :]).mean(axis=1)


def _terms(r):
    """Chebyshev products a step of spectral half width r cannot do without (tail below 1e-14)."""
    j = np.abs(_bessel(r, int(r) + 80))
    l = int(math.floor(r)) + 1
    while j[l + 1] >= 1e-14:
        l += 1
    return l


def _chain(case):
    """(states' length, states, steps, products a step, flops of one product on one state, operator bytes)."""
    kind = case["kind"]
    tri = "nb" in case
    if tri:
        n = case["nb"] + 1
        h = 2 * math.pi / 3.0 / case["period_steps"]
        # spectral half width of the dimer: about 1.33 nb (J = 1, U nb = 2, eps1 = 1.5)
        length, op, flops = _terms(h * 1.33 * n), 32.0 * n, 26.0 * n
    else:
        n = case["n"]
        amp = case.get("amp", 1.3)  # gradients: |f| up to about 1.3
        length, op, flops = _terms(case["h"] * 2.0 * (1.0 + amp)), 24.0 * n * n, 8.0 * n * n
    steps = case["m_end"] - case["m_begin"] if kind == "resume" else case["steps"]
    return n, case.get("ncols", n), steps, length, flops, op


def work(case):
    kind = case["kind"]
    if kind == "defect":
        return {"bytes": 16.0 * case["n"] ** 2, "flops": 8.0 * case["n"] ** 2 * case["cols"]}
    if kind == "scan":
        flops = bytes_ = 0.0
        sizes = np.random.default_rng(case["count"] * 10007 + case["n_hi"])
        for _ in range(case["count"]):
            n = int(sizes.integers(case["n_lo"], case["n_hi"] + 1))
            omega, amp = float(sizes.uniform(0.5, 4.0)), float(sizes.uniform(0.5, 3.0))
            length = _terms(2 * math.pi / omega / case["steps_period"] * 2.0 * (1.0 + amp))
            flops += 8.0 * n ** 3 * length * case["steps"]
            bytes_ += 40.0 * n * n
        return {"bytes": bytes_, "flops": flops}
    n, ncols, steps, length, per_state, op = _chain(case)
    chain = per_state * ncols * length * steps
    if kind == "grad":  # real operators; forward products, adjoint products and gradient dots
        return {"bytes": 32.0 * n * n + 16.0 * steps, "flops": 3.0 * 0.5 * chain}
    if kind == "average":
        dot = (4.0 * n if "n" in case else 14.0) * n * ncols * (steps + 1)
        return {"bytes": op + 16.0 * n * ncols + 8.0 * ncols, "flops": chain + dot}
    if kind == "resume":
        return {"bytes": op + 32.0 * n * ncols, "flops": chain}
    return {"bytes": op + 16.0 * n * n, "flops": chain}


# ------------------------------------------------------------------------------- tolerance
# About four times the largest distance from the exact result seen over the listed and some eighty
# drawn cases, per precision; gradients carry the relative error of tau = Tr(W^+ U_T) besides.
REL = {"fp64": 4e-12, "df32": 6e-12, "ozaki": 3e-11, "x6": 5e-5, "x3": 2e-5, "fp32": 2e-4}
REL_GRAD = {"ozaki": 2e-10, "x6": 8e-5, "x3": 8e-5}


def tolerance(case):
    if case["kind"] == "defect":
        return {"rel": 1e-8}
    return {"rel": (REL_GRAD if case["kind"] == "grad" else REL)[case["precision"]]}


# ------------------------------------------------------------------------------- exact results
def _drive(amp, omega, t):
    return amp * math.cos(omega * t), -amp * omega * math.sin(omega * t), -amp * omega * omega * math.cos(omega * t)


def _step_scalars(h, m, amp, omega):
    f, f1, f2 = _drive(amp, omega, (m + 0.5) * h)
    return h, h * f + h ** 3 * f2 / 24.0, h ** 3 * f1 / 12.0


def _chebyshev(apply, x, r, centre):
    """exp(-i Omega) x for Omega with spectrum within centre +- r, apply(x) = Omega x."""
    length = int(r + 30 + 6 * r ** (1 / 3))
    a = 2.0 * _bessel(r, length)
    prev, cur = x, (-1j / r) * (apply(x) - centre * x)
    acc = 0.5 * a[0] * x + a[1] * cur
    for k in range(2, length + 1):
        if abs(a[k]) < 1e-18 and k > r:
            break
        prev, cur = cur, prev + (-2j / r) * (apply(cur) - centre * cur)
        acc = acc + a[k] * cur
    return acc * complex(math.cos(centre), -math.sin(centre))


def _dense_steps(h0, h1, h, m0, m1, amp, omega, x):
    """States (columns of x) after each step m0 .. m1 - 1 of the dense chain."""
    k = h0 @ h1 - h1 @ h0
    n0, n1 = (float(torch.linalg.eigvalsh(q).abs().max()) for q in (h0, h1))
    kn = 2.0 * n0 * n1
    for m in range(m0, m1):
        a, b, c = _step_scalars(h, m, amp, omega)
        om = torch.complex(a * h0 + b * h1, c * k)
        r = 1.001 * (a * n0 + abs(b) * n1 + abs(c) * kn) + 1e-9
        x = _chebyshev(lambda v: om @ v, x, r, 0.0)
        yield x


def _tri_steps(diag, off, h1, h, m0, m1, amp, omega, x):
    """The same for the tridiagonal chain (H1 diagonal, [H0, H1] off-diagonal)."""
    diag, off, h1 = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (diag, off, h1))
    ko = off * (h1[:-1] - h1[1:])  # [H0, H1][i + 1, i]
    pad = torch.zeros(1, dtype=torch.complex128, device="cuda")
    for m in range(m0, m1):
        a, b, c = _step_scalars(h, m, amp, omega)
        d = a * diag + b * h1
        e = torch.complex(a * off, c * ko)
        rad = torch.cat([e, pad]).abs() + torch.cat([pad, e]).abs()
        lo, hi = float((d - rad).min()), float((d + rad).max())
        lower, upper = e[:, None], e.conj()[:, None]
        dc = d[:, None]

        def apply(v):
            y = dc * v
            y[1:] += lower * v[:-1]
            y[:-1] += upper * v[1:]
            return y

        x = _chebyshev(apply, x, 0.5 * (hi - lo) + 1e-9, 0.5 * (hi + lo))
        yield x


def _last(steps, x):
    for x in steps:
        pass
    return x


def _eye(n):
    return torch.eye(n, dtype=torch.complex128, device="cuda")


def _goe_exact(n, steps, h, amp, omega, h0, h1, x=None):
    h0, h1 = torch.from_numpy(h0).cuda(), torch.from_numpy(h1).cuda()
    return _dense_steps(h0, h1, h, 0, steps, amp, omega, _eye(n) if x is None else x)


def exact(case, seed):
    kind = case["kind"]
    if kind == "defect":
        st = prepare(case, seed)
        u, cols = st["U"], st["cols"].long()
        d = u[:, cols].conj().T @ u
        d[torch.arange(len(cols)), cols] -= 1.0
        return float(d.abs().max()), float(torch.linalg.vector_norm(d) / math.sqrt(len(cols)))
    # FP64 products and FP64 vector passes of the plain chain run at about 1e12 flops and 3e12 bytes a second here
    if kind == "scan":
        if 2.5 * work(case)["flops"] > 1.5e13:
            return None
        out = []
        for n, omega, amp, h0, h1 in _scan_models(case, seed):
            h = 2 * math.pi / omega / case["steps_period"]
            out.append(_last(_goe_exact(n, case["steps"], h, amp, omega, h0, h1), None))
        return out
    n, ncols, steps, length, _, _ = _chain(case)
    if "nb" in case:
        if 2.0 * length * steps * (6e-4 + 250.0 * n * ncols / 3e12) > 18.0:
            return None
    elif 2.5 * work(case)["flops"] > 1.5e13:
        return None
    if kind == "grad":
        return _grad_exact(case, seed)
    if "nb" in case:
        diag, off, h1, drive = _dimer_model(case, seed)
        h = 2 * math.pi / 3.0 / case["period_steps"]
        m0, m1 = (case["m_begin"], case["m_end"]) if kind == "resume" else (0, case["steps"])
        x = _eye(n) if kind == "dimer_build" else _states(n, ncols, seed).T.contiguous()
        chain = _tri_steps(diag, off, h1, h, m0, m1, drive["f_ac"], drive["omega"], x)
        if kind == "average":
            d, o, q = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (diag, off, h1))

            def energy(v, f):
                y = (d + f * q)[:, None] * v
                y[1:] += o[:, None] * v[:-1]
                y[:-1] += o[:, None] * v[1:]
                return (v.conj() * y).sum(dim=0).real

            return _average_exact(chain, x, energy, steps, h, drive["f_ac"], drive["omega"])
        x = _last(chain, x)
        return x.T.contiguous() if kind == "resume" else x
    h0, h1 = _goe_model(case, seed)
    if kind == "goe_build":
        return _last(_goe_exact(n, steps, case["h"], case["amp"], case["omega"], h0, h1), None)
    x = _states(n, ncols, seed).T.contiguous()
    chain = _goe_exact(n, steps, case["h"], case["amp"], case["omega"], h0, h1, x)
    g0, g1 = (torch.from_numpy(q).cuda().to(torch.complex128) for q in (h0, h1))
    return _average_exact(chain, x, lambda v, f: (v.conj() * ((g0 + f * g1) @ v)).sum(dim=0).real, steps, case["h"],
                          case["amp"], case["omega"])


def _average_exact(chain, x, energy, steps, h, amp, omega):
    """(1/T) times the composite Simpson sum (trapezoid for an odd number of steps) of <H(t)>."""
    w = np.full(steps + 1, 1.0)
    if steps % 2 == 0:
        w[1:-1:2], w[2:-1:2], w[0], w[-1] = 4.0 / 3.0, 2.0 / 3.0, 1.0 / 3.0, 1.0 / 3.0
    else:
        w[0] = w[-1] = 0.5
    acc = w[0] * energy(x, _drive(amp, omega, 0.0)[0])
    for m, x in enumerate(chain):
        acc = acc + w[m + 1] * energy(x, _drive(amp, omega, (m + 1) * h)[0])
    return acc / steps


def _grad_exact(case, seed):
    """Loss 1 - |Tr(W^+ U)|^2 / N^2 and its gradient from the eigenvectors of every step's H0 + f_m H1:
    d exp(-i h H) / df in that basis is -i h (V^T H1 V)_ab e^{-i h (x_a + x_b) / 2} sinc(h (x_a - x_b) / 2)."""
    st = prepare(case, seed)
    h0, h1 = (torch.from_numpy(q).cuda() for q in _goe_model(case, seed))
    f, w, n, h = st["f"].tolist(), st["W"], case["n"], case["h"]
    eig = [torch.linalg.eigh(h0 + fm * h1) for fm in f]
    vecs = [v.to(torch.complex128) for _, v in eig]
    phases = [torch.polar(torch.ones_like(x), -h * x) for x, _ in eig]

    def step(m, x):
        return vecs[m] @ (phases[m][:, None] * (vecs[m].T @ x))

    xs = [_eye(n)]
    for m in range(len(f)):
        xs.append(step(m, xs[-1]))
    tau = (w.conj() * xs[-1]).sum()
    loss = 1.0 - float(tau.abs()) ** 2 / n ** 2
    left = w.clone()  # (U_M .. U_{m+1})^+ W
    grad = np.zeros(len(f))
    for m in reversed(range(len(f))):
        x, v = eig[m]
        mean, half = 0.5 * h * (x[:, None] + x[None, :]), 0.5 * h * (x[:, None] - x[None, :])
        phi = -1j * h * torch.polar(torch.sinc(half / math.pi), -mean)
        kern = phi * (v.T @ h1 @ v)
        dtau = ((vecs[m].T @ left).conj() * (kern @ (vecs[m].T @ xs[m]))).sum()
        grad[m] = -2.0 * float((tau.conj() * dtau).real) / n ** 2
        left = vecs[m] @ (phases[m].conj()[:, None] * (vecs[m].T @ left))
    return torch.tensor([loss], dtype=torch.float64), torch.from_numpy(grad)
