"""What the performance of this framework is measured on.

Every case is a call, or a short sequence of calls, that a program using the
framework makes: whole Wiener-filter solves, runs of the iteration with the
fields and the residual read back, a batch of uneven maps, the transforms on
their own, and the warm-start network's inference and training gradient.

A case is a dict of plain values; `listed` gives the fixed ones, `draw` more of
the same ranges.  `prepare` makes the inputs on the GPU from the seed and the
plan (or batch, or network) that a program keeps; `run` is one pass; `work` the
bytes and operations of a pass; `exact` the same outputs in 64 bits, in plain
torch.
"""

from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1704_00865_gb300 import wf

# the map sides the library takes
SIDES = (32, 64, 128, 256, 384, 512, 768, 1024, 1536, 2048, 4096)
# the solver settings of the repository's benchmark: a 300-sweep first solve
# and sixteen Anderson-combined corrections of 200 sweeps
BENCH = dict(residual_every=50, max_iters=300, check_every=8, tol_u_scale=50.0, refine=16, refine_max_iters=200,
             refine_lam1_iters=50, refine_tol_scale=1.0, stall_checks=20, refine_accel=8)
BENCH_LAM, BENCH_ITERS = [40.0, 10.0, 3.0, 1.5], [1000, 2000, 2000, 2000]
BENCH_TOL = 1e-5
THETA = (0.9, 0.9, 1.0)  # wf_params defaults
# parts of the 1/f floor carried by the stripe and by the white part; the plain
# sweep keeps some of it in its own part
SPLIT = {True: (0.5, 0.5), False: (0.5, 0.0)}


def listed():
    return [
        # the single-messenger filter of a small map: white noise, no mask,
        # cooling from 1e3 to 1 over 20 levels of 10 sweeps.  The smallest
        # call: launches and host round trips count
        dict(name="white_64", kind="run", ny=64, nx=64, parts="w", mask=0.0, amp=False, merge=True, every=10,
             levels=20, per_level=10, lam0=1e3),
        # one small three-part map solved to the stop test (the size of the
        # warm-start workload's training maps)
        dict(name="solve_256", kind="solve", n=256),
        # the headline: one 1024^2 three-part map solved to the stop test
        dict(name="solve_1024", kind="solve", n=1024),
        # the adaptive cooling rule with the default parameters (a residual
        # every ten sweeps) on a ragged map with per-row stripe amplitudes
        dict(name="adaptive_512x384", kind="adaptive", ny=512, nx=384, parts="wfr", mask=0.05, amp=True, merge=True,
             sweeps=200),
        # part of a solve on a wide 3 * 2^k map
        dict(name="run_768x1536", kind="run", ny=768, nx=1536, parts="wfr", mask=0.05, amp=True, merge=True, every=50,
             levels=3, per_level=50, lam0=40.0),
        # the paper's plain sweep (the 1/f messenger stored, not marginalised)
        dict(name="plain_1024x512", kind="run", ny=1024, nx=512, parts="wfr", mask=0.05, amp=False, merge=False,
             every=50, levels=2, per_level=100, lam0=10.0),
        # part of a solve on the largest map of the batched workload
        dict(name="run_2048", kind="run", ny=2048, nx=2048, parts="wfr", mask=0.05, amp=False, merge=True, every=50,
             levels=2, per_level=50, lam0=40.0),
        # part of a solve on the largest map the library takes (its fields are
        # far larger than L2)
        dict(name="run_4096", kind="run", ny=4096, nx=4096, parts="wfr", mask=0.05, amp=False, merge=True, every=50,
             levels=1, per_level=50, lam0=1.0),
        # independent maps of uneven sizes solved together on eight lanes
        dict(name="batch_8", kind="batch", lanes=8, sizes="1024,768,512,512,384,384,256,256"),
        # the 2D transform of a device map and back
        dict(name="fft2_2048", kind="fft2", ny=2048, nx=2048, noalloc=False),
        # the warm start's inference on one map
        dict(name="fno_forward_512", kind="fno_forward", n=512, nb=1, width=32, mx=16, my=16, layers=4),
        # one training batch of the warm start's network: loss and gradient
        dict(name="fno_gradient_256", kind="fno_gradient", n=256, nb=8, width=32, mx=16, my=16, layers=4),
    ]


def draw(rng):
    kind = rng.choice(["run", "run", "run", "adaptive", "solve", "batch", "fft2", "fno_forward", "fno_gradient"])
    if kind in ("run", "adaptive"):
        # (stripes without a 1/f part have no white floor to move: their
        # messenger is pinned at the Nyquist stripe power and FP32 stalls)
        parts = rng.choice(["wfr", "wfr", "wfr", "wf", "w"])
        ny, nx = rng.choice(SIDES), rng.choice(SIDES)
        c = dict(kind=kind, ny=ny, nx=nx, parts=parts, mask=rng.choice([0.0, 0.02, 0.05, 0.1]),
                 amp="r" in parts and rng.random() < 0.5, merge=rng.random() < 0.8)
        most = max(60, min(300, 40_000_000 * 20 // (ny * nx)))  # no more than about the 4096^2 run costs
        if kind == "run":
            levels = rng.randint(1, 4)
            return dict(c, every=rng.choice([10, 20, 50]), levels=levels,
                        per_level=max(10, rng.randint(30, most) // (10 * levels) * 10),
                        lam0=round(10 ** rng.uniform(0.5, 3), 3))
        return dict(c, sweeps=rng.randint(30, min(most, 200)) // 10 * 10)
    if kind == "solve":
        return dict(kind=kind, n=rng.choice([256, 384, 512, 768]))
    if kind == "batch":
        n = rng.randint(2, 8)
        sizes = sorted((rng.choice([256, 384, 512, 768]) for _ in range(n)), reverse=True)
        return dict(kind=kind, lanes=rng.choice([1, 4, 8]), sizes=",".join(map(str, sizes)))
    if kind == "fft2":
        ny, nx = rng.choice(SIDES), rng.choice(SIDES)
        return dict(kind=kind, ny=ny, nx=nx, noalloc=ny * nx <= 1048576 and rng.random() < 0.5)
    n = rng.choice([64, 128, 256, 512])
    return dict(kind=kind, n=n, nb=rng.randint(1, max(1, min(16, 8 * 256 * 256 // (n * n)))),
                width=rng.choice([16, 24, 32, 32, 32, 48, 64]), mx=rng.choice([8, 12, 16, 16, 16]),
                my=rng.choice([8, 12, 16, 16, 16]), layers=rng.randint(2, 4))


# ------------------------------------------------------------------ inputs


def _k2d(ny, nx, device):
    ky = torch.fft.fftfreq(ny, d=1.0 / ny, device=device, dtype=torch.float64)
    kx = torch.arange(nx // 2 + 1, device=device, dtype=torch.float64)
    return torch.sqrt(ky[:, None] ** 2 + kx[None, :] ** 2)


def _problem(ny, nx, parts, mask_frac, amp, g):
    """Seeded inputs of one map, by the recipe of the repository's synthetic
    workloads: C(k) = (k+2)^-2.5; log-normal white noise at 0.3 of the signal's
    rms; 1/f and stripe noise of the same level with knees at 20 cycles; disc
    masks.  Returns (d, pixel_var, mask, C, P1f, Pst, stripe_amp2)."""
    dev = g.device
    f64 = torch.float64
    normal = lambda *shape: torch.randn(*shape, generator=g, device=dev, dtype=f64)  # noqa: E731
    k = _k2d(ny, nx, dev)
    C = (k + 2.0) ** -2.5
    w = torch.full((ny, nx // 2 + 1), 2.0, device=dev, dtype=f64)
    w[:, 0] = w[:, -1] = 1.0
    sig = 0.3 * math.sqrt(float((C * w).sum()) / (ny * nx))
    field = lambda spec: torch.fft.irfft2(spec.sqrt() * torch.fft.rfft2(normal(ny, nx)), s=(ny, nx))  # noqa: E731
    d = field(C)
    var = (sig * torch.exp(0.5 * normal(ny, nx))) ** 2
    d += var.sqrt() * normal(ny, nx)
    P1f = Pst = amp2 = mask = None
    if "f" in parts:
        P1f = sig ** 2 * (1.0 + (20.0 / k.clamp(min=1.0)) ** 2)
        d += field(P1f)
    if "r" in parts:
        kx = torch.arange(nx // 2 + 1, device=dev, dtype=f64).clamp(min=1.0)
        Pst = sig ** 2 * (20.0 / kx) ** 2.5
        st = torch.fft.irfft(Pst.sqrt()[None, :] * torch.fft.rfft(normal(ny, nx), dim=1), n=nx, dim=1)
        if amp:
            amp2 = torch.exp(normal(ny))
            st = st * amp2.sqrt()[:, None]
        d += st
    if mask_frac > 0:
        # discs of 8 to 32 px per 1024 until the fraction is reached
        scale = max(ny, nx) / 1024.0
        u = torch.rand(4096, 3, generator=g, device=dev, dtype=f64).cpu().numpy()
        m = np.zeros((ny, nx), bool)
        yy, xx, n, i = np.arange(ny), np.arange(nx), 0, 0
        while n < mask_frac * ny * nx and i < len(u):
            cy, cx, r = u[i, 0] * ny, u[i, 1] * nx, max((8.0 + 24.0 * u[i, 2]) * scale, 0.75)
            dy = np.abs(yy - cy)
            dx = np.abs(xx - cx)
            dy, dx = np.minimum(dy, ny - dy), np.minimum(dx, nx - dx)
            ry, rx = np.nonzero(dy <= r)[0], np.nonzero(dx <= r)[0]
            disc = dy[ry][:, None] ** 2 + dx[rx][None, :] ** 2 <= r * r
            old = m[np.ix_(ry, rx)]
            n += int((disc & ~old).sum())
            m[np.ix_(ry, rx)] = old | disc
            i += 1
        mask = torch.from_numpy(m.astype(np.uint8)).to(dev)
        d[mask.bool()] = 0.0
    f32 = lambda a: None if a is None else a.to(torch.float32).contiguous()  # noqa: E731
    return f32(d), f32(var), mask, f32(C), f32(P1f), f32(Pst), f32(amp2)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _inputs(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("run", "adaptive"):
        return _problem(case["ny"], case["nx"], case["parts"], case["mask"], case["amp"], g)
    if kind == "solve":
        return _problem(case["n"], case["n"], "wfr", 0.05, False, g)
    if kind == "batch":
        return [_problem(n, n, "wfr", 0.05, False, g) for n in _sizes(case)]
    if kind == "fft2":
        return torch.randn(case["ny"], case["nx"], generator=g, device="cuda")
    # the network's input: data over sigma and the log noise weight of a
    # masked map, its target a smoothed map of unit size
    n, nb = case["n"], case["nb"]
    x = torch.empty(nb, 2, n, n, device="cuda")
    t = torch.empty(nb, n, n, device="cuda")
    k = _k2d(n, n, "cuda")
    for b in range(nb):
        d, var, mask, *_ = _problem(n, n, "wfr", 0.05, False, g)
        s2 = var[mask == 0].double().mean()
        x[b, 0] = d / s2.sqrt()
        x[b, 1] = torch.where(mask.bool(), math.log(1e-6), torch.log(s2 / var))
        t[b] = torch.fft.irfft2(torch.fft.rfft2(x[b, 0].double()) / (1.0 + (k / 12.0) ** 2), s=(n, n))
    w, mx, my = case["width"], case["mx"], case["my"]
    normal = lambda scale, *shape: torch.randn(*shape, generator=g, device="cuda") * scale  # noqa: E731
    uniform = lambda scale, *shape: torch.rand(*shape, generator=g, device="cuda") * scale  # noqa: E731
    p = [normal(2 ** -0.5, w, 2), normal(0.1, w)]
    for _ in range(case["layers"]):
        p += [normal(w ** -0.5, w, w), normal(0.1, w), uniform(1.0 / (w * w), w, w, 2 * my, mx, 2)]
    p += [normal(w ** -0.5, 1, w), normal(0.1, 1)]
    return x, t, p


def _sizes(case):
    return [int(v) for v in case["sizes"].split(",")]


def _levels(case):
    """lambda of every cooling level of a `run` case, geometric down to 1."""
    n = case["levels"]
    return [1.0] if n == 1 else [case["lam0"] ** ((n - 1 - j) / (n - 1)) for j in range(n)]


def _parts(parts):
    return wf.WF_PART_WHITE | (wf.WF_PART_1F if "f" in parts else 0) | (wf.WF_PART_STRIPE if "r" in parts else 0)


def _fields(case):
    f = ["S"]
    if "f" in case["parts"]:
        f += ["D_2DF"] + ([] if case["merge"] else ["T_2DF"])
    if "r" in case["parts"]:
        f += ["T_RF", "D_RF"]
    return f


def _run_sweeps(case):
    """Sweeps of a `run` case: whole checkpoints, as the run rounds its cap up."""
    n, every = case["levels"] * case["per_level"], case["every"]
    return -(-n // every) * every


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case, inp=_inputs(case, seed))
    if kind in ("run", "adaptive"):
        ny, nx = case["ny"], case["nx"]
        if kind == "run":
            prm = wf.make_params(residual_every=case["every"], max_iters=_run_sweeps(case), merge_2df=case["merge"],
                                 split_f=SPLIT[case["merge"]][0], split_fp=SPLIT[case["merge"]][1])
            state["sched"] = wf.make_schedule("fixed", _levels(case), [case["per_level"]] * case["levels"])
        else:
            prm = wf.make_params(max_iters=case["sweeps"], merge_2df=case["merge"], split_f=SPLIT[case["merge"]][0],
                                 split_fp=SPLIT[case["merge"]][1])
            state["sched"] = wf.make_schedule("adaptive")
        state["plan"] = wf.Plan(ny, nx, _parts(case["parts"]), prm)
        state["out"] = {f: torch.empty(ny, nx, device="cuda") for f in _fields(case)}
    elif kind == "solve":
        n = case["n"]
        state["plan"] = wf.Plan(n, n, _parts("wfr"), wf.make_params(**BENCH))
        state["sched"] = wf.make_schedule("fixed", BENCH_LAM, BENCH_ITERS)
        state["out"] = torch.empty(n, n, device="cuda")
    elif kind == "batch":
        sizes = _sizes(case)
        state["batch"] = wf.Batch([(n, n) for n in sizes], params=wf.make_params(**BENCH), lanes=case["lanes"])
        state["sched"] = wf.make_schedule("fixed", BENCH_LAM, BENCH_ITERS)
        state["out"] = [torch.empty(n, n, device="cuda") for n in sizes]
    elif kind == "fft2":
        ny, nx = case["ny"], case["nx"]
        state["out"] = [torch.empty(ny, nx, device="cuda") for _ in range(2)]
        if not case["noalloc"]:
            state["plan"] = wf.Plan(ny, nx, wf.WF_PART_WHITE)
    else:
        x, t, p = state["inp"]
        flat = torch.cat([v.reshape(-1) for v in p])
        state["net"] = wf.FNO(case["n"], case["nb"], flat, width=case["width"], mx=case["mx"], my=case["my"],
                              layers=case["layers"])
        state["out"] = torch.empty(case["nb"], case["n"], case["n"], device="cuda") if kind == "fno_forward" else (
            torch.empty(flat.numel(), device="cuda"))
    return state


def run(state):
    case, inp, out = state["case"], state["inp"], state["out"]
    kind = case["kind"]
    if kind in ("run", "adaptive"):
        plan = state["plan"]
        plan.set_problem(*inp)
        st = plan.run(state["sched"], 0.0)
        for f, o in out.items():
            plan.get_field(getattr(wf, "WF_FIELD_" + f), o)
        return dict(out, iters=st["iters"])
    if kind == "solve":
        st = state["plan"].solve(*inp, state["sched"], BENCH_TOL, out=out)[1]
        return dict(s=out, iters=st["iters"])
    if kind == "batch":
        stats = state["batch"].solve(inp, state["sched"], BENCH_TOL, out)[1]
        return dict(s=out, iters=[s["iters"] for s in stats])
    if kind == "fft2":
        if case["noalloc"]:
            wf.wf_fft2_noalloc(case["ny"], case["nx"], inp, out[0])
            wf.wf_fft2_noalloc(case["ny"], case["nx"], out[0], out[1], inverse=True)
        else:
            state["plan"].fft2(inp, out=out[0])
            state["plan"].fft2(out[0], inverse=True, out=out[1])
        return out
    net = state["net"]
    x, t, _ = inp
    if kind == "fno_forward":
        return net.forward(x, out, case["nb"])
    # the C entry point with the gradient left on the device, as a training
    # loop with its own optimiser takes it
    loss = ctypes.c_double()
    rc = wf.load().wf_fno_gradient(net.h, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(t.data_ptr()), case["nb"],
                                   ctypes.c_void_p(out.data_ptr()), ctypes.byref(loss))
    if rc != wf.WF_OK:
        raise wf.WFError(rc, "wf_fno_gradient")
    return dict(grad=out, loss=loss.value)


# ------------------------------------------------------------------ work


def _sweep_work(ny, nx, parts, merge):
    """(bytes, flops) of one sweep: every kept field read and written once,
    every table read once; two real 2D transforms and about 30 operations of
    the updates per pixel."""
    px = ny * nx
    fields = 1 + ("r" in parts) + ("r" in parts or "f" in parts) + ("f" in parts and not merge)
    return px * (8 * fields + 8 + 4), px * (10 * math.log2(px) / 2 + 30)


def work(case):
    kind = case["kind"]
    if kind in ("run", "adaptive"):
        ny, nx = case["ny"], case["nx"]
        sweeps = _run_sweeps(case) if kind == "run" else case["sweeps"]
        b, f = _sweep_work(ny, nx, case["parts"], case["merge"])
        checks = 1 if kind == "run" else sweeps // 10
        io = 9 + 4 * ("f" in case["parts"]) + 4 * len(_fields(case))
        # a residual: four transforms and the data and tables once more
        return dict(bytes=sweeps * b + checks * 28 * ny * nx + io * ny * nx,
                    flops=sweeps * f + checks * ny * nx * (10 * math.log2(ny * nx) + 40))
    if kind in ("solve", "batch"):
        sweeps = BENCH["max_iters"] + BENCH["refine"] * BENCH["refine_max_iters"]
        tot = dict(bytes=0.0, flops=0.0)
        for n in [case["n"]] if kind == "solve" else _sizes(case):
            b, f = _sweep_work(n, n, "wfr", True)
            # per correction: the residual of s, the source, the history
            tot["bytes"] += sweeps * b + BENCH["refine"] * (60 + 16 * BENCH["refine_accel"]) * n * n + 17 * n * n
            tot["flops"] += sweeps * f + BENCH["refine"] * n * n * (30 * math.log2(n) + 100)
        return tot
    if kind == "fft2":
        px = case["ny"] * case["nx"]
        return dict(bytes=2 * 8 * px, flops=2 * 2.5 * px * math.log2(px))
    n, nb, w, L = case["n"], case["nb"], case["width"], case["layers"]
    px, modes = nb * n * n, 2 * case["my"] * case["mx"]
    params = 3 * w + L * (w * w + w + 2 * w * w * modes) + w + 1
    # per layer: the channel product and the transform pair of every channel,
    # the mode products; forward once, and twice more for the gradient
    fwd = px * (4 * w + 2 * w) + L * (px * (2 * w * w + w * 5 * math.log2(n * n)) + 8 * nb * w * w * modes)
    if kind == "fno_forward":
        return dict(bytes=4 * (3 * px + params), flops=fwd)
    return dict(bytes=4 * (3 * px + 2 * params), flops=3 * fwd)


# ------------------------------------------------------------------ exact values


def _to(b, x):
    return x if b == "P" else torch.fft.rfft(x, dim=1) if b == "R" else torch.fft.rfft2(x)


def _from(b, X, shape):
    return X if b == "P" else (
        torch.fft.irfft(X, n=shape[1], dim=1) if b == "R" else torch.fft.irfft2(X, s=shape))


def _mean(A, a, B, b):
    """Mean under (x-a)^2/A + (x-b)^2/B; A infinite gives b."""
    A, B = torch.as_tensor(A, dtype=torch.float64, device="cuda"), torch.as_tensor(
        B, dtype=torch.float64, device="cuda")
    x = (B * a + A * b) / (A + B)
    return torch.where(torch.isinf(A), b, x) if bool(torch.isinf(A).any()) else x


class _Chain:
    """The messenger iteration (Huffenberger 2017, Sec. 2 and Appendix A) in
    64 bits, fields kept in pixels."""

    def __init__(self, inp, merge):
        d, var, mask, C, P1f, Pst, amp2 = (None if a is None else a.double() if a.is_floating_point() else a.bool()
                                           for a in inp)
        self.shape = tuple(d.shape)
        self.um = torch.ones_like(d, dtype=torch.bool) if mask is None else ~mask
        self.d, self.C, self.var = torch.where(self.um, d, 0.0), C, var
        self.P1f = P1f
        self.N1 = None if Pst is None else (Pst[None, :] if amp2 is None else amp2[:, None] * Pst[None, :])
        self.merge = merge and P1f is not None
        wf_ = SPLIT[merge][0] * float(P1f.min()) if P1f is not None and Pst is not None else 0.0
        wfp = SPLIT[merge][1] * float(P1f.min()) if P1f is not None else 0.0
        self.parts = []  # (basis, N, tau, Nbar), signal end first
        if P1f is not None:
            n0 = P1f - wf_ - wfp
            tau = 0.0 if self.merge else THETA[0] * float(n0.min())
            self.parts.append(("F", n0, tau, n0 - tau))
        if self.N1 is not None:
            n1 = self.N1 + wf_
            tau = THETA[1] * float(n1.min())
            self.parts.append(("R", n1, tau, n1 - tau))
        n2 = var + wfp
        tau = THETA[2] * float(n2[self.um].min())
        self.parts.append(("P", n2, tau, torch.where(self.um, n2 - tau, math.inf)))
        z = torch.zeros_like(d)
        K = len(self.parts)
        self.s, self.t, self.dd = z, [z] * K, [z] * (K - 1) + [self.d]

    def sweep(self, lam):
        T = [lam * p[2] for p in self.parts]
        for i in range(len(self.parts) - 1, 0 if self.merge else -1, -1):
            b, _, _, nbar = self.parts[i]
            sig = self.dd[i - 1] if i > 0 else self.s
            self.t[i] = _from(b, _mean(nbar, _to(b, self.dd[i]), T[i], _to(b, sig)), self.shape)
            if i > (1 if self.merge else 0):
                pb, _, _, pn = self.parts[i - 1]
                self.dd[i - 1] = _from(pb, _mean(T[i], _to(pb, self.t[i]), pn, _to(pb, self.t[i - 1])), self.shape)
        if self.merge:
            N0 = self.parts[0][1]
            D0 = (self.C + N0) / (self.C + N0 + T[1]) * _to("F", self.t[1])
            self.dd[0] = _from("F", D0, self.shape)
            self.s = _from("F", self.C / (self.C + N0) * D0, self.shape)
        else:
            self.s = _from("F", self.C / (self.C + T[0]) * _to("F", self.t[0]), self.shape)

    def apply_n(self, x):
        y = self.var * x
        if self.P1f is not None:
            y = y + _from("F", self.P1f * _to("F", x), self.shape)
        if self.N1 is not None:
            y = y + _from("R", self.N1 * _to("R", x), self.shape)
        return y

    def rho2(self):
        """||Delta d||^2 on the unmasked pixels, Delta d = (I + N S^-1) s - d."""
        g = _from("F", _to("F", self.s) / self.C, self.shape)
        rho = torch.where(self.um, self.apply_n(torch.where(self.um, g, 0.0)) + self.s - self.d, 0.0)
        return float((rho * rho).sum())

    def solution(self, tol=1e-10, most=6000):
        """The Wiener solution by conjugate gradients on the unmasked pixels,
        (S + N)_uu x = d_u, s = S x, or None if it needs too many steps."""
        um = self.um
        nk = self.C + float(self.var[um].mean())
        if self.P1f is not None:
            nk = nk + self.P1f
        if self.N1 is not None:
            nk = nk + self.N1.mean(dim=0, keepdim=True)

        def A(x):
            return torch.where(um, self.apply_n(x) + _from("F", self.C * _to("F", x), self.shape), 0.0)

        def M(r):
            return torch.where(um, _from("F", _to("F", r) / nk, self.shape), 0.0)

        x, r = torch.zeros_like(self.d), self.d.clone()
        z = M(r)
        p, rz, bn = z, (r * z).sum(), float(self.d.norm())
        for i in range(most):
            Ap = A(p)
            al = rz / (p * Ap).sum()
            x, r = x + al * p, r - al * Ap
            if i % 20 == 0 and float(r.norm()) <= tol * bn:
                return _from("F", self.C * _to("F", x), self.shape)
            z = M(r)
            new = (r * z).sum()
            p, rz = z + (new / rz) * p, new
        return None


def _exact_run(case, inp):
    ch = _Chain(inp, case["merge"])
    if case["kind"] == "run":
        lam = _levels(case)
        n, every = _run_sweeps(case), case["every"]
        lev, at = 0, 0
        for i in range(1, n + 1):
            ch.sweep(lam[lev])
            at += 1
            if i % every == 0 and lev < len(lam) - 1 and at >= case["per_level"]:
                lev, at = lev + 1, 0
    else:  # the adaptive rule: lambda^0.7 once the residual falls by under 1% a sweep, 1 below 1.01
        n, lam, prev = case["sweeps"], 5e5, None
        for i in range(1, n + 1):
            ch.sweep(lam)
            if i % 10:
                continue
            if lam > 1.0:
                rho2 = ch.rho2()
                if prev is not None and abs(1.0 - (rho2 / prev) ** 0.1) < 1e-2:
                    lam = lam ** 0.7
                    lam, prev = (1.0 if lam < 1.01 else lam), None
                else:
                    prev = rho2
    idx = {b: i for i, (b, *_) in enumerate(ch.parts)}
    out = {}
    for f in _fields(case):
        if f == "S":
            out[f] = ch.s
        elif f.endswith("2DF"):
            out[f] = (ch.dd if f[0] == "D" else ch.t)[idx["F"]]
        else:
            out[f] = (ch.dd if f[0] == "D" else ch.t)[idx["R"]]
    return dict(out, iters=n)


def _exact_fft(x):
    X = torch.fft.rfft2(x.double())
    h = X.shape[1] - 1
    Z = torch.cat([X[:, :1] + 1j * X[:, h:], X[:, 1:h]], dim=1)
    return [torch.view_as_real(Z).reshape(x.shape), x.double()]


def _exact_fno(case, inp):
    """The network in 64 bits on the FP16-rounded matrices, its loss and the
    gradient with respect to them."""
    x, t, p = inp
    n, mx, my, L = case["n"], case["mx"], case["my"], case["layers"]
    bias = lambda i: i == 1 or i == len(p) - 1 or (2 <= i < len(p) - 2 and (i - 2) % 3 == 1)  # noqa: E731
    q = [(v if bias(i) else v.half()).double().requires_grad_(case["kind"] == "fno_gradient") for i, v in enumerate(p)]
    h = torch.einsum("oi,bixy->boxy", q[0], x.double()) + q[1][None, :, None, None]
    rows = list(range(my)) + list(range(n - my, n))
    for layer in range(L):
        W, w, R = q[2 + 3 * layer: 5 + 3 * layer]
        X = torch.fft.rfft2(h)[:, :, rows, :mx]
        Y = torch.einsum("iokm,bikm->bokm", torch.view_as_complex(R), X)
        full = torch.zeros(h.shape[0], h.shape[1], n, n // 2 + 1, dtype=torch.complex128, device=h.device)
        full[:, :, rows, :mx] = Y
        # k_x > 0 counted twice, k_x = 0 by its real part row by row
        r = torch.fft.ifft(full, dim=2)
        r = torch.cat([r[..., :1].real + 0j, r[..., 1:]], dim=3)
        z = torch.fft.irfft(r, n=n, dim=3) + torch.einsum("oi,bixy->boxy", W, h) + w[None, :, None, None]
        h = torch.nn.functional.gelu(z) if layer < L - 1 else z
    y = torch.einsum("oi,bixy->boxy", q[-2], h)[:, 0] + q[-1]
    if case["kind"] == "fno_forward":
        return y
    td = t.double()
    loss = (((y - td) ** 2).sum((1, 2)) / (td ** 2).sum((1, 2))).mean()
    loss.backward()
    return dict(grad=torch.cat([v.grad.reshape(-1) for v in q]), loss=float(loss.detach()))


def exact(case, seed):
    kind = case["kind"]
    inp = _inputs(case, seed)
    if kind in ("run", "adaptive"):
        return _exact_run(case, inp)
    if kind == "solve":
        return dict(s=_Chain(inp, True).solution(), iters=None)
    if kind == "batch":
        return dict(s=[_Chain(i, True).solution() for i in inp], iters=[None] * len(inp))
    if kind == "fft2":
        return _exact_fft(inp)
    return _exact_fno(case, inp)
