"""The work that users of the library have it do, as cases that can be timed:
forward solves of candidate parameter sets, the misfit, sensitivities and
gradients, single and batched inversions, in the sizes of the workloads in
``paper_1109_0334_gb300/workloads.py`` and of the ranges around them.

A case is a dict of plain values.  ``prepare`` makes what a program has in
hand before the call (problem, record, candidates), ``run`` is one pass
through the public entry points of ``paper_1109_0334_gb300.afminv``, ``work``
what the pass cannot do without, and ``exact`` the same outputs in 64 bits by
plain torch.

Kinds:
  forward   candidates integrated over the record, with the misfit and, where
            ``defl``, every deflection (f32 or f64)
  fe        the same on the finite-element beam
  misfit    the misfit of stored deflections
  normal    misfit, Gauss-Newton matrix and gradient (forward sensitivities)
  adjoint   misfit and gradient (reverse mode, torch.autograd)
  invert    one particle-swarm inversion of one record
  batch     inversions of many pixels with records of uneven length
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1109_0334_gb300 import afminv as A
from paper_1109_0334_gb300 import workloads as W


# --------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: the point-mass swarm of one small inversion, its
        # 20-cycle traces kept (plots, a hand-written optimiser's inner loop)
        dict(name="forward_c1_64", kind="forward", load="c1", modes=1, P=64, steps=4000,
             defl=True, f64=False),
        # traces of a set of viscoelastic candidates (a law with a rate term)
        # over a whole record, an odd number of them
        dict(name="forward_c4_trace", kind="forward", load="c4", modes=3, P=1001, steps=25600,
             defl=True, f64=False),
        # a wide scan of the parameter cube, misfits only
        dict(name="forward_c2_wide", kind="forward", load="c2", modes=3, P=262144, steps=6400,
             defl=False, f64=False),
        # the swarm of the paper's own experiment: 8 modes, 8 cycles
        dict(name="forward_f2_8modes", kind="forward", load="f2_hooke", modes=8, P=512,
             steps=4096, defl=False, f64=False),
        # reference traces in 64 bits (truths, checks of an inversion's result)
        dict(name="forward_c2_f64", kind="forward", load="c2", modes=3, P=96, steps=10240,
             defl=True, f64=True),
        # one Levenberg-Marquardt step's sensitivities for one inversion: 64
        # candidates x 8 damping values.  Derivatives are taken over records
        # of up to ten cycles: over longer ones, and with the viscoelastic
        # law's square root at the onset of contact, those of candidates that
        # graze the sample amplify the rounding of any 32-bit solve
        dict(name="normal_c2_512", kind="normal", load="c2", modes=3, P=512, steps=2560),
        # the same for the best 32 of each of 512 pixels
        dict(name="normal_c2_wide", kind="normal", load="c2", modes=3, P=16384, steps=1280),
        # gradients of the best 32 particles through torch.autograd
        dict(name="adjoint_c2_32", kind="adjoint", load="c2", modes=3, P=32, steps=2560),
        # one inversion, the 1024-particle swarm on a 100-cycle record
        dict(name="invert_c2", kind="invert", load="c2", modes=3, P=1024, iters=5, steps=25600),
        # an image line's pixels: uneven records of 20 to 60 cycles
        dict(name="batch_c3", kind="batch", load="c3", modes=3, P=256, iters=2, pixels=304,
             lo=5120, hi=15360),
        # the finite-element swarm's evaluation
        dict(name="fe_c5", kind="fe", load="c5", P=8192, steps=12800, defl=False),
        # misfits of stored deflections (another record against the same runs)
        dict(name="misfit_stored", kind="misfit", P=4096, steps=25600),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "forward64", "normal", "adjoint", "invert", "batch",
                       "fe", "misfit"])
    if kind in ("forward", "forward64"):
        f64 = kind == "forward64"
        load = rng.choice(["c1", "c2", "c2", "c4", "f2_hooke"])
        f2 = load == "f2_hooke"
        # the highest mode a step of 1/256 cycle resolves is the fifth or sixth
        modes = 1 if load == "c1" else rng.choice([1, 3, 5, 8] if f2 else [1, 2, 3, 3, 5])
        steps = _log_int(rng, 500, 4096 if f2 else 10000 if f64 else 25600)
        P = _log_int(rng, 16, 128) if f64 else _log_int(
            rng, 48, 4000 if f2 else min(200000, 8e8 / steps))
        defl = rng.random() < 0.5 and P * steps < 30e6
        return dict(kind="forward", load=load, modes=modes, P=P, steps=steps, defl=defl, f64=f64)
    if kind == "normal":
        # (the slope of Hooke's law jumps at contact: few candidates, so that
        # a stage within rounding of the jump stays the exception)
        steps = _log_int(rng, 300, 2560)
        load = rng.choice(["c2", "c2", "f2_hooke"])
        top = 700 if load == "f2_hooke" else min(17000, 2.1e7 / steps)
        return dict(kind="normal", load=load, modes=rng.choice([1, 3, 3]),
                    P=_log_int(rng, 16, top), steps=steps)
    if kind == "adjoint":
        return dict(kind="adjoint", load="c2", modes=rng.choice([1, 3, 3]),
                    P=_log_int(rng, 8, 512), steps=_log_int(rng, 300, 2560))
    if kind == "invert":
        load = rng.choice(["c1", "c2", "c4", "f2_hooke"])
        return dict(kind="invert", load=load, modes={"c1": 1, "f2_hooke": 8}.get(load, 3),
                    P=_log_int(rng, 64, 1500), iters=rng.randint(1, 5),
                    steps=_log_int(rng, 1000, 4096 if load == "f2_hooke" else 20000))
    if kind == "batch":
        lo = _log_int(rng, 600, 5000)
        return dict(kind="batch", load="c3", modes=rng.choice([1, 3, 3]),
                    P=rng.choice([64, 100, 128, 200, 256]), iters=rng.randint(0, 2),
                    pixels=rng.randint(20, 300), lo=lo, hi=rng.randint(lo, 3 * lo))
    if kind == "fe":
        return dict(kind="fe", load="c5", P=_log_int(rng, 64, 8192), steps=_log_int(rng, 1000, 10000),
                    defl=rng.random() < 0.3)
    return dict(kind="misfit", P=_log_int(rng, 30, 8000), steps=_log_int(rng, 1000, 12000))


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
def _spec(case):
    spec = W.get(case["load"])
    if "modes" in case and spec["model"] != "fe_hermite":
        if spec["model"] == "point_mass":
            assert case["modes"] == 1
        else:
            spec["n_modes"] = case["modes"]
    return spec


def _noise(n, sigma, gen):
    return sigma * torch.randn(n, dtype=torch.float64, device="cuda", generator=gen)


def _truth(D, n, seed):
    """Truths in the interior of the normalised cube, [D][n]."""
    return torch.from_numpy(np.random.default_rng(seed).uniform(0.1, 0.9, (D, n))).cuda()


def _record(prob, spec, D, seed, gen):
    """One measured record: a truth's deflection in 64 bits plus noise."""
    defl, _ = A.forward_batch_f64(prob, _truth(D, 1, seed), None)
    return defl[:, 0] + _noise(prob.n_steps, spec["sigma"] * 1e9, gen)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "misfit":
        n, P = case["steps"], case["P"]
        t = torch.arange(n, device="cuda", dtype=torch.float32) * (2 * math.pi / 256)
        amp = 15.0 + 6.0 * torch.rand(P, device="cuda", generator=gen)
        ph = 0.3 * torch.rand(P, device="cuda", generator=gen)
        defl = torch.cos(t[:, None] + ph[None, :])
        defl *= amp[None, :]
        U = (18.0 * torch.cos(t + 0.1)
             + 0.1 * torch.randn(n, device="cuda", generator=gen))
        return dict(case=case, defl=defl, U=U)
    spec = _spec(case)
    D = len(spec["free"])
    if kind == "batch":
        rng = np.random.default_rng(seed)
        n_i = rng.integers(case["lo"], case["hi"] + 1, case["pixels"])
        off = np.concatenate([[0], np.cumsum(n_i)]).astype(np.int64)
        prob = A.make_problem(spec, n_steps=int(n_i.max()))
        defl, _ = A.forward_batch_f64(prob, _truth(D, case["pixels"], seed + 1), None)
        U = torch.cat([defl[:int(n), i] for i, n in enumerate(n_i)])
        U = (U + _noise(U.numel(), spec["sigma"] * 1e9, gen)).float()
        spec.update(P=case["P"], iters=case["iters"], seed=1000 + seed)
        ws = torch.empty(A.invert_batch_workspace_size(prob, case["pixels"]), dtype=torch.uint8,
                         device="cuda")
        return dict(case=case, prob=prob, U=U, off=torch.from_numpy(off).cuda(),
                    cfg=A.make_pso(spec), workspace=ws)
    prob = A.make_problem(spec, n_steps=case["steps"])
    U = _record(prob, spec, D, seed, gen)
    state = dict(case=case, prob=prob, U=U.float())
    if kind == "invert":
        spec.update(P=case["P"], iters=case["iters"], seed=1000 + seed)
        state["cfg"] = A.make_pso(spec)
        return state
    x = torch.rand((D, case["P"]), dtype=torch.float32, device="cuda", generator=gen)
    if case.get("f64"):
        state.update(x=x.double(), U=state["U"].double())
    else:
        state["x"] = x.requires_grad_(kind == "adjoint")
    return state


# --------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------
def _result_fields(res):
    """Columns of afm_result records (bytes) on the device.  S is an FP32
    misfit held in a double."""
    f = res.reshape(-1, res.shape[-1]).view(torch.float64)
    i = res.reshape(-1, res.shape[-1]).view(torch.int32)
    return dict(x=f[:, 0:5], theta=f[:, 5:10], S=f[:, 10].float(), S_f64=f[:, 11], J_rel=f[:, 12],
                run=i[:, 26:30])   # updates, winner, non-finite count, status


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("forward", "fe"):
        fwd = A.forward_batch_f64 if case.get("f64") else A.forward_batch
        defl, S = fwd(state["prob"], state["x"], state["U"], want_defl=case["defl"])
        return dict(defl=defl, S=S) if case["defl"] else dict(S=S)
    if kind == "misfit":
        return dict(S=A.misfit(state["defl"], state["U"]))
    if kind == "normal":
        S, H, b = A.normal_equations(state["prob"], state["x"], state["U"])
        # FP64 totals of FP32 sensitivities: 32-bit numbers
        return dict(S=S, H=H.float(), b=b.float())
    if kind == "adjoint":
        x = state["x"]
        S = A.misfit_autograd(state["prob"], x, state["U"])
        (G,) = torch.autograd.grad(S.sum(), x)
        return dict(S=S.detach(), G=G)
    if kind == "invert":
        res, hist = A.invert(state["prob"], state["U"], state["cfg"])
        return dict(_result_fields(res), history=hist)
    res, _ = A.invert_batch(state["prob"], state["U"], state["off"], state["cfg"],
                            workspace=state["workspace"])
    return _result_fields(res)


def work(case):
    kind, P = case["kind"], case["P"]
    if kind == "misfit":
        n = case["steps"]
        return dict(bytes=4.0 * (n * P + n + P), flops=3.0 * n * P)
    size = 8 if case.get("f64") else 4
    if kind == "fe":
        # per mode 4 fused operations and 4 more, the tip force and misfit 27
        n = case["steps"]
        out = P * (n if case["defl"] else 0) + P
        return dict(bytes=4.0 * (4 * P + n + out), flops=2.0 * 539 * n * P)
    D = len(W.get(case["load"])["free"])
    per_step = 2.0 * (36 * case["modes"] + 24)     # RK4 of Eq. 2, tip force, misfit
    if kind == "batch":
        mean = 0.5 * (case["lo"] + case["hi"])
        evals = case["P"] * (case["iters"] + 1) * case["pixels"]
        return dict(bytes=4.0 * mean * case["pixels"] + 160.0 * case["pixels"],
                    flops=per_step * evals * mean)
    n = case["steps"]
    if kind == "invert":
        return dict(bytes=4.0 * n + 160.0, flops=per_step * P * (case["iters"] + 1) * n)
    if kind == "normal":
        return dict(bytes=4.0 * (D * P + n + P) + 8.0 * P * (D * D + D),
                    flops=(per_step * (1 + 0.8 * D) + D * (D + 3)) * P * n)
    if kind == "adjoint":
        return dict(bytes=4.0 * (2 * D * P + n + P), flops=3 * per_step * P * n)
    out = P * (n if case["defl"] else 0) + P
    return dict(bytes=float(size) * (D * P + n + out), flops=per_step * P * n)


# --------------------------------------------------------------------------
# The same in 64 bits, by plain torch
# --------------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind in ("invert", "batch"):
        return None                                 # a swarm's path has no value of its own
    s = prepare(case, seed)
    if kind == "misfit":
        S = torch.zeros(case["P"], dtype=torch.float64, device="cuda")
        for k in range(0, case["steps"], 1024):
            S += (s["U"][k:k + 1024, None].double() - s["defl"][k:k + 1024].double()).square().sum(0)
        return dict(S=S)
    x, U = s["x"].detach().double(), s["U"].double()
    spec = _spec(case)
    if kind == "fe":
        defl, S = _fe64(spec, x, U, case["steps"], case["defl"])
        return dict(defl=defl, S=S) if case["defl"] else dict(S=S)
    if kind == "forward":
        defl, S, _, _ = _solve64(spec, x, U, case["steps"], case["defl"], False)
        return dict(defl=defl, S=S) if case["defl"] else dict(S=S)
    if case["P"] * case["steps"] * x.shape[0] > 2e9:
        return None                                 # over 20 seconds
    _, S, H, b = _solve64(spec, x, U, case["steps"], False, True)
    return dict(S=S, G=-2.0 * b.t().contiguous()) if kind == "adjoint" else dict(S=S, H=H, b=b)


def _theta(spec, x):
    """Parameter slots (SI) [5][P] and their derivatives by x [D][P]."""
    th = [torch.full_like(x[0], v) for v in spec["fixed"]]
    dth = []
    for d, (slot, lo, hi, log) in enumerate(spec["free"]):
        if log:
            la, lb = math.log10(lo), math.log10(hi)
            th[slot] = torch.pow(10.0, la + x[d] * (lb - la))
            dth.append((slot, th[slot] * (math.log(10.0) * (lb - la))))
        else:
            th[slot] = lo + x[d] * (hi - lo)
            dth.append((slot, torch.full_like(x[0], hi - lo)))
    return th, dth


def _beam(spec):
    """Natural frequencies (rad/s), base participations, Q per mode."""
    w1 = 2 * math.pi * spec["f1_hz"]
    m = int(spec.get("n_modes", 1))
    if spec["model"] == "point_mass":
        return np.array([w1]), np.array([1.0]), m
    w, gam = [], []
    b1 = None
    for i in range(1, m + 1):
        b = (2 * i - 1) * math.pi / 2
        for _ in range(60):                          # cos b cosh b + 1 = 0, scaled by sech b
            f = math.cos(b) + 1 / math.cosh(b)
            b -= f / (-math.sin(b) - math.tanh(b) / math.cosh(b))
        b1 = b1 or b
        e = math.exp(-b)
        sig = (1 + e * e + 2 * e * math.cos(b)) / (1 - e * e + 2 * e * math.sin(b))
        w.append(w1 * (b / b1) ** 2)
        gam.append(4 * sig / b * (1 if i % 2 else -1))
    return np.array(w), np.array(gam), m


def _graph_loop(step, n, spc, before, after):
    """step(j) for n steps, j the step within the period; whole periods run
    as one captured graph, with before(period) and after(period) around it."""
    full = n // spc
    side = torch.cuda.Stream()
    if full >= 2:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            for j in range(spc):
                step(j)
        for k in range(full):
            before(k, spc)
            g.replay()
            after(k, spc)
    else:
        full = 0
    for k in range(full, (n + spc - 1) // spc):
        cnt = min(spc, n - k * spc)
        before(k, cnt)
        for j in range(cnt):
            step(j)
        after(k, cnt)
    torch.cuda.synchronize()


def _solve64(spec, x, U, n, want_defl, tangents):
    """RK4 of the modal cantilever for candidates x [D][P], time in steps and
    lengths in nm.  Returns deflections, misfits and the normal equations."""
    w, gam, m = _beam(spec)
    D, P = x.shape
    spc = spec["spc"]
    h = 1.0 / (spec["f1_hz"] * spc)
    wd, Q = w[0], spec["Q"]
    Hc = gam / (w * w - wd * wd + 1j * wd * w / Q)
    amp = spec["A0"] / (wd * wd * abs(Hc.sum()))
    psi = math.pi / 2 - np.angle(Hc.sum())
    c0 = amp * wd * wd * Hc * np.exp(1j * psi) / 1e-9
    col = lambda a: torch.tensor(np.asarray(a, dtype=np.float64), device="cuda")[:, None]  # noqa: E731
    W2, WQ, GA = col((w * h) ** 2), col(w * h / Q), col(gam)
    g_amp = amp * (wd * h) ** 2 / 1e-9

    def g_of(phase):
        return g_amp * math.sin(2 * math.pi * phase / spc + psi)

    th, dth = _theta(spec, x)
    kk, fs = spec["k"], (w[0] * h) ** 2              # force unit: k * 1 nm, scaled by (w1 h)^2
    law = spec["force"]
    zero = torch.zeros_like(x[0])
    # coefficients of the law in scaled units and their derivatives by theta
    if law in ("dmt", "dmt_kv"):
        sR, rt = torch.sqrt(th[2]), math.sqrt(1e-9)
        hz, vw = 4.0 / 3.0 * rt / kk * fs, fs / (6e-27 * kk)
        kv = rt * fs / (kk * h) if law == "dmt_kv" else 0.0
        cf = [hz * th[0] * sR, vw * th[1] * th[2], kv * th[4] * sR, th[3] * 1e9]
        dcf = {0: [hz * sR, zero, zero, zero], 1: [zero, vw * th[2], zero, zero],
               2: [hz * th[0] / (2 * sR), vw * th[1], kv * th[4] / (2 * sR), zero],
               3: [zero, zero, zero, zero + 1e9], 4: [zero, zero, kv * sR, zero]}
    else:
        cf = [fs / kk * th[0], th[1] * 1e9, fs / (kk * h) * th[2], zero]
        dcf = {0: [zero + fs / kk, zero, zero, zero], 1: [zero, zero + 1e9, zero, zero],
               2: [zero, zero, zero + fs / (kk * h), zero], 3: [zero] * 4, 4: [zero] * 4}
    # d c_k / d x_d, [4][D][P]
    J = [torch.stack([dcf[slot][k] * dv for slot, dv in dth]) for k in range(4)]
    rate = law in ("dmt_kv", "spring_damper")
    Zc = spec["Zc"] / 1e-9

    def force(d, dd):
        if law in ("dmt", "dmt_kv"):
            de = torch.clamp(cf[3] - d, min=0.0)
            sq = torch.sqrt(de)
            r = 1.0 / torch.maximum(d, cf[3])
            r2 = r * r
            F = cf[0] * (de * sq) - cf[1] * r2
            if rate:
                F = F - cf[2] * (sq * dd)
            if not tangents:
                return F, None, None, None
            con = d < cf[3]
            Fa = 1.5 * cf[0] * sq + 2.0 * cf[1] * r2 * r
            Fd = torch.where(con, -1.5 * cf[0] * sq, 2.0 * cf[1] * r2 * r)
            Fx = J[0] * (de * sq) - J[1] * r2
            Fr = None
            if rate:
                half = torch.where(con, 0.5 * cf[2] * dd / torch.where(con, sq, sq + 1.0), zero)
                Fd, Fa, Fr = Fd + half, Fa - half, -cf[2] * sq
                Fx = Fx - J[2] * (sq * dd)
            return F, Fd, Fr, Fx + J[3] * torch.where(con, Fa, zero)
        con = d < cf[1]
        if law == "hooke":
            F = torch.where(con, cf[0] * (cf[1] - d), zero)
        else:
            F = torch.where(con, cf[0] * (cf[1] - d) - cf[2] * dd, zero)
        if not tangents:
            return F, None, None, None
        one = con.double()
        Fx = one * (J[0] * (cf[1] - d) + J[1] * cf[0])
        if rate:
            Fx = Fx - one * J[2] * dd
        return F, -one * cf[0], (-one * cf[2] if rate else None), Fx

    q = col(c0.imag).repeat(1, P)
    v = col((1j * c0 * wd * h).imag).repeat(1, P)     # d/dt of Im(c e^{iwt}), per step
    tq = torch.zeros(D, m, P, dtype=torch.float64, device="cuda")
    tv = torch.zeros_like(tq)
    S = torch.zeros(P, dtype=torch.float64, device="cuda")
    Hm = torch.zeros(P, D, D, dtype=torch.float64, device="cuda")
    bm = torch.zeros(P, D, dtype=torch.float64, device="cuda")
    Ub = torch.zeros(spc, dtype=torch.float64, device="cuda")
    buf = torch.zeros(spc, P, dtype=torch.float64, device="cuda") if want_defl else None
    defl = torch.empty(n, P, dtype=torch.float64, device="cuda") if want_defl else None

    def rhs(qq, vv, g, tqq, tvv):
        F, Fd, Fr, Fx = force(Zc + qq.sum(0), vv.sum(0) if rate else None)
        a = torch.addcmul(GA * g - W2 * qq, WQ, vv, value=-1.0) + F
        if not tangents:
            return a, None
        dF = Fx + Fd * tqq.sum(1)
        if rate:
            dF = dF + Fr * tvv.sum(1)
        return a, dF[:, None, :] - W2 * tqq - WQ * tvv

    def step(j):
        g0, gh, g1 = g_of(j), g_of(j + 0.5), g_of(j + 1.0)
        qs, vs, ts, us = q, v, tq, tv
        kq, kv_, kt, ku = None, None, None, None
        for s, (wt, f, g) in enumerate(((1, 0.5, g0), (2, 0.5, gh), (2, 1.0, gh), (1, 0.0, g1))):
            a, ta = rhs(qs, vs, g, ts, us)
            kq, kv_ = (vs, a) if s == 0 else (torch.add(kq, vs, alpha=wt), torch.add(kv_, a, alpha=wt))
            if tangents:
                kt, ku = (us, ta) if s == 0 else (torch.add(kt, us, alpha=wt),
                                                  torch.add(ku, ta, alpha=wt))
            if f:
                qs, vs = torch.add(q, vs, alpha=f), torch.add(v, a, alpha=f)
                if tangents:
                    ts, us = torch.add(tq, us, alpha=f), torch.add(tv, ta, alpha=f)
        q.add_(kq, alpha=1.0 / 6.0)
        v.add_(kv_, alpha=1.0 / 6.0)
        u = q.sum(0)
        if want_defl:
            buf[j].copy_(u)
        r = Ub[j] - u
        S.addcmul_(r, r)
        if tangents:
            tq.add_(kt, alpha=1.0 / 6.0)
            tv.add_(ku, alpha=1.0 / 6.0)
            au = tq.sum(1).t()
            bm.addcmul_(au, r[:, None])
            Hm.addcmul_(au[:, :, None], au[:, None, :])

    def before(k, cnt):
        Ub[:cnt].copy_(U[k * spc:k * spc + cnt])

    def after(k, cnt):
        if want_defl:
            defl[k * spc:k * spc + cnt].copy_(buf[:cnt])

    _graph_loop(step, n, spc, before, after)
    return defl, S, Hm, bm


def _fe64(spec, x, U, n, want_defl):
    """The Hermite beam by Newmark's average acceleration in the eigenbasis of
    the element model, the tip force implicit (Newton on the tip deflection)."""
    ne, L, E, kk, spc = spec["n_elem"], spec["L"], spec["E"], spec["k"], spec["spc"]
    he, nd = L / ne, 2 * ne
    I = kk * L ** 3 / (3 * E)  # noqa: E741
    b = 1.8751040687119611
    mu = E * I * (b / L) ** 4 / (2 * math.pi * spec["f1_hz"]) ** 2
    me = mu * he / 420 * np.array([[156, 22 * he, 54, -13 * he], [22 * he, 4 * he * he, 13 * he, -3 * he * he],
                                   [54, 13 * he, 156, -22 * he], [-13 * he, -3 * he * he, -22 * he, 4 * he * he]])
    ke = E * I / he ** 3 * np.array([[12, 6 * he, -12, 6 * he], [6 * he, 4 * he * he, -6 * he, 2 * he * he],
                                     [-12, -6 * he, 12, -6 * he], [6 * he, 2 * he * he, -6 * he, 4 * he * he]])
    M, K = np.zeros((nd + 2, nd + 2)), np.zeros((nd + 2, nd + 2))
    for e in range(ne):
        M[2 * e:2 * e + 4, 2 * e:2 * e + 4] += me
        K[2 * e:2 * e + 4, 2 * e:2 * e + 4] += ke
    M, K = M[2:, 2:], K[2:, 2:]
    Lc = np.linalg.cholesky(M)
    Li = np.linalg.inv(Lc)
    _, Y = np.linalg.eigh(Li @ K @ Li.T)
    Phi = Li.T @ Y
    # eigenvalues as Rayleigh quotients in extended precision: the resonance
    # amplifies an error of the drive frequency
    Pl, Ml, Kl = Phi.astype(np.longdouble), M.astype(np.longdouble), K.astype(np.longdouble)
    mass = (Pl * (Ml @ Pl)).sum(0)
    lam = ((Pl * (Kl @ Pl)).sum(0) / mass).astype(np.float64)
    Phi = Phi / np.sqrt(mass.astype(np.float64))
    wA, wB = math.sqrt(lam[0]), math.sqrt(lam[1])
    beta = 1.0 / spec["Q"] / (wA + wB)
    alpha = beta * wA * wB
    w, h = wA, 2 * math.pi / (wA * spc)
    c = alpha + beta * lam
    Gam = Phi.T @ M[:, 0::2].sum(1)
    tip = Phi[nd - 2]
    Hc = Gam / (lam - w * w + 1j * w * c)
    a = spec["A0"] / (w * w * abs((tip * Hc).sum()))
    psi = math.pi / 2 - np.angle((tip * Hc).sum())
    z0 = (a * w * w * Hc * np.exp(1j * psi) / 1e-9).imag
    zm = (a * w * w * Hc * np.exp(1j * (psi - w * h)) / 1e-9).imag
    sm = 1 + 0.5 * h * c + 0.25 * h * h * lam
    D, P = x.shape
    col = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")[:, None]  # noqa: E731
    B1, D2, GG = col(-h * h * lam / sm), col(-h * c / sm), col(Gam / sm)
    FF, PT = col(0.25 * h * h * kk * tip / sm), col(tip)
    ctip = float((tip * (0.25 * h * h * kk * tip / sm)).sum())
    th, _ = _theta(spec, x)
    sR, rt, Zc = torch.sqrt(th[2]), math.sqrt(1e-9), spec["Zc"] / 1e-9
    hz, vw, a0 = 4.0 / 3.0 * th[0] * sR * rt / kk, th[1] * th[2] / (6e-27 * kk), th[3] * 1e9

    def force(d):
        de = torch.clamp(a0 - d, min=0.0)
        sq = torch.sqrt(de)
        r = 1.0 / torch.maximum(d, a0)
        return hz * (de * sq) - vw * r * r, torch.where(d > a0, 2 * vw * r ** 3, -1.5 * hz * sq)

    z, dz = col(z0).repeat(1, P), col(z0 - zm).repeat(1, P)
    Fn = force(Zc + torch.full_like(x[0], float((tip * z0).sum())))[0]
    Fm = force(Zc + torch.full_like(x[0], float((tip * zm).sum())))[0]
    S = torch.zeros(P, dtype=torch.float64, device="cuda")
    Ub = torch.zeros(spc, dtype=torch.float64, device="cuda")
    buf = torch.zeros(spc, P, dtype=torch.float64, device="cuda") if want_defl else None
    defl = torch.empty(n, P, dtype=torch.float64, device="cuda") if want_defl else None
    amp = 0.25 * h * h * a * w * w / 1e-9

    def table(j):
        ph = 2 * math.pi / spc
        return amp * (math.sin(ph * (j + 1) + psi) + 2 * math.sin(ph * j + psi) + math.sin(ph * (j - 1) + psi))

    def step(j):
        dz.add_(torch.addcmul(B1 * z, D2, dz) + GG * table(j) + FF * (2.0 * Fn + Fm))
        z.add_(dz)
        base = (PT * z).sum(0)
        u = base + ctip * Fn
        for _ in range(3):
            F, dF = force(Zc + u)
            u = u - (u - base - ctip * F) / (1.0 - ctip * dF)
        F, _ = force(Zc + u)
        dz.addcmul_(FF, F[None, :])
        z.addcmul_(FF, F[None, :])
        Fm.copy_(Fn)
        Fn.copy_(F)
        if want_defl:
            buf[j].copy_(u)
        r = Ub[j] - u
        S.addcmul_(r, r)

    def before(k, cnt):
        Ub[:cnt].copy_(U[k * spc:k * spc + cnt])

    def after(k, cnt):
        if want_defl:
            defl[k * spc:k * spc + cnt].copy_(buf[:cnt])

    _graph_loop(step, n, spc, before, after)
    return defl, S
