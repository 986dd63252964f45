"""The work that users of the library have it do, as cases that can be timed and checked.

A case is one run of a group of chains through the public entry points: restart from given conformations
(`bd_set_positions`), integrate some sampling windows (`bd_step`), and read back what the run computes - the
replica-averaged and time-averaged force of every window, conformations, kinetics and events, or the Eq. 5 diagnostics -
or, for the differentiation workload, one forward and backward pass of `replica_averaged_run`.

The sizes are those of the workloads in `paper_2206_05851_gb300/inputs.py` and of the tests, with fewer windows where one
pass would take long; `draw` spreads sizes over the ranges these stand for. The outputs of a float32 run are kept in
float32, the precision it integrates in (as `replica_averaged_run` does with the gradient of float32 parameters); those
of a float64 run are float64. `exact` is the method in plain float64 torch (Eq. 1 on bead positions, Eqs. 2-5, the
published Philox4x32-10 generator), written from the definitions and sharing nothing with the kernels.
"""
import math

import numpy as np
import torch

from paper_2206_05851_gb300 import bdra, inputs
from paper_2206_05851_gb300.autograd import RunSpec, replica_averaged_run

S_MIN = 1e-3


# ---------------------------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------------------------

def _case(model, bits, chains, beads, replicas, window, windows, **more):
    """model: fene / collapsed / rpy / vwf (chain model), `bits`: integration precision; beads_max: chains of uneven
    length, beads .. beads_max (0: all `beads`), replicas_min likewise; per_call: windows per bd_step call (0: the whole
    run in one call); kinetics: threshold and Bell criteria on ISF, TSF and RSF, and the event list; conformation: the
    Eq. 5 diagnostics; gradient: forward and backward pass; flow: the imposed flow and its Weissenberg number wi."""
    c = {"model": model, "bits": bits, "chains": chains, "beads": beads, "replicas": replicas, "window": window,
         "windows": windows, "beads_max": 0, "replicas_min": 0, "per_call": 0, "kinetics": False, "conformation": False,
         "gradient": False, "flow": "uniaxial", "wi": 5.0}
    c.update(more)
    return c


def listed():
    cases = [
        # one chain in float64 with a replica set: a user's first run, and a check of the method
        dict(_case("fene", 64, 1, 20, 16, 100, 10, wi=2.0), name="single_fp64"),
        # a handful of uneven chains watched as they run: one window per call, profile and events read after each
        dict(_case("fene", 32, 24, 3, 13, 25, 8, beads_max=61, replicas_min=2, per_call=1, kinetics=True, flow="shear"),
             name="small_watched"),
        # the benchmark workload: 1024 chains of 100 beads, 64 replicas, planar elongation
        dict(_case("fene", 32, 1024, 100, 64, 100, 10, flow="planar"), name="planar_1024"),
        # chains of 20 to 500 beads and 8 to 128 replicas in one batch, shear and uniaxial flow
        dict(_case("fene", 32, 512, 20, 128, 100, 2, beads_max=500, replicas_min=8, flow="mixed", wi=10.0), name="uneven_512"),
        # many short chains with every criterion: the rupture kinetics workload
        dict(_case("fene", 32, 16384, 50, 32, 100, 2, kinetics=True, wi=10.0), name="bell_16384"),
        # the benchmark's chains in float64, the reference precision
        dict(_case("fene", 64, 64, 100, 64, 100, 2, flow="planar"), name="planar_fp64"),
        # the Eq. 5 conformation diagnostics beside the forces
        dict(_case("fene", 32, 256, 100, 64, 100, 4, conformation=True, flow="planar"), name="conformation_256"),
        # the collapsed chain (harmonic springs, Lennard-Jones), free draining, in shear: S = 0.003 tau
        dict(_case("collapsed", 32, 1024, 50, 50, 300, 1, flow="shear", wi=0.0), name="collapsed_1024"),
        # the paper's model: collapsed chains with hydrodynamic interaction in shear
        dict(_case("rpy", 32, 128, 50, 50, 100, 1, flow="shear", wi=0.0), name="rpy_128"),
        # the von Willebrand factor chain at rest with hydrodynamic interaction and its unfolding kinetics
        dict(_case("vwf", 32, 64, 50, 40, 50, 2, kinetics=True, flow="none", wi=0.0), name="vwf_64"),
        # the paper's model in float64
        dict(_case("rpy", 64, 8, 50, 40, 20, 1, flow="shear", wi=0.0), name="rpy_fp64"),
        # gradients of the force profile and the survival with respect to rate, b and H
        dict(_case("fene", 32, 256, 200, 32, 100, 10, gradient=True), name="gradient_256"),
    ]
    return cases


# seconds of a bead-step (model, bits), for the sizes of drawn cases only
_COST = {("fene", 32): 4e-12, ("fene", 64): 4e-10, ("collapsed", 32): 3e-11, ("collapsed", 64): 3e-9, ("rpy", 32): 2e-9,
         ("rpy", 64): 1e-7, ("vwf", 32): 2e-9}


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))

    kind = rng.choice(["fene", "fene", "fene64", "conformation", "collapsed", "rpy", "vwf", "rpy64", "collapsed64", "gradient"])
    model = {"fene64": "fene", "conformation": "fene", "collapsed64": "collapsed", "rpy64": "rpy", "gradient": "fene"}.get(kind, kind)
    bits = 64 if kind.endswith("64") else 32
    longest = {"fene": 500, "collapsed": 200, "rpy": 64, "vwf": 50}[model]
    beads = log(4, longest)
    replicas = log(2, 128)
    window = log(10, 200)
    windows = log(1, 12)
    uneven = rng.random() < 0.4
    # a pass of at most about 60 ms, a fifth of a second in float64 and with hydrodynamic interaction
    budget = 0.06 if model in ("fene", "collapsed") and bits == 32 else 0.1
    gradient = kind == "gradient"
    if gradient:
        windows = 2 * max(1, windows // 2)
    if model in ("rpy", "vwf"):
        window = min(window, 150)
        windows = min(windows, max(1, 150 // window))
    if bits == 64:
        windows = min(windows, max(1, 1000 // window))
    # a pass of at most about 50 ms
    size = min(2.5 * beads, 0.5 * (beads + longest)) if uneven else beads
    each = _COST[(model, bits)] * replicas * window * windows * size
    each *= size / 50.0 if model == "collapsed" else max(0.2, (size / 50.0) ** 2) if model in ("rpy", "vwf") else 1.0
    most = max(1, min(256 if gradient else 16384, int(0.05 / each)))
    return _case(model, bits, log(1, most), beads, replicas, window, windows,
                 beads_max=min(longest, 4 * beads) if uneven and beads < longest else 0,
                 replicas_min=max(1, replicas // 4) if uneven else 0,
                 per_call=0 if gradient else rng.choice([0, 0, 1]), kinetics=not gradient and rng.random() < 0.4,
                 conformation=kind == "conformation", gradient=gradient,
                 flow="none" if model == "vwf" else rng.choice(["shear", "uniaxial", "planar", "mixed"] if model == "fene" else ["shear", "none"]),
                 wi=round(math.exp(rng.uniform(0.0, math.log(20.0))), 2) if model == "fene" else 0.0)


def _table(case):
    """Per-chain parameters of a case, as a dict of arrays (the case alone decides them, not the seed)."""
    C = case["chains"]
    r = np.random.default_rng(case["beads"] * 1009 + C)
    lo, hi = case["beads"], case["beads_max"] or case["beads"]
    N = r.integers(lo, hi + 1, size=C)
    R = r.integers(case["replicas_min"], case["replicas"] + 1, size=C) if case["replicas_min"] else np.full(C, case["replicas"])
    flow = np.full(C, {"none": inputs.FLOW_NONE, "shear": inputs.FLOW_SHEAR, "uniaxial": inputs.FLOW_UNIAXIAL,
                       "planar": inputs.FLOW_PLANAR, "mixed": 0}[case["flow"]])
    if case["flow"] == "mixed":
        flow = np.where(np.arange(C) % 2 == 0, inputs.FLOW_SHEAR, inputs.FLOW_UNIAXIAL)
    t = {"N": N, "R": R, "flow": flow}
    one = np.ones(C)
    if case["model"] == "fene":
        b = r.uniform(20.0, 200.0, size=C) if case["beads_max"] else 100.0 * one
        t.update(spring=inputs.SPRING_FENE, H=one, b=b, rate=case["wi"] * 2.0 * np.sin(np.pi / (2.0 * N)) ** 2,
                 f_c=0.9 * np.sqrt(b), k0=1e-6 * one, dx=20.0 / np.sqrt(b), dt=5e-4 if case["flow"] == "planar" else 1e-3,
                 chain={})
    else:
        ch = inputs.vwf_chain(1, 50, hi=True) if case["model"] == "vwf" else inputs.collapsed_chain(1)
        same = {k: getattr(ch, k) for k in ("r0", "lj_u", "lj_sigma", "vwf_fa", "vwf_fb", "vwf_xmax")}
        same["hi_a"] = 1.0 if case["model"] in ("rpy", "vwf") else 0.0
        t.update(spring=ch.spring, H=ch.H * one, b=ch.b * one, rate=(7.5 if case["flow"] == "shear" else 0.0) * one,
                 f_c=10.0 * one, k0=(ch.k0 or 1e-4) * one, dx=(ch.dx or 0.25) * one, dt=inputs.COLLAPSED_DT, chain=same)
    return t


def _seed(seed):
    return (int(seed) * 0x9E3779B97F4A7C15 + 0x1234567) & (2 ** 63 - 1)


def _positions(case, t, seed):
    """Starting conformations [sum N][3] float64: equilibrium coils (FENE) or compact globules."""
    r = np.random.default_rng([int(seed), 77])
    N = t["N"]
    if case["model"] == "fene":
        nb = int((N - 1).sum())
        chain = np.repeat(np.arange(len(N)), N - 1)
        # p(Q) ~ (1 - H Q^2 / b)^(b / 2): H Q^2 / b is Beta(3/2, b/2 + 1), the direction uniform
        x = r.beta(1.5, t["b"][chain] / 2.0 + 1.0)
        u = r.normal(size=(nb, 3))
        q = u / np.linalg.norm(u, axis=1, keepdims=True) * np.sqrt(x * (t["b"] / t["H"])[chain])[:, None]
        first = np.cumsum(N) - N
        steps = np.zeros((int(N.sum()), 3))
        is_first = np.zeros(len(steps), dtype=bool)
        is_first[first] = True
        steps[~is_first] = q
        run = np.cumsum(steps, axis=0)
        pos = run - np.repeat(run[first], N, axis=0)
    else:
        # a few globules grown once, each chain one of them (its first beads) in an orientation of its own, with thermal bond noise
        longest = int(N.max())
        shape = inputs.Chain(n_beads=longest, n_replicas=1, spring=inputs.SPRING_HARMONIC, r0=2.0, lj_sigma=2.0)
        pool = [inputs.initial_globule(r, shape) for _ in range(min(8, len(N)))]
        a = r.normal(size=(len(N), 4))
        w, x, y, z = (a / np.linalg.norm(a, axis=1, keepdims=True)).T
        rot = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                        2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                        2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], axis=1).reshape(-1, 3, 3)
        pos = np.concatenate([pool[c % len(pool)][:n] @ rot[c].T for c, n in enumerate(N)])
        pos = pos + r.normal(scale=0.02, size=pos.shape)
    first = np.cumsum(N) - N
    return pos - np.repeat(np.add.reduceat(pos, first, axis=0) / N[:, None], N, axis=0)


def _chains(t):
    return [inputs.Chain(n_beads=int(t["N"][c]), n_replicas=int(t["R"][c]), spring=t["spring"], flow=int(t["flow"][c]),
                         H=float(t["H"][c]), b=float(t["b"][c]), rate=float(t["rate"][c]), f_c=float(t["f_c"][c]),
                         k0=float(t["k0"][c]), dx=float(t["dx"][c]), **t["chain"]) for c in range(len(t["N"]))]


def _weights(case, t, seed, device):
    """Cotangents of a training step: dL/dRSF [windows][M] and dL/dlog S [chains]."""
    g = torch.Generator().manual_seed(int(seed) + 5)
    M = int((t["N"] - 1).sum())
    return (torch.randn(case["windows"], M, generator=g, dtype=torch.float64).to(device),
            torch.randn(case["chains"], generator=g, dtype=torch.float64).to(device))


# ---------------------------------------------------------------------------------------------------------------------
# preparing and running
# ---------------------------------------------------------------------------------------------------------------------

def prepare(case, seed):
    t = _table(case)
    pos = _positions(case, t, seed)
    chains = _chains(t)
    prec = bdra.BD_PREC_FP64 if case["bits"] == 64 else bdra.BD_PREC_FP32
    dtype = torch.float64 if case["bits"] == 64 else torch.float32
    W, S = case["windows"], case["window"]
    if case["gradient"]:
        # K: the recommended thousand steps, or half the run where that is shorter
        K = S * max(1, min(1000 // S, W // 2))
        spec = RunSpec(chains=chains, dt=t["dt"], window_steps=S, n_steps=W * S, seed=_seed(seed), init_pos=pos,
                       checkpoint_steps=K, precision=prec)
        params = torch.tensor(np.stack([t["rate"], t["b"], t["H"]], axis=1), dtype=dtype, device="cuda")
        return {"case": case, "spec": spec, "params": params, "cotangents": _weights(case, t, seed, "cuda"), "dtype": dtype}
    # both criteria for FENE chains; the chains with a rest length have the Bell criterion only, as the vWF workload
    mask = inputs.CRIT_ALL if case["kinetics"] else 0
    ctx = bdra.Context(chains, t["dt"], S, _seed(seed), pos, precision=prec, max_windows=W,
                       thr_mask=mask if case["model"] == "fene" else 0, bell_mask=mask,
                       flags=bdra.BD_FLAG_CONFORMATION if case["conformation"] else 0, s_min=S_MIN,
                       stream=torch.cuda.current_stream().cuda_stream)
    state = {"case": case, "ctx": ctx, "dtype": dtype, "pos0": torch.from_numpy(pos).cuda()}

    def f64(*shape):
        return torch.zeros(shape, dtype=torch.float64, device="cuda")

    state["rsf"], state["tsf"], state["pos"] = f64(W, ctx.M), f64(W, ctx.M), f64(ctx.n_beads, 3)
    if case["kinetics"]:
        state["hazard"] = f64(3, ctx.M)
        state["first"] = torch.zeros((2, 3, ctx.M), dtype=torch.int64, device="cuda")
        state["events"] = torch.zeros((6 * ctx.M, 6), dtype=torch.int32, device="cuda")     # bd_event records, 24 bytes each
        state["survival"] = f64(len(chains), 3)
    if case["conformation"]:
        state["dbar"], state["dbead"], state["rgz"] = f64(W, int(t["R"].sum()), 3), f64(W, ctx.n_beads, 3), f64(W, len(chains))
    return state


def run(state):
    case, dtype = state["case"], state["dtype"]
    W, S = case["windows"], case["window"]
    if case["gradient"]:
        p = state["params"].detach().requires_grad_(True)
        rsf, survival = replica_averaged_run(p, state["spec"])
        torch.autograd.backward((rsf, survival), state["cotangents"])
        return {"rsf": rsf.detach().to(dtype), "survival": survival.detach().to(dtype), "grad": p.grad}
    ctx = state["ctx"]
    out = {}
    bdra.bd_set_positions(ctx.ptr, state["pos0"], 0)
    done = 0
    while done < W:
        n = case["per_call"] or W
        ctx.step(min(n, W - done) * S)
        for w in range(done, min(W, done + n)):
            ctx.replica_average(w, state["rsf"][w])
        if case["kinetics"] and case["per_call"]:
            out["n_events"] = bdra.bd_detect_events(ctx.ptr, state["events"], 6 * ctx.M, state["survival"])
        done += n
    for w in range(W):
        ctx.time_average(w, state["tsf"][w])
        if case["conformation"]:
            bdra.bd_conformation(ctx.ptr, w, state["dbar"][w], state["dbead"][w], state["rgz"][w])
    bdra.bd_get_positions(ctx.ptr, False, state["pos"])
    if case["kinetics"]:
        out["n_events"] = bdra.bd_detect_events(ctx.ptr, state["events"], 6 * ctx.M, state["survival"])
        bdra.bd_get_kinetics(ctx.ptr, state["hazard"], state["first"][0], state["first"][1])
        out["first"], out["events"] = state["first"], state["events"]
    for k in ("rsf", "tsf", "pos", "hazard", "survival", "dbar", "dbead", "rgz"):
        if k in state:
            out[k] = state[k].to(dtype)
    return out


def work(case):
    t = _table(case)
    N, R = t["N"].astype(np.float64), t["R"].astype(np.float64)
    steps = case["windows"] * case["window"]
    slots, M, beads = (N * (R + 1)).sum(), (N - 1).sum(), N.sum()
    # a bead-step: three normals (about 40 operations), spring force and update (about 45)
    flops = 85.0 * slots
    if case["model"] != "fene":
        flops += 17.0 * ((R + 1) * (N - 1) * (N - 2) / 2.0).sum()         # each Lennard-Jones pair once
    if case["model"] in ("rpy", "vwf"):
        n = 3.0 * N
        flops += ((R + 1) * (n ** 3 / 3.0 + 3.0 * n * n + 30.0 * N * (N - 1) / 2.0)).sum()   # factor, W F, L xi, pair coefficients
    flops *= steps
    if case["gradient"]:
        flops *= 3.0                                                      # the forward pass again, and the backward one
    bytes_ = 48.0 * beads + 16.0 * M * case["windows"]                    # positions in and out, two profiles a window
    if case["kinetics"]:
        bytes_ += 3 * M * 24.0
    if case["conformation"]:
        bytes_ += case["windows"] * 24.0 * (R.sum() + beads)
    return {"bytes": float(bytes_), "flops": float(flops)}


# ---------------------------------------------------------------------------------------------------------------------
# the method in plain float64
# ---------------------------------------------------------------------------------------------------------------------

def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors that hold 32-bit words."""
    lo = 0xFFFFFFFF
    k0, k1 = key & lo, (key >> 32) & lo
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & lo) ^ c1 ^ k0, p1 & lo, ((p0 >> 32) & lo) ^ c3 ^ k1, p0 & lo
        k0, k1 = (k0 + 0x9E3779B9) & lo, (k1 + 0xBB67AE85) & lo
    return c0, c1, c2, c3


def _noise(step, ids, pairs, beads, key):
    """Normals [chains][1 + 2 pairs][beads][3] of the parent and the replicas: slots 2j - 1 and 2j share the output of
    counter (bead, j, step, chain): six 21-bit uniforms, three Box-Muller pairs, three normals each; the parent is j = 0."""
    dev = ids.device
    bead = torch.arange(beads, device=dev).view(1, 1, -1)
    word = torch.arange(pairs + 1, device=dev).view(1, -1, 1)
    x = _philox(*torch.broadcast_tensors(bead, word, torch.full((1, 1, 1), step, device=dev), ids.view(-1, 1, 1)), key)
    m = [x[0] >> 11, x[1] >> 11, x[2] >> 11, x[3] >> 11, ((x[0] & 0x7FF) << 10) | (x[1] & 0x3FF), ((x[2] & 0x7FF) << 10) | (x[3] & 0x3FF)]
    u = [(v.to(torch.float64) + 0.5) / 2097152.0 for v in m]
    z = []
    for k in range(3):
        rho, th = torch.sqrt(-2.0 * torch.log(u[2 * k])), 2.0 * math.pi * u[2 * k + 1]
        z += [rho * torch.cos(th), rho * torch.sin(th)]
    z = torch.stack(z, dim=-1)
    rep = z[:, 1:].unflatten(-1, (2, 3)).permute(0, 1, 3, 2, 4).flatten(1, 2)
    return torch.cat([z[:, :1, :, :3], rep], dim=1)


class _Model:
    """Spring forces, pair forces and one Eq. 1 update of bead positions r [chains][slots][beads][3] (padded)."""

    def __init__(self, t, rows, dev):
        self.N = torch.tensor(t["N"][rows], device=dev)
        B = int(self.N.max())
        at = torch.arange(B, device=dev)
        self.bead = (at < self.N.view(-1, 1)).double().view(len(rows), 1, B, 1)
        self.spring = (at[:-1] < (self.N.view(-1, 1) - 1)).view(len(rows), 1, B - 1)
        self.kind, self.dt, self.c = t["spring"], t["dt"], t["chain"]

        def col(k):
            return torch.tensor(np.asarray(t[k][rows], dtype=np.float64), device=dev).view(-1, 1, 1)

        self.H, self.b, self.rate, self.k0, self.dx = (col(k) for k in ("H", "b", "rate", "k0", "dx"))
        flow = t["flow"][rows]
        hat = np.zeros((len(rows), 3, 3))
        hat[flow == inputs.FLOW_SHEAR, 0, 2] = 1.0
        hat[flow == inputs.FLOW_UNIAXIAL] = np.diag([1.0, -0.5, -0.5])
        hat[flow == inputs.FLOW_PLANAR] = np.diag([1.0, -1.0, 0.0])
        self.hat = torch.tensor(hat, device=dev)
        self.a2 = (at[:-1] % 2 == 0).view(1, 1, -1)
        if self.c.get("lj_u"):
            i, j = at.view(-1, 1), at.view(1, -1)
            ok = self.bead[:, 0, :, 0].bool()
            self.pair = ((i - j).abs() >= 2) & ok.view(len(rows), 1, -1, 1) & ok.view(len(rows), 1, 1, -1)
            self.off = (i != j) & ok.view(len(rows), 1, -1, 1) & ok.view(len(rows), 1, 1, -1)

    def force(self, r):
        """(spring force vectors, sampled force of each spring)."""
        Q = r[:, :, 1:] - r[:, :, :-1]
        q2 = (Q * Q).sum(-1)
        if self.kind == inputs.SPRING_FENE:
            c = self.H / torch.clamp(1.0 - self.H * q2 / self.b, min=S_MIN)
            f = c * torch.sqrt(torch.where(self.spring, q2, torch.ones_like(q2)))
        else:
            q = torch.sqrt(torch.where(self.spring, q2, torch.ones_like(q2)))
            x = q - self.c["r0"]
            f = self.H * x
            if self.kind == inputs.SPRING_VWF:
                s = torch.clamp(1.0 - x * x / self.c["vwf_xmax"] ** 2, min=S_MIN)
                f = torch.where(self.a2, self.c["vwf_fb"] * x + self.c["vwf_fa"] * x / s, f)
            c = f / q
        zero = torch.zeros((), dtype=r.dtype, device=r.device)
        return torch.where(self.spring, c, zero).unsqueeze(-1) * Q, torch.where(self.spring, f, zero)

    def step(self, r, xi):
        F, _ = self.force(r)
        pad = torch.zeros_like(F[:, :, :1])
        Fb = torch.cat([F, pad], 2) - torch.cat([pad, F], 2)
        amp = math.sqrt(0.5 * self.dt)
        hi = self.c.get("hi_a", 0.0)
        if self.c.get("lj_u"):
            d = r.unsqueeze(2) - r.unsqueeze(3)                           # [.., i, j, :] = r_j - r_i
            rr = (d * d).sum(-1)
            rr = torch.where(self.off, rr, torch.ones_like(rr))
            x6 = (self.c["lj_sigma"] ** 2 / rr) ** 3
            w = torch.where(self.pair, 12.0 * self.c["lj_u"] * (x6 - x6 * x6) / rr, torch.zeros_like(rr))
            Fb = Fb + (w.unsqueeze(-1) * d).sum(3)
            del x6, w
        if hi:
            rn = torch.sqrt(rr)
            far = rr >= 4.0 * hi * hi
            pre = 3.0 * hi / (4.0 * rn)
            ci = torch.where(far, pre * (1.0 + 2.0 * hi * hi / (3.0 * rr)), pre * rn / (2.0 * hi) * (8.0 / 3.0 - 3.0 * rn / (4.0 * hi)))
            cd = torch.where(far, pre * (1.0 - 2.0 * hi * hi / rr), pre * rn / (2.0 * hi) * rn / (4.0 * hi)) / rr
            ci = torch.where(self.off, ci, torch.zeros_like(ci))
            cd = torch.where(self.off, cd, torch.zeros_like(cd))
            B = r.shape[2]
            eye = torch.eye(3, dtype=r.dtype, device=r.device)
            Wt = ci[..., None, None] * eye + cd[..., None, None] * d.unsqueeze(-1) * d.unsqueeze(-2)
            Wt = Wt.transpose(3, 4).reshape(*r.shape[:2], 3 * B, 3 * B) + torch.eye(3 * B, dtype=r.dtype, device=r.device)
            L = torch.linalg.cholesky_ex(Wt)[0]
            drift = (Wt @ Fb.flatten(2).unsqueeze(-1)).view_as(r)
            noise = (L @ (xi * self.bead).flatten(2).unsqueeze(-1)).view_as(r)
        else:
            drift, noise = Fb, xi
        flow = self.rate.unsqueeze(-1) * torch.einsum("cde,cske->cskd", self.hat, r)
        return (r + (flow + 0.25 * drift) * self.dt + amp * noise) * self.bead


def _simulate(case, t, rows, seed, dev, params=None):
    """The run of chains `rows` (RSF, TSF, positions, hazards, Eq. 5). params: (rate, b, H) tensors to differentiate."""
    m = _Model(t, rows, dev)
    if params is not None:
        m.rate, m.b, m.H = params
    N, R = t["N"], t["R"]
    S, W, B, Rm = case["window"], case["windows"], int(N[rows].max()), int(R[rows].max())
    pairs = (Rm + 1) // 2
    pos = _positions(case, t, seed)
    first = np.cumsum(N) - N
    r0 = np.zeros((len(rows), B, 3))
    for k, c in enumerate(rows):
        r0[k, :N[c]] = pos[first[c]:first[c] + N[c]]
    reps = (torch.arange(1, Rm + 1, device=dev) <= torch.tensor(R[rows], device=dev).view(-1, 1)).double()
    nrep = reps.sum(1).view(-1, 1)
    ids = torch.tensor(rows, device=dev)
    key = _seed(seed)
    parent = torch.tensor(r0, device=dev)
    times = 1 if params is None else params[0].shape[0] // len(rows)
    parent = parent.repeat(times, 1, 1)
    out = {"rsf": [], "tsf": [], "dbar": [], "dbead": [], "rgz": []}
    hazard = torch.zeros(3, len(rows), B - 1, dtype=torch.float64, device=dev)
    if times > 1:
        m.bead, m.spring, m.hat = m.bead.repeat(times, 1, 1, 1), m.spring.repeat(times, 1, 1), m.hat.repeat(times, 1, 1)
        reps, nrep = reps.repeat(times, 1), nrep.repeat(times, 1)
    react = m.spring[:len(rows), 0] & (m.a2[0] if t["spring"] == inputs.SPRING_VWF else True)

    def add(q, f, dT):
        if case["kinetics"]:
            hazard[q] += torch.where(react, m.k0[:, 0] * torch.exp(f * m.dx[:, 0]) * dT, torch.zeros_like(f))

    def centred(r):
        return (r - r.sum(2, keepdim=True) / m.bead.sum(2, keepdim=True)) * m.bead

    for w in range(W):
        r = parent.unsqueeze(1).expand(-1, Rm + 1, -1, -1)
        start, tsum = parent, 0.0
        for s in range(S):
            xi = _noise(w * S + s, ids, pairs, B, key)[:, :Rm + 1]
            r = m.step(r, xi.repeat(times, 1, 1, 1) if times > 1 else xi)
            f = m.force(r[:, :1])[1][:, 0]
            tsum = tsum + f
            add(0, f, m.dt)
        parent = r[:, 0]
        f = (m.force(r[:, 1:])[1] * reps.unsqueeze(-1)).sum(1) / nrep
        out["rsf"].append(f)
        out["tsf"].append(tsum / S)
        add(1, tsum / S, S * m.dt)
        add(2, f, S * m.dt)
        if case["conformation"]:
            d = (centred(r[:, 1:]) - centred(start.unsqueeze(1))).abs()
            out["dbar"].append(d.sum(2) / m.bead.sum(2))
            out["dbead"].append((d * reps.view(*reps.shape, 1, 1)).sum(1) / nrep.unsqueeze(-1))
            out["rgz"].append(torch.sqrt((centred(start.unsqueeze(1))[:, 0, :, 2] ** 2).sum(1) / m.bead.sum((1, 2, 3))))
    out["hazard"], out["pos"] = hazard, centred(parent.unsqueeze(1))[:, 0]
    return out


def exact(case, seed):
    t = _table(case)
    N, R = t["N"], t["R"]
    C, steps = case["chains"], case["window"] * case["windows"]
    padded = C * (int(R.max()) + 1) * int(N.max())
    # seconds on a GPU in float64: per bead, per pair with Lennard-Jones, per tensor entry with hydrodynamic interaction
    hydro = case["model"] in ("rpy", "vwf")
    cost = padded * (2e-9 + (4e-10 * N.max() if case["model"] != "fene" else 0.0) + (4e-9 * N.max() if hydro else 0.0)) + 2e-3
    if cost * steps * (3.5 if case["gradient"] else 1.0) > 20.0:
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    size = int(R.max() + 1) * int(N.max()) * (int(N.max()) * 60 if hydro else int(N.max()) if case["model"] != "fene" else 4) * (3 if case["gradient"] else 1)
    block = max(1, int(4e8 / size))
    parts = [np.arange(C)[i:i + block] for i in range(0, C, block)]
    if case["gradient"]:
        return _exact_gradient(case, t, seed, dev, parts)
    got = [_simulate(case, t, p, seed, dev) for p in parts]

    def per_chain(key, n, of):
        """Windows (or criteria) by concatenated chains: n(c) entries of each chain, `of(part result)` [rows][chains][..]."""
        return torch.cat([x[:, k, :n(c)].reshape(len(x), n(c), *x.shape[3:]) for g, p in zip(got, parts) for x in [of(g)] for k, c in enumerate(p)], dim=1)

    def stack(k):
        return lambda g: torch.stack(g[k])

    out = {k: per_chain(k, lambda c: int(N[c]) - 1, stack(k)) for k in ("rsf", "tsf")}
    out["pos"] = per_chain("pos", lambda c: int(N[c]), lambda g: g["pos"].unsqueeze(0))[0]
    if case["kinetics"]:
        out["hazard"] = per_chain("hazard", lambda c: int(N[c]) - 1, lambda g: g["hazard"])
        out["survival"] = -torch.cat([g["hazard"].sum(2).T for g in got])
        out["first"] = out["events"] = out["n_events"] = None
    if case["conformation"]:
        out["dbar"] = per_chain("dbar", lambda c: int(R[c]), stack("dbar"))
        out["dbead"] = per_chain("dbead", lambda c: int(N[c]), stack("dbead"))
        out["rgz"] = torch.cat([torch.stack(g["rgz"]) for g in got], dim=1)
    return out


def _exact_gradient(case, t, seed, dev, parts):
    """Forward-mode derivatives in rate, b and H, the three directions as three copies of the chains."""
    import torch.autograd.forward_ad as fw

    G, gs = _weights(case, t, seed, dev)
    N, at = t["N"], np.cumsum(t["N"] - 1) - (t["N"] - 1)
    rsf, survival, grad = [], [], []
    for p in parts:
        n = len(p)
        vals = [torch.tensor(np.asarray(t[k][p], dtype=np.float64), device=dev).repeat(3).view(-1, 1, 1) for k in ("rate", "b", "H")]
        # the parameters are float32 numbers in a float32 run
        if case["bits"] == 32:
            vals = [v.float().double() for v in vals]
        tang = [torch.zeros(3 * n, 1, 1, dtype=torch.float64, device=dev) for _ in range(3)]
        for k in range(3):
            tang[k][k * n:(k + 1) * n] = 1.0
        with fw.dual_level():
            r = _simulate(case, t, p, seed, dev, [fw.make_dual(v, d) for v, d in zip(vals, tang)])
            f = [fw.unpack_dual(x) for x in r["rsf"]]
        val, dot = torch.stack([x.primal[:n] for x in f]), torch.stack([x.tangent.view(3, n, -1) for x in f])
        k0, dx = (torch.tensor(t[k][p], device=dev).view(1, -1, 1) for k in ("k0", "dx"))
        ok = torch.arange(val.shape[2], device=dev) < torch.tensor(N[p] - 1, device=dev).view(-1, 1)
        h = torch.where(ok, k0 * torch.exp(val * dx) * case["window"] * t["dt"], torch.zeros_like(val))
        g = torch.zeros_like(val)
        for k, c in enumerate(p):
            g[:, k, :N[c] - 1] = G[:, at[c]:at[c] + N[c] - 1]
        g = g - gs[torch.tensor(p, device=dev)].view(1, -1, 1) * h * dx
        grad.append((g.unsqueeze(1) * dot).sum((0, 3)).T)
        survival.append(-h.sum((0, 2)))
        rsf += [val[:, k, :N[c] - 1] for k, c in enumerate(p)]
    return {"rsf": torch.cat(rsf, dim=1), "survival": torch.cat(survival), "grad": torch.cat(grad)}
