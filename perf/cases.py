"""Workloads that a program using this library runs, for timing it and comparing outputs.

Each case is one call pattern through the public entry points:

  run       a context advanced by `calls` calls of run(`steps`), the state read back into the
            program's own CUDA tensors, and G(t) (levels > 0) or the stress log (log_every > 0)
  batched   many small elements with their own size, length and velocity gradient in one graph launch
            per chunk, then the stress log of every element, as a flow solver takes it
  gradient  one evaluation and gradient of a G(t) fit (adjoint.GFit) from a stored start state
  noalloc   ss_run_noalloc on the caller's own device state

The parameters are the paper's (Sec. 4.1).  Start states are equilibrium samples (Sec. 3.1): Gaussian
bonds of variance kT/k_b, Poisson(N/4) springs on uniform beads, anchors with variance kT/k_s.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1106_2899_gb300 import SlipSpring
from paper_1106_2899_gb300 import _native as nat
from paper_1106_2899_gb300.adjoint import GFit, window_G

PAPER = dict(N0=4.0, Ns=0.5, zeta_s=0.1, dt=0.01, b=1.0, kT=1.0, zeta=1.0)
K_B, K_S, DT = 3.0, 6.0, 0.01
LENGTHS = (16, 24, 32, 48)  # chain lengths of the multiscale workload
OPS = 145.0  # operations of the method per bead and step (tests/golden/alg_ops.txt, equilibrium N = 32)


def _run(name, chains, beads, steps, **kw):
    c = dict(name=name, kind="run", elements=1, chains=chains, beads=beads, precision="fp32", integrator=0,
             shear=0.0, levels=24, tt=False, log_every=0, steps=steps, calls=1)
    c.update(kw)
    return c


def listed():
    return [
        # the linear-viscoelasticity workload at full size: the benchmark's ensemble, a G(t) read every 2048 steps
        _run("lve-65536x32", 65536, 32, 2048),
        # the short and the long end of the chain-length sweep of the linear viscoelasticity
        _run("lve-16384x8", 16384, 8, 2048),
        _run("lve-4096x80", 4096, 80, 2048),
        # virtual-stress share: channel TT beside the others, a ragged ensemble
        _run("virtual-16385x40", 16385, 40, 1024, tt=True),
        # viscosity growth: one ensemble per shear rate in one context, stress logs instead of the correlator
        _run("shear-6x4096x40", 4096, 40, 1000, elements=6, shear=0.1, levels=-1, log_every=100),
        # the stochastic Heun integrator, a length and size off every tile
        _run("heun-9999x27", 9999, 27, 1024, integrator=1),
        # the FP64 parity workload, and a larger odd one: reference runs in double precision
        _run("fp64-256x16", 256, 16, 1000, precision="fp64"),
        _run("fp64-3001x23", 3001, 23, 256, precision="fp64"),
        # a program that does something of its own between steps: one step per call, correlator on
        _run("stepwise-65536x32", 65536, 32, 1, calls=16),
        # coupling to a flow solver: 512 fluid elements over one interval of their velocity gradients
        dict(name="batched-512", kind="batched", elements=512, m_lo=64, m_hi=1024, steps=1000),
        # fit of (k_b, k_s, zeta) to a relaxation modulus: loss and gradient of one window
        dict(name="gradient-8192x24", kind="gradient", chains=8192, beads=24, steps=2048, every=256),
        # the smallest call: a few steps of a small ensemble on device memory the host program owns
        dict(name="noalloc-512x32", kind="noalloc", chains=512, beads=32, precision="fp32", steps=10, levels=-1,
             shear=0.01),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pad(n):
    return -(-n // 16) * 16 if n <= 64 else 128


def draw(rng):
    kind = rng.choice(["lve", "lve", "shear", "heun", "fp64", "stepwise", "batched", "gradient", "noalloc", "noalloc"])
    n = _log_int(rng, 4, 128)
    if kind == "batched":
        return dict(kind="batched", elements=_log_int(rng, 32, 512), m_lo=_log_int(rng, 16, 64),
                    m_hi=_log_int(rng, 128, 1024), steps=rng.randint(300, 1000))
    if kind == "gradient":
        n = _log_int(rng, 8, 64)
        m = min(_log_int(rng, 512, 8192), 8192 * 32 // _pad(n))
        return dict(kind="gradient", chains=m, beads=n, steps=rng.randint(600, 2048),
                    every=rng.choice([128, 200, 256]))
    if kind == "noalloc":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        levels = rng.choice([-1, 10])
        return dict(kind="noalloc", chains=_log_int(rng, 16, 2000), beads=n, precision=prec,
                    steps=_log_int(rng, 1, 100), levels=levels, shear=rng.choice([0.0, 0.05]))
    if kind == "stepwise":
        return _unnamed(_run("", _log_int(rng, 256, 65536 * 32 // _pad(n)), n, 1, calls=rng.randint(4, 16)))
    if kind == "fp64":
        return _unnamed(_run("", _log_int(rng, 64, 3001 * 32 // _pad(n)), n, rng.randint(100, 256), precision="fp64",
                             integrator=rng.choice([0, 0, 1]), shear=rng.choice([0.0, 0.05])))
    m = _log_int(rng, 512, 65536 * 32 // _pad(n))
    steps = rng.randint(300, 2048)
    if kind == "heun":
        return _unnamed(_run("", m // 2, n, steps, integrator=1, shear=rng.choice([0.0, 0.05])))
    if kind == "shear":
        e = rng.randint(1, 8)
        return _unnamed(_run("", max(64, m // e), n, steps // 100 * 100, elements=e, shear=10 ** rng.uniform(-4, -1),
                             levels=-1, log_every=100))
    return _unnamed(_run("", m if n <= 64 else m // 2, n, steps, tt=rng.random() < 0.25))


def _unnamed(c):
    return {k: v for k, v in c.items() if k != "name"}


# ------------------------------------------------------------------ inputs --
def _equilibrium(m, n, seed):
    """Equilibrium sample in the layout of set_state_dev: R [M][N][3], Z [M], S [M][zm], A [M][zm][3]."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    zm = min(n, 64)
    f8 = dict(dtype=torch.float64, device="cuda")
    q = torch.randn(m, n, 3, generator=g, **f8) * math.sqrt(1.0 / K_B)
    q[:, 0] = 0.0
    R = q.cumsum(1)
    Z = torch.poisson(torch.full((m,), n / 4.0, **f8), generator=g).clamp(max=zm).to(torch.int32)
    S = torch.randint(0, n, (m, zm), generator=g, device="cuda", dtype=torch.int64)
    A = torch.gather(R, 1, S[:, :, None].expand(-1, -1, 3)) + math.sqrt(1.0 / K_S) * torch.randn(m, zm, 3, generator=g,
                                                                                               **f8)
    empty = torch.arange(zm, device="cuda")[None, :] >= Z[:, None]
    S = torch.where(empty, -1, S).to(torch.int32)
    A[empty] = 0.0
    return R, Z, S.contiguous(), A


def _shear(case, e=0):
    """Simple shear; the elements of one context differ in rate by factors of two."""
    k = np.zeros((3, 3))
    k[0, 1] = case["shear"] / 2**e
    return k


def prepare(case, seed):
    return {"run": _prepare_run, "batched": _prepare_batched, "gradient": _prepare_gradient,
            "noalloc": _prepare_noalloc}[case["kind"]](case, seed)


def _prepare_run(c, seed):
    m, n, ne = c["chains"], c["beads"], c["elements"]
    ens = SlipSpring([(m, n)] * ne, precision=c["precision"], seed=seed,
                     stream=torch.cuda.current_stream().cuda_stream)
    kw = dict(PAPER, corr_levels=c["levels"], groups=32, integrator=c["integrator"], corr_tt=int(c["tt"]))
    if c["log_every"]:
        kw.update(log_every=c["log_every"], max_logs=c["steps"] * c["calls"] // c["log_every"] + 1)
    ens.set_params(**kw)
    out = []
    for e in range(ne):
        st = _equilibrium(m, n, seed * 16 + e)
        ens.set_state_dev(*st, elem=e)
        if c["shear"]:
            ens.set_flow(_shear(c, e), 0, elem=e)
        out.append(tuple(torch.empty_like(t) for t in st))
    return dict(case=c, ens=ens, out=out)


def _prepare_batched(c, seed):
    rng = np.random.default_rng(seed)
    ms = np.rint(np.exp(rng.uniform(math.log(c["m_lo"]), math.log(c["m_hi"]), c["elements"]))).astype(int)
    ns = rng.choice(LENGTHS, c["elements"])
    kap = rng.normal(0.0, 1e-2, (c["elements"], 3, 3))
    kap -= np.trace(kap, axis1=1, axis2=2)[:, None, None] / 3.0 * np.eye(3)
    ens = SlipSpring(list(zip(ms.tolist(), ns.tolist())), precision="fp32", seed=seed,
                     stream=torch.cuda.current_stream().cuda_stream)
    ens.set_params(**PAPER, corr_levels=-1, groups=4, log_every=100, max_logs=c["steps"] // 100 + 1, chunk_steps=1000)
    ens.set_batched(True)
    ens.set_flow_table(np.arange(c["elements"]), np.zeros(c["elements"]), kap)
    ens.run(0)
    return dict(case=c, ens=ens)


def _prepare_gradient(c, seed):
    m, n = c["chains"], c["beads"]
    ens = SlipSpring([(m, n)], precision="fp32", seed=seed, stream=torch.cuda.current_stream().cuda_stream)
    ens.set_params(**PAPER, corr_levels=14, groups=32)
    ens.set_state_dev(*_equilibrium(m, n, seed))
    start = ens.get_state()
    ens.set_coefficients(1.1 * K_B, 1.1 * K_S, 1.1)  # the target: the same window at other coefficients
    ens.window_forward(c["steps"], c["every"])
    target = window_G(ens)[0]
    ens.step = 0
    fit = GFit(ens, start, c["steps"], checkpoint_every=c["every"], target=target)
    return dict(case=c, fit=fit, theta=torch.tensor([K_B, K_S, 1.0], dtype=torch.float64))


def _prepare_noalloc(c, seed):
    m, n = c["chains"], c["beads"]
    R, Z, S, A = _equilibrium(m, n, seed)
    dt = torch.float64 if c["precision"] == "fp64" else torch.float32
    Rd, Ad, Sd = _device_layout(R, S, A, n, dt)
    p = nat.ss_params()
    for k, v in PAPER.items():
        setattr(p, k, v)
    p.corr_levels = c["levels"]
    corr = torch.zeros(max(c["levels"], 1), 16, 2, 3, dtype=torch.float64, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    return dict(case=c, lib=nat.load(), params=p, seed=seed, t0=0, R=Rd, A=Ad, S=Sd, Z=Z.contiguous(), corr=corr,
                status=status, kappa=np.ascontiguousarray(_shear(c)) if c["shear"] else None)


def _device_layout(R, S, A, n, dt):
    """R, A [M][3][NP] and S [M][NP] of ss_run_noalloc."""
    m, zm = S.shape
    Rd = torch.zeros(m, 3, _pad(n), dtype=dt, device="cuda")
    Ad = torch.zeros(m, 3, _pad(n), dtype=dt, device="cuda")
    Sd = torch.full((m, _pad(n)), -1, dtype=torch.int32, device="cuda")
    Rd[:, :, :n] = R.transpose(1, 2)
    Ad[:, :, :zm] = A.transpose(1, 2)
    Sd[:, :zm] = S
    return Rd, Ad, Sd


# -------------------------------------------------------------------- runs --
def run(state):
    return {"run": _run_run, "batched": _run_batched, "gradient": _run_gradient,
            "noalloc": _run_noalloc}[state["case"]["kind"]](state)


def _run_run(s):
    c, ens = s["case"], s["ens"]
    if c["log_every"]:
        ens.reset_observables()  # the log holds this window
    for _ in range(c["calls"]):
        ens.run(c["steps"])
    got = []
    for e, st in enumerate(s["out"]):
        R, Z, S, A = st
        ens.get_state_dev(R, Z, S, A, elem=e)
        obs = [ens.stress(e)] if c["log_every"] else []
        if c["levels"] > 0:
            obs += [ens.correlator("total", e)] + ([ens.correlator("virtual", e)] if c["tt"] else [])
        got.append({"state": st, "obs": obs})
    return got


def _run_batched(s):
    ens = s["ens"]
    ens.reset_observables()
    ens.run(s["case"]["steps"])
    got = [ens.stress(e) for e in range(len(ens.elements))]
    return {"mean": np.stack([g[1] for g in got]), "sem": np.stack([g[2] for g in got])}


def _run_gradient(s):
    theta = s["theta"].clone().requires_grad_(True)
    loss = s["fit"](theta)
    loss.backward()
    return {"loss": loss.detach(), "grad": theta.grad, "G": s["fit"].G}


def _run_noalloc(s):
    c, vp = s["case"], ctypes.c_void_p
    kap = s["kappa"].ctypes.data_as(ctypes.POINTER(ctypes.c_double)) if s["kappa"] is not None else None
    rc = s["lib"].ss_run_noalloc(
        ctypes.byref(s["params"]), nat.SS_FP64 if c["precision"] == "fp64" else nat.SS_FP32, s["seed"], c["chains"],
        c["beads"], 0, s["t0"], c["steps"], kap, vp(s["R"].data_ptr()), vp(s["A"].data_ptr()), vp(s["S"].data_ptr()),
        vp(s["Z"].data_ptr()), vp(s["corr"].data_ptr()) if c["levels"] > 0 else None, vp(s["status"].data_ptr()),
        vp(torch.cuda.current_stream().cuda_stream))
    nat.check(rc, None, "ss_run_noalloc")
    s["t0"] += c["steps"]
    return {"R": s["R"], "A": s["A"], "S": s["S"], "Z": s["Z"], "status": s["status"],
            "corr": s["corr"] if c["levels"] > 0 else None}


# -------------------------------------------------------------------- work --
def work(case):
    """Operations of the method (bead steps) and the bytes that enter and leave the call."""
    c = case
    if c["kind"] == "batched":
        lo, hi = math.log(c["m_lo"]), math.log(c["m_hi"])
        m = c["elements"] * (math.exp(hi) - math.exp(lo)) / max(hi - lo, 1e-9)  # expected chains
        n = sum(LENGTHS) / len(LENGTHS)
        return {"flops": OPS * m * n * c["steps"], "bytes": 2 * m * (12 * n + 4 * n) + 8 * 12 * c["elements"]}
    m, n = c["chains"], c["beads"]
    z = n / 4.0
    if c["kind"] == "gradient":  # the window forward, and about twice that backward
        return {"flops": 3 * OPS * m * n * c["steps"], "bytes": m * (24.0 * n + 28 * z + 4)}
    el = 8 if c["precision"] == "fp64" else 4
    state = m * (3 * el * n + (3 * el + 4) * z + 4)
    if c["kind"] == "noalloc":
        return {"flops": OPS * m * n * c["steps"], "bytes": 2 * state}
    ne, steps = c["elements"], c["steps"] * c["calls"]
    export = m * (24 * n + 28 * min(n, 64) + 4)
    return {"flops": OPS * (2 if c["integrator"] else 1) * m * n * steps * ne,
            "bytes": ne * (2 * state * c["calls"] + export)}


# ------------------------------------------------------- the method in FP64 --
# The same scheme in plain torch, for the cases whose outputs have such values: a run in double
# precision, or one of so few steps that no rounding of single precision has turned a discrete move.
_STEP, _CREATE = 1, 2


def _philox(idx, step, purpose, chain, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of counter (idx, step, purpose, chain), int64 tensors of 32-bit words."""
    mask = 0xFFFFFFFF
    c0, c1, c2, c3 = torch.broadcast_tensors(idx, torch.full_like(idx, step), torch.full_like(idx, purpose), chain)
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & mask) ^ c1 ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c3 ^ k1, p0 & mask
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c0, c1, c2, c3


def _normals(w):
    out = []
    for a, b in ((w[0], w[1]), (w[2], w[3])):
        r = torch.sqrt(-2.0 * torch.log(((a >> 8) + 1).double() / 2**24))
        th = math.pi * (2.0 * (b >> 8).double() / 2**24 - 1.0)
        out += [r * torch.cos(th), r * torch.sin(th)]
    return torch.stack(out, -1)


def _at(R, i):
    return torch.gather(R, 1, i[:, :, None].expand(-1, -1, 3))


def _force(R, S, A, occ):
    q = R[:, 1:] - R[:, :-1]
    F = torch.zeros_like(R)
    F[:, :-1] += K_B * q
    F[:, 1:] -= K_B * q
    d = torch.where(occ[:, :, None], A - _at(R, S), 0.0)
    return F.scatter_add(1, S[:, :, None].expand(-1, -1, 3), K_S * d)


def _norm_ppf(p):
    lo, hi = -40.0, 40.0
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if 0.5 * math.erfc(-mid / math.sqrt(2.0)) < p else (lo, mid)
    return 0.5 * (lo + hi)


def _steps64(case, st, seed, chain0, kap, n_steps):
    """n_steps of the scheme from st: (state, series [n][M][6] of sigma_off and (sigma + sigma_v)_off,
    {step: sigma xx, yy, zz [M][3]} of the log steps)."""
    R, Z, S, A = st
    m, n = R.shape[:2]
    zm = S.shape[1]
    S, Z = S.clamp(min=0).long(), Z.long()
    dev = R.device
    chain = torch.arange(chain0, chain0 + m, device=dev)[:, None]
    bead, slot = torch.arange(n, device=dev)[None, :], torch.arange(zm, device=dev)[None, :]
    pref, sa, cd = DT / PAPER["zeta_s"], math.sqrt(1.0 / K_S), _norm_ppf(DT / PAPER["zeta_s"])
    amp = math.sqrt(2.0 * DT)
    flow = torch.tensor(kap, device=dev) if kap is not None else None
    series, logs = [], {}
    for t in range(n_steps):
        w = _philox(bead.expand(m, n), t, _STEP, chain, seed)
        nrm = _normals(w)
        u = ((w[0] & 255) | ((w[1] & 255) << 8) | ((w[2] & 255) << 16)).double() / 2**24
        n3, u = nrm[:, :zm, 3], u[:, :zm]
        occ = slot < Z[:, None]
        F = _force(R, S, A, occ)
        fR = R @ flow.T if flow is not None else 0.0
        fA = A @ flow.T if flow is not None else 0.0
        Rn, An = R + DT * F + DT * fR + amp * nrm[:, :, :3], A + DT * fA
        if case.get("integrator"):
            F2 = _force(Rn, S, An, occ)
            gR = Rn @ flow.T if flow is not None else 0.0
            gA = An @ flow.T if flow is not None else 0.0
            Rn = R + 0.5 * DT * (F + F2) + 0.5 * DT * (fR + gR) + amp * nrm[:, :, :3]
            An = A + 0.5 * DT * (fA + gA)
        R, A = Rn, An
        # hops
        d0 = ((_at(R, S) - A) ** 2).sum(-1)

        def prob(s):
            y = (K_S / 4.0 * (((_at(R, s) - A) ** 2).sum(-1) - d0)).clamp(-40.0, 40.0)
            return (pref * 2.0 / (1.0 + torch.exp(2.0 * y))).clamp(max=0.5)

        pp = torch.where(S < n - 1, prob((S + 1).clamp(max=n - 1)), 0.0)
        pm = torch.where(S > 0, prob((S - 1).clamp(min=0)), 0.0)
        up = occ & (u < pp)
        dn = occ & ~up & (u < pp + pm)
        S = S + up.long() - dn.long()
        # creation at the ends, destruction at the ends, new slot order
        K = (zm - Z).clamp(min=1)[:, None]
        pc = (pref / (PAPER["N0"] * K.double())).clamp(max=0.5)
        at0, atN = ~occ & (u < pc), ~occ & (u >= pc) & (u < 2.0 * pc)
        dead = occ & ((S == 0) | (S == n - 1)) & (n3 < cd)
        S = torch.where(at0, 0, torch.where(atN, n - 1, S))
        if bool((at0 | atN).any()):
            xi = _normals(_philox(slot.expand(m, zm), t, _CREATE, chain, seed))[:, :, :3]
            A = torch.where((at0 | atN)[:, :, None], _at(R, S) + sa * xi, A)
        key = torch.where(occ & ~dead, 0, torch.where(at0, 1, torch.where(atN, 2, 3)))
        order = torch.argsort(key, dim=1, stable=True)
        S, A = torch.gather(S, 1, order), _at(A, order)
        Z = (key < 3).sum(1)
        occ = slot < Z[:, None]
        S, A = torch.where(occ, S, 0), torch.where(occ[:, :, None], A, 0.0)
        # stress of the new state, then the shift to the centre of mass under a flow
        q = R[:, 1:] - R[:, :-1]
        d = torch.where(occ[:, :, None], _at(R, S) - A, 0.0)
        sb = torch.stack([K_B * (q[:, :, i] * q[:, :, j]).sum(1) for i, j in ((0, 1), (0, 2), (1, 2))], -1)
        sv = torch.stack([K_S * (d[:, :, i] * d[:, :, j]).sum(1) for i, j in ((0, 1), (0, 2), (1, 2))], -1)
        if case["levels"] > 0:
            series.append(torch.cat([sb, sb + sv], 1))
        if case.get("log_every") and (t + 1) % case["log_every"] == 0:
            logs[t + 1] = torch.cat([K_B * (q * q).sum(1) - n, sb], 1)
        if flow is not None and (t + 1) % 100 == 0:
            com = R.mean(1, keepdim=True)
            R, A = R - com, torch.where(occ[:, :, None], A - com, 0.0)
    S = torch.where(slot < Z[:, None], S, -1).to(torch.int32)
    return (R, Z.to(torch.int32), S, A), torch.stack(series) if series else None, logs


def _lag_sums(x, y, levels):
    """Per chain sums [levels][16][M] over components and pairs of x(later) y(origin), multiple-tau."""
    out = torch.zeros(levels, 16, x.shape[1], 3, dtype=torch.float64, device=x.device)
    for lev in range(levels):
        n = x.shape[0]
        for k in range(0 if lev == 0 else 8, min(16, n)):
            out[lev, k] = (x[k:] * y[: n - k]).sum(0)
        x, y = (0.5 * (v[: n // 2 * 2 : 2] + v[1 : n // 2 * 2 : 2]) for v in (x, y))
    return out


def _groups(m, groups=32):
    """Group of each chain: runs of 64 chains dealt to the groups in order."""
    slices = -(-m // 64)
    g = min(groups, slices)
    return (torch.arange(m) // 64 * g // slices).cuda(), g


def _mean_sem(v):
    """Mean over chains and its standard error over groups of v [..., M]."""
    grp, g = _groups(v.shape[-1])
    size = torch.bincount(grp, minlength=g).double()
    gm = torch.zeros(*v.shape[:-1], g, dtype=torch.float64, device=v.device).index_add_(-1, grp, v) / size
    sem = gm.std(-1) / math.sqrt(g) if g > 1 else torch.zeros_like(gm[..., 0])
    return v.mean(-1).cpu().numpy(), sem.cpu().numpy()


def _modulus(x, y, levels, n_beads):
    n = x.shape[0]
    sums = _lag_sums(x, y, levels).mean(-1) / n_beads
    t, v = [], []
    for lev in range(levels):
        for k in range(0 if lev == 0 else 8, 16):
            cnt = (n >> lev) - k
            if cnt > 0:
                t.append((k << lev) * DT)
                v.append(sums[lev, k] / cnt)
    return (np.array(t),) + _mean_sem(torch.stack(v))


def exact(case, seed):
    c = case
    if c["kind"] not in ("run", "noalloc"):
        return None  # thousands of FP32 steps: discrete moves turn on rounding
    steps, m, n = c["steps"] * c.get("calls", 1), c["chains"], c["beads"]
    if (c["precision"] == "fp32" and steps > 32) or c.get("elements", 1) * steps * (2000 + m * n / 500) > 4e6:
        return None
    if c["kind"] == "noalloc":
        st, series, _ = _steps64(c, _equilibrium(m, n, seed), seed, 0, _shear(c) if c["shear"] else None, steps)
        R, A, S = _device_layout(st[0], st[2], st[3], n, torch.float64)
        corr = None
        if c["levels"] > 0:
            x, y = series[:, :, :3], series[:, :, 3:]
            parts = [_lag_sums(x, v, c["levels"]).sum(2) for v in (x, y)]
            corr = torch.stack(parts, 2)
        return {"R": R, "A": A, "S": S, "Z": st[1], "status": None, "corr": corr}
    got = []
    for e in range(c["elements"]):
        kap = _shear(c, e) if c["shear"] else None
        st, series, logs = _steps64(c, _equilibrium(m, n, seed * 16 + e), seed, e * m, kap, steps)
        obs = []
        if c["log_every"]:
            mean, sem = _mean_sem(torch.stack(list(logs.values())).transpose(1, 2))
            obs.append((np.array(list(logs), dtype=float) * DT, mean, sem))
        if c["levels"] > 0:
            x, y = series[:, :, :3], series[:, :, 3:]
            obs.append(_modulus(x, y, c["levels"], n))
            if c["tt"]:
                obs.append(_modulus(y - x, y, c["levels"], n))
        got.append({"state": st, "obs": obs})
    return got
