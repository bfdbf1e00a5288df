"""The calls that a program using this package makes, as measurable cases.

A propagation is one call sequence: set_rho0, step(n), rho(0, n + 1) on a
context whose influence coefficients and mask were set once.  That is how the
package is used: the same model is propagated from several initial states, or
several models one after another, and rho(t) of every step is what comes out.
The learned surrogate has two calls, training steps and the rollout.

Sizes are those of workloads.py, bench.py and the tests; draw() spreads over
the ranges between the smallest and the largest of them.  Bath strengths,
frequencies and the bias of H_S are drawn from the seed, around the values of
workloads.py.

complex64 contexts return rho as complex64, the precision of their stored
amplitudes; FP64 contexts as complex128.
"""
from __future__ import annotations

import math
from dataclasses import replace

import numpy as np
import torch

import workloads as W


def _case(name, kind, **kw):
    return dict(name=name, kind=kind, **kw)


def listed():
    return [
        # a quick look at a short memory: latency, launches and host work
        _case("full_dk5_fp64", "full", M=2, dkmax=5, steps=40, precision="fp64", max_paths=1 << 20, engine="auto"),
        # the eight-step model of the tests and the bench over its whole length
        _case("full_dk8_c64", "full", M=2, dkmax=8, steps=100, precision="c64", max_paths=1 << 20, engine="auto"),
        # full QUAPI as the paper scales it: 2^26 stored paths once the window is full
        _case("full_dk13_c64", "full", M=2, dkmax=13, steps=30, precision="c64", max_paths=1 << 26, engine="stream"),
        # the same model in the default precision
        _case("full_dk11_fp64", "full", M=2, dkmax=11, steps=40, precision="fp64", max_paths=1 << 22,
              engine="stream"),
        # the bench's headline model: long memory, masked and filtered
        _case("structured_dk16_c64", "masked", M=2, dkmax=16, prefix=9, extra=12, log_theta=-9.0, steps=200,
              precision="c64", max_paths=1 << 22),
        # the same in the default precision
        _case("structured_dk16_fp64", "masked", M=2, dkmax=16, prefix=9, extra=12, log_theta=-9.0, steps=100,
              precision="fp64", max_paths=1 << 22),
        # the three-level chain, 1.5e7 stored paths: a large propagation
        _case("chain3_dk12_c64", "masked", M=3, dkmax=12, prefix=9, extra=0, log_theta=-10.0, steps=30,
              precision="c64", max_paths=1 << 26),
        # a mask with several coarse positions (any mask the stream layout does not take)
        _case("coarse_dk16_c64", "coarse", M=2, dkmax=16, prefix=7, extras="8,10,13", log_theta=-9.0, steps=60,
              precision="c64", max_paths=1 << 22),
        # the bench's parameter sweep: 64 instances of uneven size in one context
        _case("sweep64_c64", "sweep", n_inst=64, log_theta=-7.0, steps=100, precision="c64", max_paths=1 << 23),
        # the paper's eight-state reaction-coordinate model, keys of 96 bits, at a looser filter
        _case("wide8_dk12_c64", "wide", nvib=4, dkmax=12, prefix=9, extra=10, log_theta=-7.0, steps=20,
              precision="c64", max_paths=1 << 25),
        # training the surrogate: full-batch epochs on the windows of 48 trajectories
        _case("train_48x69", "train", n_inst=48, L=32, width=256, T=101, epochs=8),
        # the surrogate's use: 16 held-out instances extended to t = 1000
        _case("rollout_16x968", "rollout", n_inst=16, L=32, width=256, T=1000),
    ]


def draw(rng):
    kind = rng.choice(["full", "full", "masked", "masked", "chain", "chain", "coarse", "sweep", "wide", "train",
                       "rollout"])
    precision = rng.choice(["c64", "fp64"])
    if kind == "full":
        if rng.random() < 0.25:   # three levels, no mask: 9^dkmax paths
            dk = rng.randint(3, 6)
            return dict(kind="full", M=3, dkmax=dk, steps=rng.randint(20, 60), precision=precision,
                        max_paths=1 << 20, engine="auto")
        dk = rng.randint(4, 13 if precision == "c64" else 11)
        return dict(kind="full", M=2, dkmax=dk, steps=rng.randint(20, 120 if dk < 11 else 30), precision=precision,
                    max_paths=max(1 << 20, 1 << (2 * dk)), engine="auto" if dk < 11 else "stream")
    if kind == "masked":
        dk = rng.randint(9, 16)
        prefix = rng.randint(6, min(9, dk - 1))
        extra = rng.choice([0, rng.randint(prefix + 1, dk - 1) if prefix + 1 <= dk - 1 else 0])
        return dict(kind="masked", M=2, dkmax=dk, prefix=prefix, extra=extra,
                    log_theta=round(rng.uniform(-9.0, -6.5), 2), steps=rng.randint(40, 200), precision=precision,
                    max_paths=1 << 22)
    if kind == "chain":
        dk = rng.randint(6, 11)
        return dict(kind="masked", M=3, dkmax=dk, prefix=rng.randint(5, min(8, dk - 1)), extra=0,
                    log_theta=round(rng.uniform(-9.5, -7.5), 2), steps=rng.randint(16, 40), precision=precision,
                    max_paths=1 << (24 if dk < 9 else 26))
    if kind == "coarse":
        dk = rng.randint(11, 16)
        prefix = rng.randint(5, 6)
        ex = sorted(rng.sample(range(prefix + 1, dk), rng.randint(2, 3)))
        return dict(kind="coarse", M=2, dkmax=dk, prefix=prefix, extras=",".join(str(e) for e in ex),
                    log_theta=round(rng.uniform(-9.0, -7.0), 2), steps=rng.randint(30, 80), precision=precision,
                    max_paths=1 << 22)
    if kind == "sweep":
        return dict(kind="sweep", n_inst=rng.randint(5, 80), log_theta=round(rng.uniform(-8.0, -6.5), 2),
                    steps=rng.randint(30, 100), precision="c64", max_paths=1 << 23)
    if kind == "wide":
        nvib, dk = rng.choice([3, 4]), rng.randint(9, 12)
        prefix = rng.randint(7, min(9, dk - 1))
        return dict(kind="wide", nvib=nvib, dkmax=dk, prefix=prefix,
                    extra=rng.choice([0, dk - 1]) if dk - 1 > prefix else 0,
                    log_theta=round(rng.uniform(-6.5, -5.0), 2), steps=rng.randint(14, 20), precision=precision,
                    max_paths=1 << 25)
    if kind == "train":
        return dict(kind="train", n_inst=rng.randint(9, 48), L=rng.randint(16, 32), width=rng.choice([128, 192, 256]),
                    T=rng.randint(80, 101), epochs=rng.randint(4, 8))
    return dict(kind="rollout", n_inst=rng.randint(1, 48), L=rng.randint(16, 32), width=rng.choice([128, 192, 256]),
                T=rng.randint(200, 1000))


# ------------------------------------------------------------------ the models

def _model(case, seed):
    """The workload of a propagation case; seed None: the nominal values."""
    rng = np.random.default_rng(seed)

    def vary(x, by):
        return x if seed is None else float(x * math.exp(rng.uniform(-by, by)))

    theta = 10.0 ** case["log_theta"] if "log_theta" in case else 0.0
    bias = 0.0 if seed is None else float(rng.uniform(-0.3, 0.3))
    M, dk = case.get("M", 2), case.get("dkmax", 8)
    if case["kind"] == "wide":
        mask = tuple(range(case["prefix"])) + ((case["extra"],) if case["extra"] else ())
        w = W.reaction_coordinate(case["nvib"], dk, mask, theta, case["steps"])
        return replace(w, bath=replace(w.bath, ohmic_alpha=vary(w.bath.ohmic_alpha, 0.2)))
    if case["kind"] == "full":
        base = W.SPIN_BOSON_OHMIC_DK8 if dk < 10 else W.tls_ohmic_full(dk)
        bath = replace(base.bath, ohmic_alpha=vary(base.bath.ohmic_alpha, 0.2), ohmic_wc=vary(base.bath.ohmic_wc, 0.1))
        mask = None
    else:
        base = W.SPIN_BOSON_STRUCTURED_DK16
        b = base.bath
        bath = replace(b, ohmic_alpha=vary(b.ohmic_alpha, 0.1), res_w0=vary(b.res_w0, 0.1),
                       res_lambda=vary(b.res_lambda, 0.1))
        extras = [case["extra"]] if case.get("extra") else [int(e) for e in case.get("extras", "").split(",") if e]
        mask = tuple(range(case["prefix"])) + tuple(extras)
    if M == 3:
        c3 = W.CHAIN3_STRUCTURED_DK12
        base = replace(base, M=3, q=c3.q, rho0=c3.rho0, hs=c3.hs, dt=min(base.dt, c3.dt))
    hs = base.hs_array() + 0.5 * bias * np.diag(base.q)
    return replace(base, hs=tuple(tuple(complex(v) for v in row) for row in hs), bath=bath, dkmax=dk, mask=mask,
                   theta=theta)


def _models(case, seed):
    """The instances of a batched case."""
    draw_seed = W.SWEEP_SEED if seed is None else W.SWEEP_SEED + 17 * (1 + seed)
    return W.coupling_sweep(case["n_inst"], seed=draw_seed, theta=10.0 ** case["log_theta"])


def _trajectories(n, T, seed):
    """Damped oscillations of n two-level systems, [T][n][2][2], and the two
    parameters of each: what the surrogate is trained on and started from."""
    rng = np.random.default_rng(seed)
    w0, lam = rng.uniform(0.5, 2.0, n), rng.choice([0.05, 0.1, 0.2], n)
    t = 0.25 * np.arange(T)[:, None]
    env = np.exp(-0.3 * lam * t)
    z = env * np.cos((0.8 + 0.2 * w0) * t) - 0.2 * lam * (1.0 - env)
    x = -0.3 * w0 * lam * (1.0 - env)
    y = env * np.sin((0.8 + 0.2 * w0) * t) * 0.9
    rho = np.empty((T, n, 2, 2), dtype=np.complex128)
    rho[..., 0, 0], rho[..., 1, 1] = 0.5 * (1.0 + z), 0.5 * (1.0 - z)
    rho[..., 0, 1], rho[..., 1, 0] = 0.5 * (x - 1j * y), 0.5 * (x + 1j * y)
    return rho, np.stack([w0, 10.0 * lam], axis=1).astype(np.float32)


# ------------------------------------------------------------------ the calls

def prepare(case, seed):
    from paper_2506_03127_gb300 import Propagator, WidePropagator, batch_from_workloads, eta_from_bath
    kind = case["kind"]
    if kind in ("train", "rollout"):
        from paper_2506_03127_gb300.surrogate import Surrogate, rho_to_device
        s = Surrogate(L=case["L"], width=case["width"], max_batch=8192)
        s.net.init(seed, out_gain=0.1 if kind == "train" else 0.02)
        if kind == "rollout":
            rho, par = _trajectories(case["n_inst"], case["L"], seed)
            return {"case": case, "s": s, "rho": rho.transpose(1, 0, 2, 3), "par": par}
        rho, par = _trajectories(case["n_inst"], case["T"], seed)
        rho_dev, par_dev = rho_to_device(torch, rho, s.device), torch.from_numpy(par).to(s.device)
        torch.cuda.synchronize()
        x, t = s.windows(rho_dev, case["n_inst"], par_dev, 0, case["n_inst"], case["L"], case["T"])
        torch.cuda.synchronize()
        return {"case": case, "s": s, "x": x, "t": t}
    if kind == "sweep":
        ws = _models(case, seed)
        p = batch_from_workloads(ws, precision=case["precision"], max_paths=case["max_paths"])
        return {"case": case, "p": p, "rho0": ws[0].rho0_array()}
    w = _model(case, seed)
    if kind == "wide":
        p = WidePropagator(w.M, w.dkmax, w.dt, w.q, w.hs_array(), w.theta, case["precision"],
                           max_paths=case["max_paths"], max_groups=case["max_paths"] // 4)
        p.set_eta(eta_from_bath(w.bath, w.dt, w.dkmax))
        p.set_mask(w.mask)
    else:
        p = Propagator.from_workload(w, precision=case["precision"], engine=case.get("engine", "auto"),
                                     max_paths=case["max_paths"])
    return {"case": case, "p": p, "rho0": w.rho0_array()}


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        for e in range(case["epochs"]):
            state["s"].net.train_step(state["x"], state["t"], _rate(e))
        return state["s"].net.params()
    if case["kind"] == "rollout":
        return state["s"].rollout(state["rho"], state["par"], case["T"]).astype(np.complex64)
    p = state["p"]
    p.set_rho0(state["rho0"])
    p.step(case["steps"])
    rho = p.rho(0, case["steps"] + 1)
    return rho if case["precision"] == "fp64" else rho.astype(np.complex64)


def _rate(e):
    return 2e-3 * 0.998 ** e


# ------------------------------------------------------------------ the work

def work(case):
    """Propagations: every step reads the stored set and writes the next one
    (key and amplitude of each path); per child the propagator, the
    influence factor and the filter, per group the history sum.  Training:
    weights, moments and activations once per epoch, the products of the
    three layers forward and backward.  Rollout: the three layers per step."""
    kind = case["kind"]
    if kind in ("train", "rollout"):
        d, w = 8 * case["L"] + 2, case["width"]
        par = d * w + w * w + 8 * w + 2 * w + 8
        macs = d * w + w * w + 8 * w
        if kind == "train":
            rows = case["n_inst"] * (case["T"] - case["L"])
            return {"bytes": case["epochs"] * (24.0 * par + rows * (4.0 * (d + 8) + 8.0 * w)),
                    "flops": case["epochs"] * rows * (6.0 * macs - 2.0 * d * w)}
        steps = case["T"] - case["L"]
        return {"bytes": 2.0 * par + 32.0 * case["n_inst"] * case["T"], "flops": 2.0 * macs * case["n_inst"] * steps}
    counts = _plain(case, None)[1]
    ws = _models(case, None) if kind == "sweep" else [_model(case, None)]
    w = ws[0]
    entry = (16.0 if kind == "wide" else 8.0) + (8.0 if case["precision"] == "c64" else 16.0)
    M2 = w.M * w.M
    moved = sum(n_in + n_out for n_in, _, n_out in counts)
    groups = sum(g for _, g, _ in counts)
    return {"bytes": entry * moved, "flops": groups * (4.0 * w.dkmax + 22.0 * M2) + 2.0 * moved}


# ------------------------------------------------------------------ 64-bit results

def exact(case, seed):
    if case["kind"] == "train":
        return _plain_train(case, seed)
    if case["kind"] == "rollout":
        return _plain_rollout(case, seed)
    return _plain(case, seed)[0]


def _eta(bath, dt, n):
    """Influence coefficients by composite Gauss-Legendre quadrature in the
    frequency (point k on the box ((k-1) dt, k dt])."""
    edges = np.concatenate([np.linspace(0.0, 6.0, 601), np.linspace(6.0, 60.0, 109)[1:], np.linspace(60.0, 2000.0, 971)[1:]])
    x, wt = np.polynomial.legendre.leggauss(16)
    half, mid = 0.5 * np.diff(edges), 0.5 * (edges[1:] + edges[:-1])
    w, wt = (mid[:, None] + half[:, None] * x).ravel(), (half[:, None] * wt).ravel()
    J = 0.5 * np.pi * bath.ohmic_alpha * w * np.exp(-w / bath.ohmic_wc)
    if bath.res_lambda:
        W0, g = bath.res_w0, bath.res_gamma
        a = bath.res_lambda * g / (np.pi * W0 ** 2)
        J = J + 2.0 * a * w * W0 ** 4 / ((W0 ** 2 - w ** 2) ** 2 + (g * w) ** 2)
    f, coth, y = wt * J / w ** 2 / np.pi, 1.0 / np.tanh(0.5 * bath.beta * w), w * dt
    s2 = np.sin(0.5 * y) ** 2
    y2 = y * y
    small = y * y2 / 6.0 * (1 - y2 / 20.0 * (1 - y2 / 42.0 * (1 - y2 / 72.0 * (1 - y2 / 110.0))))
    lin = np.where(y < 0.1, small, y - np.sin(y))
    out = [np.sum(f * coth * 2.0 * s2) - 1j * np.sum(f * lin)]
    for d in range(1, n):
        out.append(np.sum(4.0 * f * s2 * coth * np.cos(d * y)) - 1j * np.sum(4.0 * f * s2 * np.sin(d * y)))
    return np.array(out)


def _expm(hs, dt):
    e, v = np.linalg.eigh(hs)
    return (v * np.exp(-1j * e * dt)) @ v.conj().T


def _plain(case, seed):
    """The path update in plain 64-bit torch: rho(t) of every step and, per
    step, the stored paths before, the groups and the stored paths after.
    Paths merge on the shifted mask once the window is full: the group's
    amplitudes are added and its largest path stands for it (among equal
    weights, equal to the tie window of the precision, the smallest key)."""
    batch = case["kind"] == "sweep"
    ws = _models(case, seed) if batch else [_model(case, seed)]
    w = ws[0]
    n_inst, M, dk, MM = len(ws), w.M, w.dkmax, w.M * w.M
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    i64, f64, c128 = torch.int64, torch.float64, torch.complex128
    eta = torch.tensor(np.array([_eta(v.bath, v.dt, dk) for v in ws]), dtype=c128, device=dev)
    q = torch.tensor(w.q, dtype=f64, device=dev)
    U = torch.tensor(_expm(w.hs_array(), w.dt), dtype=c128, device=dev)
    bs = max(1, (M - 1).bit_length())
    b, pt = 2 * bs, (1 << (2 * bs)) - 1
    word, st = (1 << (8 * b)) - 1, (1 << bs) - 1
    keep = {0} | {p - 1 for p in w.mask_list() if p >= 1}
    Pp, rest = sorted(keep), [p for p in range(dk) if p not in keep]
    tie = 1.0 - (1e-6 if case["precision"] == "c64" else 1e-12)

    def point(lo, hi, p):
        return ((lo >> (b * p)) if p < 8 else (hi >> (b * (p - 8)))) & pt

    def pack(lo, hi, positions):
        k = torch.zeros_like(lo)
        for i, p in enumerate(positions):
            k |= point(lo, hi, p) << (b * i)
        return k

    rho0 = w.rho0_array()
    nz = [(a, c) for a in range(M) for c in range(M) if rho0[a, c] != 0]
    lo = torch.tensor([a | (c << bs) for a, c in nz], dtype=i64, device=dev).repeat(n_inst)
    amp = torch.tensor([rho0[a, c] for a, c in nz], dtype=c128, device=dev).repeat(n_inst)
    hi = torch.zeros_like(lo)
    inst = torch.arange(n_inst, device=dev).repeat_interleave(len(nz))
    rhos, counts = [torch.tensor(rho0, device=dev).reshape(1, MM).repeat(n_inst, 1)], []
    theta2 = w.theta ** 2
    for tn in range(1, case["steps"] + 1):
        n_in = lo.numel()
        if tn >= dk:
            gk = pack(lo, hi, Pp)
            if batch:
                gk |= inst << (b * len(Pp))
            u, inv = torch.unique(gk, return_inverse=True)
            ng = u.numel()
            del gk, u
            S = torch.zeros(ng, 2, dtype=f64, device=dev).index_add_(0, inv, torch.view_as_real(amp))
            wt = amp.real ** 2 + amp.imag ** 2
            top = torch.zeros(ng, dtype=f64, device=dev).scatter_reduce_(0, inv, wt, "amax")
            tk = torch.where(wt >= tie * top[inv], pack(lo, hi, rest), (1 << 62))
            best = torch.full((ng,), (1 << 62), dtype=i64, device=dev).scatter_reduce_(0, inv, tk, "amin")
            sel = torch.nonzero((tk == best[inv]) & (tk < (1 << 62))).squeeze(1)
            rep = torch.empty(ng, dtype=i64, device=dev)
            rep[inv[sel]] = sel
            del wt, top, tk, best, sel, inv
            lo, hi, inst, amp = lo[rep], hi[rep], inst[rep], torch.view_as_complex(S)
            del rep, S
        H = torch.zeros_like(amp)
        for j in range(min(tn, dk) - 1):
            v = point(lo, hi, j)
            e = eta[inst, j + 1] if batch else eta[0, j + 1]
            H += e * q[v & st] - e.conj() * q[v >> bs]
        L = min(tn + 1, dk)
        mlo = word if L >= 8 else (1 << (b * L)) - 1
        mhi = 0 if L <= 8 else (1 << (b * (L - 8))) - 1
        par = lo & pt
        pa, pb = par & st, par >> bs
        chi = ((hi << b) | (lo >> (7 * b))) & mhi
        clo = (lo << b) & mlo
        e0 = eta[inst, 0] if batch else eta[0, 0]
        out, rho = [], torch.zeros(n_inst, MM, dtype=c128, device=dev)
        for a in range(M):
            for c in range(M):
                ch = amp * U[a, pa] * U[c, pb].conj() * torch.exp(-(q[a] - q[c]) * (H + e0 * q[a] - e0.conj() * q[c]))
                k = torch.nonzero(ch.real ** 2 + ch.imag ** 2 >= theta2).squeeze(1)
                ch, ci = ch[k], inst[k]
                if batch:
                    torch.view_as_real(rho)[:, a * M + c].index_add_(0, ci, torch.view_as_real(ch))
                else:
                    rho[0, a * M + c] = ch.sum()
                out.append((clo[k] | (a | (c << bs)), chi[k], ci, ch))
        groups = lo.numel()
        del H, par, pa, pb, chi, clo, ch, ci, k
        lo, hi, inst, amp = (torch.cat([o[i] for o in out]) for i in range(4))
        del out
        rhos.append(rho)
        counts.append((n_in, groups, lo.numel()))
    r = torch.stack(rhos).cpu().numpy()
    r = r.reshape(-1, n_inst, M, M) if batch else r.reshape(-1, M, M)
    return r, counts


def _net(case, seed, out_gain):
    """The network's initial weights (Surrogate's initialisation) in 64 bits."""
    d, w, o = 8 * case["L"] + 2, case["width"], 8
    rng = np.random.default_rng(seed)
    shapes = [rng.normal(size=(d, w)) * np.sqrt(1.0 / d), np.zeros(w), rng.normal(size=(w, w)) * np.sqrt(1.0 / w),
              np.zeros(w), rng.normal(size=(w, o)) * np.sqrt(1.0 / w) * out_gain, np.zeros(o)]
    return [torch.tensor(s.astype(np.float32).astype(np.float64)) for s in shapes]


def _features(rho):
    """[..., 2, 2] complex -> [..., 8]: (Re, Im) of rho_00, rho_01, rho_10, rho_11."""
    r = rho.reshape(rho.shape[:-2] + (4,))
    return np.stack([r.real, r.imag], axis=-1).reshape(rho.shape[:-2] + (8,))


def _plain_train(case, seed):
    n, L, T = case["n_inst"], case["L"], case["T"]
    rho, par = _trajectories(n, T, seed)
    f = _features(rho).transpose(1, 0, 2)                      # [n][T][8]
    x = np.stack([f[:, t - L:t].reshape(n, 8 * L) for t in range(L, T)], axis=1)
    x = np.concatenate([x, np.repeat(par[:, None].astype(np.float64), T - L, axis=1)], axis=2).reshape(n * (T - L), -1)
    y = ((f[:, L:] - f[:, L - 1:-1]) * 10.0).reshape(n * (T - L), 8)
    X, Y = torch.tensor(x), torch.tensor(y)
    p = _net(case, seed, 0.1)
    m, v = [torch.zeros_like(t) for t in p], [torch.zeros_like(t) for t in p]
    for e in range(case["epochs"]):
        h1 = torch.tanh(X @ p[0] + p[1])
        h2 = torch.tanh(h1 @ p[2] + p[3])
        dy = 2.0 * (h2 @ p[4] + p[5] - Y) / Y.numel()
        d2 = (dy @ p[4].T) * (1.0 - h2 * h2)
        d1 = (d2 @ p[2].T) * (1.0 - h1 * h1)
        g = [X.T @ d1, d1.sum(0), h1.T @ d2, d2.sum(0), h2.T @ dy, dy.sum(0)]
        for i in range(6):
            m[i] = 0.9 * m[i] + 0.1 * g[i]
            v[i] = 0.999 * v[i] + 0.001 * g[i] * g[i]
            p[i] = p[i] - _rate(e) * (m[i] / (1 - 0.9 ** (e + 1))) / (torch.sqrt(v[i] / (1 - 0.999 ** (e + 1))) + 1e-8)
    return torch.cat([t.reshape(-1) for t in p]).numpy()


def _plain_rollout(case, seed):
    n, L, T = case["n_inst"], case["L"], case["T"]
    rho, par = _trajectories(n, L, seed)
    f = np.zeros((n, T, 8))
    f[:, :L] = _features(rho).transpose(1, 0, 2)
    p = [t.numpy() for t in _net(case, seed, 0.02)]
    par = par.astype(np.float64)
    for t in range(L, T):
        x = np.concatenate([f[:, t - L:t].reshape(n, 8 * L), par], axis=1)
        h = np.tanh(np.tanh(x @ p[0] + p[1]) @ p[2] + p[3])
        d = (h @ p[4] + p[5]) / 10.0
        tr = 0.5 * (d[:, 0] + d[:, 6])
        r = f[:, t - 1] + d
        r[:, 0] -= tr
        r[:, 6] -= tr
        re, im = 0.5 * (r[:, 2] + r[:, 4]), 0.5 * (r[:, 3] - r[:, 5])
        c, z = 0.5 * (r[:, 0] + r[:, 6]), 0.5 * (r[:, 0] - r[:, 6])
        rad = np.sqrt(z * z + re * re + im * im)
        k = np.where((c > 0) & (rad > c), c / np.maximum(rad, 1e-300), 1.0)
        f[:, t] = np.stack([c + k * z, 0 * c, k * re, k * im, k * re, -k * im, c - k * z, 0 * c], axis=1)
    return (f[..., 0::2] + 1j * f[..., 1::2]).reshape(n, T, 2, 2)
