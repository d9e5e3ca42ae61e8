"""What the filter and smoother is used for, as cases that a timing program can run.

A case is a dict of plain values.  ``kind`` names the entry point:

``single``    one time-invariant sequence through ``ks.smooth`` (``want``: all four
              moments, the smoothed ones alone, the filter alone, or all of them
              and the marginal log-likelihood)
``varying``   the same call with one parameter set per step
``elements``  the three-call form: elements built, scanned forward, scanned back
``batch``     sequences of one state size through ``ks.smooth_batch``
``mixed``     sequences of nx = 2, 4 and 6 through ``ks.smooth_batched``
``hmm``       a discrete-state model through ``ks.hmm_smooth``

Models and measurements are simulated: ``wiener`` is the Wiener-velocity
tracking model in nx/2 axes that observes positions, ``stable`` the random
stable model F = O diag(U[0.9, 0.99]) with H ~ N(0, 1/nx).  Everything follows
from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1905_13002_gb300 as ks

DEV = "cuda"
F32, F64 = torch.float32, torch.float64
NY = {1: 1, 2: 1, 4: 2, 6: 3, 8: 4, 32: 8}


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest real call: one short track, answered at once (latency and launches)
        {"name": "track_1k", "kind": "single", "model": "wiener", "nx": 4, "T": 1024, "q": 1.0, "r": 1.0,
         "offsets": False, "want": "all"},
        # an ordinary call of an odd length with known inputs u, d
        {"name": "axis_9973_offsets", "kind": "single", "model": "wiener", "nx": 2, "T": 9973, "q": 0.7, "r": 0.3,
         "offsets": True, "want": "all"},
        # the filter alone in 3-D, an ordinary ragged length
        {"name": "filter_3d_100k", "kind": "single", "model": "wiener", "nx": 6, "T": 100003, "q": 1.6, "r": 0.5,
         "offsets": False, "want": "filter"},
        # the headline: one long track
        {"name": "track_1M", "kind": "single", "model": "wiener", "nx": 4, "T": 1 << 20, "q": 1.0, "r": 1.0,
         "offsets": False, "want": "all"},
        # the large dense state
        {"name": "dense32_64k", "kind": "single", "model": "stable", "nx": 32, "T": 65536, "q": 0.1, "r": 0.5,
         "offsets": False, "want": "all"},
        # one admitted launch of a request server: uneven requests of one size
        {"name": "requests_nx8", "kind": "batch", "model": "stable", "nx": 8, "B": 24, "lo": 64, "hi": 65536},
        # the largest: a whole fleet's tracks of three sizes in one call
        {"name": "fleet_4096", "kind": "mixed", "B": 4096, "lo": 256, "hi": 16384},
        # irregular sampling: every step has its own parameters
        {"name": "irregular_1M", "kind": "varying", "model": "wiener", "nx": 4, "T": 1 << 20},
        # a dense model with its own parameters at every step, odd length
        {"name": "varying8_20k", "kind": "varying", "model": "stable", "nx": 8, "T": 20011},
        # materialised elements, each scan called by itself
        {"name": "elements_262k", "kind": "elements", "model": "wiener", "nx": 4, "T": 262147, "q": 1.0, "r": 1.0},
        # regime switching with few states, a long sequence
        {"name": "regimes8_1M", "kind": "hmm", "K": 8, "T": 1 << 20, "stay": 0.95},
        # regime switching with many states
        {"name": "regimes32_131k", "kind": "hmm", "K": 32, "T": 131072, "stay": 0.95},
    ]


def _length(rng, lo, hi):
    return min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) | rng.randint(0, 1))


def draw(rng):
    kind = rng.choice(["single", "single", "single", "single", "batch", "batch", "mixed", "varying", "varying",
                       "elements", "hmm", "hmm"])
    if kind == "single":
        nx = rng.choice([2, 4, 4, 6, 8, 32])
        want = rng.choice(["all", "all", "smoothed", "filter", "loglik"])
        if nx <= 6 and want == "loglik":    # a track's likelihood is lost to the resolution of its far positions
            want = "all"
        return {"kind": kind, "model": "wiener" if nx <= 6 else "stable", "nx": nx,
                "T": _length(rng, 256, {8: 1 << 18, 32: 65536}.get(nx, 1 << 21)),
                "q": round(rng.uniform(0.5, 2.0), 3) if nx <= 6 else 0.1,
                "r": round(rng.uniform(0.1, 1.0), 3) if nx <= 6 else 0.5,
                "offsets": rng.random() < 0.3, "want": want}
    if kind == "batch":
        nx = rng.choice([2, 4, 6, 8])
        return {"kind": kind, "model": "wiener" if nx <= 6 else "stable", "nx": nx,
                "B": _length(rng, 2, 64 if nx == 8 else 512), "lo": 64, "hi": _length(rng, 4096, 32768)}
    if kind == "mixed":
        return {"kind": kind, "B": _length(rng, 16, 2048), "lo": 256, "hi": 16384}
    if kind == "varying":
        nx = rng.choice([2, 4, 4, 6, 8])
        return {"kind": kind, "model": "wiener" if nx <= 6 else "stable", "nx": nx,
                "T": _length(rng, 256, 65536 if nx == 8 else 1 << 20)}
    if kind == "elements":
        nx = rng.choice([2, 4, 6])
        return {"kind": kind, "model": "wiener", "nx": nx, "T": _length(rng, 1024, 1 << 19),
                "q": round(rng.uniform(0.5, 2.0), 3), "r": round(rng.uniform(0.1, 1.0), 3)}
    K = rng.choice([2, 4, 8, 8, 16, 32])
    return {"kind": kind, "K": K, "T": _length(rng, 512, {16: 1 << 19, 32: 1 << 17}.get(K, 1 << 20)),
            "stay": round(rng.uniform(0.8, 0.98), 3)}


# ---------------------------------------------------------------- models and simulated measurements (float64)
def _f32(t):
    return t.to(F32).to(F64)


def _wiener(nx, q, r, dt=0.1):
    """The Wiener-velocity model in nx/2 axes (positions first), as float32 values in float64."""
    n = nx // 2
    I, Z = np.eye(n), np.zeros((n, n))
    return {"F": np.block([[I, dt * I], [Z, I]]),
            "Q": q * np.block([[dt ** 3 / 3 * I, dt ** 2 / 2 * I], [dt ** 2 / 2 * I, dt * I]]),
            "H": np.hstack([I, Z]), "R": r * np.eye(n), "m0": np.zeros(nx), "P0": np.eye(nx)}


def _stable(nx, ny, rng, q=0.1, r=0.5):
    O, U = np.linalg.qr(rng.standard_normal((nx, nx)))
    return {"F": (O * np.sign(np.diag(U))[None, :]) * rng.uniform(0.9, 0.99, nx)[None, :], "Q": q * np.eye(nx),
            "H": rng.standard_normal((ny, nx)) / math.sqrt(nx), "R": r * np.eye(ny), "m0": np.zeros(nx), "P0": np.eye(nx)}


def _rounded(m):
    return {k: v if k in ("m0", "P0") else v.astype(np.float32).astype(np.float64) for k, v in m.items()}


class _Plain:
    """A model's arrays as attributes, the form ``ModelBatch.create`` takes."""

    def __init__(self, m):
        self.__dict__.update(m)


def _models(case, seed):
    """The models of a case's sequences, and their lengths."""
    rng = np.random.default_rng(seed)
    nx = case.get("nx", 4)
    if case["kind"] in ("single", "elements"):
        m = _wiener(nx, case["q"], case["r"]) if case["model"] == "wiener" else _stable(nx, NY[nx], rng, case["q"], case["r"])
        if case.get("offsets"):
            m["u"], m["d"] = 0.05 * rng.standard_normal(nx), rng.standard_normal(NY[nx])
            if case["model"] == "wiener":
                m["u"][nx // 2:] = 0.0
        return [_rounded(m)], [case["T"]]
    # the lengths and sizes are the case's own; models and measurements follow from the seed
    own = np.random.default_rng([case["B"], case["lo"], case["hi"]])
    lengths = np.rint(np.exp(own.uniform(math.log(case["lo"]), math.log(case["hi"]), case["B"]))).astype(int).tolist()
    if case["kind"] == "batch":
        nxs = [nx] * case["B"]
    else:
        nxs = own.choice([2, 4, 6], case["B"]).tolist()
        nxs[:3] = [2, 4, 6]
    return [_rounded(_wiener(n, rng.uniform(0.5, 2.0), rng.uniform(0.1, 1.0)) if n <= 6 else _stable(n, NY[n], rng))
            for n in nxs], lengths


def _segment_sum(x, first):
    """Running sums of x [T, n] that begin anew at each sequence; first[k]: the first step of step k's sequence."""
    c = torch.cumsum(x, 0)
    return c - (c - x)[first]


def _simulate(models, lengths, g):
    """Measurements [total, ny] (float32 values) of sequences laid end to end."""
    nx, ny = models[0]["F"].shape[0], models[0]["H"].shape[0]
    T = int(sum(lengths))
    lens = torch.tensor(lengths, device=DEV)
    seg = torch.repeat_interleave(torch.arange(len(lengths), device=DEV), lens)
    off = torch.cumsum(lens, 0) - lens
    first = off[seg]
    st = {k: torch.tensor(np.stack([m[k] for m in models]), device=DEV) for k in ("F", "Q", "H", "R")}
    u = torch.tensor(np.stack([m.get("u", np.zeros(nx)) for m in models]), device=DEV)
    d = torch.tensor(np.stack([m.get("d", np.zeros(ny)) for m in models]), device=DEV)
    x0 = torch.randn(len(models), nx, generator=g, device=DEV, dtype=F64)
    v = torch.randn(T, ny, generator=g, device=DEV, dtype=F64)
    w = torch.randn(T, nx, generator=g, device=DEV, dtype=F64)
    n = nx // 2
    if nx <= 6:     # per axis: the velocity is a running sum, the position another
        a, b, c = st["Q"][:, 0, 0], st["Q"][:, n, n], st["Q"][:, 0, n]
        l1 = a.sqrt()
        l2 = c / l1
        l3 = (b - l2 * l2).sqrt()
        wp = l1[seg, None] * w[:, :n]
        wv = l2[seg, None] * w[:, :n] + l3[seg, None] * w[:, n:]
        at = first == torch.arange(T, device=DEV)
        vel = _segment_sum(wv + u[seg, n:], first) + x0[seg, n:]
        before = torch.where(at[:, None], x0[seg, n:], torch.roll(vel, 1, 0))
        pos = _segment_sum(st["F"][seg, 0, n][:, None] * before + wp + u[seg, :n], first) + x0[seg, :n]
        y = pos
    else:           # x_k = F x_{k-1} + w_k by doubling the span summed
        x = math.sqrt(float(st["Q"][0, 0, 0])) * w + u[seg]
        x[off] += torch.einsum("bij,bj->bi", st["F"], x0)
        step, P, place = 1, st["F"].clone(), torch.arange(T, device=DEV) - first
        while step < max(lengths):
            k = torch.nonzero(place >= step).squeeze(1)
            parts = [torch.einsum("tij,tj->ti", P[seg[p]], x[p - step]) if len(models) > 1 else x[p - step] @ P[0].T
                     for p in k.split(1 << 17)]
            x[k] += torch.cat(parts)
            P = P @ P
            step *= 2
        y = torch.einsum("tij,tj->ti", st["H"][seg], x) if len(models) > 1 else x @ st["H"][0].T
    return (y + d[seg] + st["R"][seg, 0, 0][:, None].sqrt() * v).to(F32)


def _varying(case, seed):
    """One parameter set per step: the tracking model at irregular times, or a dense random model."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    nx, T = case["nx"], case["T"]
    ny = NY[nx]

    def rand(*s):
        return torch.rand(*s, generator=g, device=DEV, dtype=F64)

    def randn(*s):
        return torch.randn(*s, generator=g, device=DEV, dtype=F64)

    m = {"m0": torch.zeros(nx, device=DEV, dtype=F64), "P0": torch.eye(nx, device=DEV, dtype=F64)}
    if case["model"] == "wiener":
        n = nx // 2
        dt = torch.exp(math.log(0.02) + math.log(25.0) * rand(T))
        r = torch.exp(math.log(0.25) + math.log(16.0) * rand(T))
        I = torch.eye(n, device=DEV, dtype=F64)
        F = torch.eye(nx, device=DEV, dtype=F64).repeat(T, 1, 1)
        F[:, :n, n:] = dt[:, None, None] * I
        Q = torch.zeros(T, nx, nx, device=DEV, dtype=F64)
        Q[:, :n, :n] = (dt ** 3 / 3)[:, None, None] * I
        Q[:, :n, n:] = (dt ** 2 / 2)[:, None, None] * I
        Q[:, n:, :n] = Q[:, :n, n:]
        Q[:, n:, n:] = dt[:, None, None] * I
        H = torch.zeros(T, ny, nx, device=DEV, dtype=F64)
        H[:, :, :n] = I
        m |= {"F": _f32(F), "Q": _f32(Q), "H": _f32(H), "R": _f32(r[:, None, None] * torch.eye(ny, device=DEV, dtype=F64))}
        z, v, x0 = randn(T, nx), randn(T, ny), randn(nx)
        vel = x0[n:] + torch.cumsum(0.75 ** 0.5 * dt.sqrt()[:, None] * z[:, :n] + 0.5 * dt.sqrt()[:, None] * z[:, n:], 0)
        before = torch.cat([x0[None, n:], vel[:-1]])
        pos = x0[:n] + torch.cumsum(dt[:, None] * before + (dt ** 1.5 / 3 ** 0.5)[:, None] * z[:, :n], 0)
        y = pos + r.sqrt()[:, None] * v
    else:
        # F_k = O_k diag(U[0.9, 0.99]) with O_k a product of two reflections
        a = torch.nn.functional.normalize(randn(2, T, nx), dim=-1)
        E = torch.eye(nx, device=DEV, dtype=F64)
        O = (E - 2 * a[0, :, :, None] * a[0, :, None, :]) @ (E - 2 * a[1, :, :, None] * a[1, :, None, :])
        G, B = randn(T, nx, nx), randn(T, ny, ny)
        m |= {"F": _f32(O * (0.9 + 0.09 * rand(T, 1, nx))), "Q": _f32(0.1 * (E + G @ G.mT / nx)),
              "H": _f32(randn(T, ny, nx) / math.sqrt(nx)),
              "R": _f32(0.5 * (torch.eye(ny, device=DEV, dtype=F64) + B @ B.mT / ny)),
              "u": _f32(0.3 * randn(T, nx)), "d": _f32(0.3 * randn(T, ny))}
        # the states of a stable model forget their past: draw them from blocks of steps run side by side
        w = (torch.linalg.cholesky(m["Q"]) @ randn(T, nx, 1)).squeeze(-1) + m["u"]
        L, lead = 512, 512
        starts = torch.arange(0, T, L, device=DEV)
        x, out = torch.zeros(len(starts), nx, device=DEV, dtype=F64), torch.zeros(T + 1, nx, device=DEV, dtype=F64)
        for i in range(-lead, L):
            k = starts + i
            kc = k.clamp(0, T - 1)
            x = torch.where((k >= 0)[:, None], torch.einsum("bij,bj->bi", m["F"][kc], x) + w[kc], x)
            if i >= 0:
                out[torch.where(k < T, k, T)] = x
        y = torch.einsum("tij,tj->ti", m["H"], out[:T]) + m["d"]
        y = y + (torch.linalg.cholesky(m["R"]) @ randn(T, ny, 1)).squeeze(-1)
    return m, y.to(F32)


def _hmm(case, seed):
    rng = np.random.default_rng(seed)
    K, T, stay, sigma = case["K"], case["T"], case["stay"], 0.6
    Pi = np.zeros((K, K))
    for i in range(K):
        Pi[i, [j for j in range(K) if j != i]] = (1 - stay) * rng.dirichlet(np.ones(K - 1))
        Pi[i, i] = stay
    Pi = (Pi / Pi.sum(1, keepdims=True)).astype(np.float32)
    g = torch.Generator(device=DEV).manual_seed(seed)
    # regimes last a geometric number of steps; the next one is drawn anew
    jump = torch.rand(T, generator=g, device=DEV, dtype=F64) >= stay
    state = torch.randint(0, K, (T + 1,), generator=g, device=DEV)[torch.cumsum(jump, 0)]
    y = state + sigma * torch.randn(T, generator=g, device=DEV, dtype=F64)
    lik = torch.exp(-0.5 * ((y[:, None] - torch.arange(K, device=DEV)) / sigma) ** 2) / (sigma * math.sqrt(2 * math.pi))
    return np.full(K, 1 / K, np.float32), Pi, lik.to(F32).contiguous()


# ---------------------------------------------------------------- prepare and run
def prepare(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    kind = case["kind"]
    if kind == "hmm":
        pi, Pi, lik = _hmm(case, seed)
        ws = _hmm_workspace(case["K"], case["T"])
        return {"case": case, "model": ks.HmmModel.create(pi, Pi), "lik": lik, "ws": ws}
    if kind == "varying":
        m, y = _varying(case, seed)
        model = ks.Model.create(m["F"], m["Q"], m["H"], m["R"], m["m0"], m["P0"], u=m.get("u"), d=m.get("d"))
        return {"case": case, "model": model, "y": y.contiguous(), "ws": ks.alloc_workspace(model, case["T"], ks.KS_WS_ELEMENTS)}
    models, lengths = _models(case, seed)
    if kind in ("single", "elements"):
        m = models[0]
        model = ks.Model.create(m["F"], m["Q"], m["H"], m["R"], m["m0"], m["P0"], u=m.get("u"), d=m.get("d"))
        purpose = ks.KS_WS_ELEMENTS if kind == "elements" or case["want"] == "smoothed" else ks.KS_WS_SMOOTH
        return {"case": case, "model": model, "y": _simulate(models, lengths, g),
                "ws": ks.alloc_workspace(model, case["T"], purpose)}
    groups = []
    for nx in sorted({m["F"].shape[0] for m in models}):
        at = [i for i, m in enumerate(models) if m["F"].shape[0] == nx]
        ms, ls = [models[i] for i in at], [lengths[i] for i in at]
        groups.append((ks.ModelBatch.create([_Plain(m) for m in ms], ls), _simulate(ms, ls, g)))
    if kind == "batch":
        batch, y = groups[0]
        nbytes = ks.workspace_bytes_batch(batch.nx, batch.ny, batch.B, int(y.shape[0]))
        return {"case": case, "batch": batch, "y": y, "ws": torch.zeros(nbytes, dtype=torch.uint8, device=DEV)}
    nbytes = ks.workspace_bytes_batched([(b.nx, b.ny, b.B, int(y.shape[0])) for b, y in groups])
    return {"case": case, "groups": groups, "ws": torch.zeros(nbytes, dtype=torch.uint8, device=DEV)}


def _hmm_workspace(K, T):
    return torch.zeros(ks.hmm_workspace_bytes(K, T), dtype=torch.uint8, device=DEV)


def run(s):
    kind = s["case"]["kind"]
    if kind == "single":
        want = s["case"]["want"]
        if want == "smoothed":
            return list(ks.smooth(s["model"], s["y"], s["ws"], keep_filtered=False)[2:])
        if want == "filter":
            return list(ks.smooth(s["model"], s["y"], s["ws"], filter_only=True)[:2])
        out = list(ks.smooth(s["model"], s["y"], s["ws"]))
        if want == "loglik":
            out += list(ks.loglik(s["model"], s["y"], out[0], out[1])[:2])
        return out
    if kind == "varying":
        return list(ks.smooth(s["model"], s["y"], s["ws"]))
    if kind == "elements":
        ks.build_elements(s["model"], s["y"], s["ws"])
        fmean, fcov = ks.filter_scan(s["model"], int(s["y"].shape[0]), s["ws"])
        return [fmean, fcov, *ks.smooth_scan(s["model"], fmean, fcov, s["ws"])]
    if kind == "batch":
        return list(ks.smooth_batch(s["batch"], s["y"], s["ws"]))
    if kind == "mixed":
        return [list(o) for o in ks.smooth_batched(s["groups"], s["ws"])]
    return list(ks.hmm_smooth(s["model"], s["lik"], s["ws"])[:3])


# ---------------------------------------------------------------- the work no path can do without
def _per_step(nx, ny):
    """Sequential filter and smoother: (filter flops, smoother flops) of one step."""
    n, m = nx, ny
    f = 4 * n ** 3 + 4 * n * n * m + 4 * n * m * m + 2 * m ** 3 // 3 + 2 * n * n + 4 * n * m
    return f, 6 * n ** 3 + 2 * n ** 3 // 3 + 4 * n * n


def work(case):
    kind = case["kind"]
    if kind == "hmm":
        K, T = case["K"], case["T"]
        return {"bytes": 4 * T * (3 * K + 1), "flops": T * (8 * K * K + 8 * K)}
    if kind in ("single", "elements", "varying"):
        sizes = [(case["nx"], case["T"])]
    else:
        lo, hi = case["lo"], case["hi"]
        total = int(case["B"] * (hi - lo) / math.log(hi / lo))      # the expected total of log-uniform lengths
        sizes = [(case["nx"], total)] if kind == "batch" else [(n, total // 3) for n in (2, 4, 6)]
    nbytes = flops = 0
    for nx, T in sizes:
        ny = NY[nx]
        moments = {"filter": 1, "smoothed": 1}.get(case.get("want"), 2)
        nbytes += 4 * T * (ny + moments * (nx + nx * nx))
        if kind == "varying":
            nbytes += 4 * T * (2 * nx * nx + ny * nx + ny * ny + (nx + ny if case["model"] == "stable" else 0))
        if case.get("want") == "loglik":
            nbytes += 4 * T
        f, s = _per_step(nx, ny)
        flops += T * (f if case.get("want") == "filter" else f + s)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits
def _blocks(lengths, chunk, lead):
    """Blocks of at most `chunk` steps that run side by side, each begun `lead` steps early: the filter and the
    smoother forget what lies that far away.  (sequence, first step within it, steps) of each."""
    return [(i, s, min(chunk, n - s)) for i, n in enumerate(lengths) for s in range(0, n, chunk)]


def _kalman64(par, off, lengths, y, nx, ny, lead, chunk, loglik=False):
    """Filter and smoother in float64; par(name, seq, step) gives the parameters of steps [blocks]."""
    T = int(sum(lengths))
    blocks = _blocks(lengths, chunk, lead)
    seq = torch.tensor([b[0] for b in blocks], device=DEV)
    s0 = torch.tensor([b[1] for b in blocks], device=DEV)
    cnt = torch.tensor([b[2] for b in blocks], device=DEV)
    base = torch.tensor(off, device=DEV)[seq]
    n_seq = torch.tensor(lengths, device=DEV)[seq]
    most = int(cnt.max())
    fm, fP = (torch.empty(T + 1, *s, device=DEV, dtype=F64) for s in ((nx,), (nx, nx)))
    sm, sP = torch.empty_like(fm), torch.empty_like(fP)
    ll = torch.zeros(T + 1, device=DEV, dtype=F64)
    m, P = par("m0", seq, None).clone(), par("P0", seq, None).clone()
    for i in range(-lead, most):
        k = s0 + i
        on = (k >= 0) & (i < cnt)
        kc = torch.minimum(k.clamp(min=0), n_seq - 1)
        F, Q, H, R = (par(v, seq, kc) for v in "FQHR")
        mp = torch.einsum("bij,bj->bi", F, m) + par("u", seq, kc)
        Pp = F @ P @ F.mT + Q
        HP = H @ Pp
        S = HP @ H.mT + R
        e = y[base + kc].to(F64) - torch.einsum("bij,bj->bi", H, mp) - par("d", seq, kc)
        L = torch.linalg.cholesky(S)
        X = torch.linalg.solve_triangular(L, torch.cat([HP, e[:, :, None]], 2), upper=False)
        G, z = X[:, :, :nx], X[:, :, nx]
        m1 = mp + torch.einsum("bji,bj->bi", G, z)
        P1 = Pp - G.mT @ G
        m = torch.where(on[:, None], m1, m)
        P = torch.where(on[:, None, None], 0.5 * (P1 + P1.mT), P)
        if i >= 0:
            at = torch.where(on, base + kc, T)
            fm[at], fP[at] = m, P
            if loglik:
                ll[at] = -0.5 * (z * z).sum(1) - torch.log(torch.diagonal(L, dim1=1, dim2=2)).sum(1) - 0.5 * ny * math.log(2 * math.pi)
    m = P = None
    for i in range(most + lead - 1, -1, -1):
        k = s0 + i
        last = k >= n_seq - 1
        kc = torch.minimum(k, n_seq - 1)
        kn = torch.minimum(k + 1, n_seq - 1)
        fk, Fk = fm[base + kc], fP[base + kc]
        if m is None:
            m, P = fk, Fk
        F, Q = par("F", seq, kn), par("Q", seq, kn)
        Pp = F @ Fk @ F.mT + Q
        G = torch.linalg.solve(Pp, F @ Fk).mT
        m1 = fk + torch.einsum("bij,bj->bi", G, m - torch.einsum("bij,bj->bi", F, fk) - par("u", seq, kn))
        P1 = Fk + G @ (P - Pp) @ G.mT
        m = torch.where(last[:, None], fk, m1)
        P = torch.where(last[:, None, None], Fk, 0.5 * (P1 + P1.mT))
        at = torch.where((k < n_seq) & (i < cnt), base + kc, T)
        sm[at], sP[at] = m, P
    return fm[:T], fP[:T], sm[:T], sP[:T], ll[:T]


def _exact_group(models, lengths, y, loglik=False):
    nx, ny = models[0]["F"].shape[0], models[0]["H"].shape[0]
    st = {k: torch.tensor(np.stack([np.asarray(m.get(k, np.zeros({"u": nx, "d": ny}.get(k, 1)))) for m in models]), device=DEV)
          for k in ("F", "Q", "H", "R", "u", "d", "m0", "P0")}
    off = np.concatenate([[0], np.cumsum(lengths)])[:-1].tolist()
    lead = 1024 if nx <= 6 else 2048
    chunk = 1024 if nx <= 6 else 2048
    return _kalman64(lambda v, seq, k: st[v][seq], off, lengths, y, nx, ny, lead, chunk, loglik)


def exact(case, seed):
    kind = case["kind"]
    if kind == "hmm":
        return _exact_hmm(case, seed)
    if kind == "varying":
        m, y = _varying(case, seed)
        nx, T = case["nx"], case["T"]
        ny = NY[nx]
        zero = {"u": torch.zeros(T, nx, device=DEV, dtype=F64), "d": torch.zeros(T, ny, device=DEV, dtype=F64)}
        m = {**zero, **m}

        def par(v, seq, k):
            return m[v].expand(len(seq), *m[v].shape) if k is None else m[v][k]

        return list(_kalman64(par, [0], [T], y, nx, ny, 1024, 1024)[:4])
    g = torch.Generator(device=DEV).manual_seed(seed)
    models, lengths = _models(case, seed)
    if kind in ("single", "elements"):
        y = _simulate(models, lengths, g)
        fm, fP, sm, sP, ll = _exact_group(models, lengths, y, case.get("want") == "loglik")
        return {"filter": [fm, fP], "smoothed": [sm, sP],
                "loglik": [fm, fP, sm, sP, ll, ll.sum().reshape(1)]}.get(case.get("want"), [fm, fP, sm, sP])
    out = []
    for nx in sorted({m["F"].shape[0] for m in models}):
        at = [i for i, m in enumerate(models) if m["F"].shape[0] == nx]
        ms, ls = [models[i] for i in at], [lengths[i] for i in at]
        out.append(list(_exact_group(ms, ls, _simulate(ms, ls, g))[:4]))
    return out[0] if kind == "batch" else out


def _exact_hmm(case, seed):
    pi, Pi, lik = _hmm(case, seed)
    K, T = case["K"], case["T"]
    Pi, lik = torch.tensor(Pi, device=DEV).to(F64), lik.to(F64)
    lead = chunk = 1024
    blocks = _blocks([T], chunk, lead)
    s0 = torch.tensor([b[1] for b in blocks], device=DEV)
    p = torch.tensor(pi, device=DEV).to(F64).expand(len(blocks), K).clone()
    filt, smooth = (torch.empty(T + 1, K, device=DEV, dtype=F64) for _ in range(2))
    inc = torch.zeros(T + 1, device=DEV, dtype=F64)
    for i in range(-lead, chunk):
        k = s0 + i
        on = (k >= 0) & (k < T)
        w = (p @ Pi) * lik[k.clamp(0, T - 1)]
        c = w.sum(1)
        p = torch.where(on[:, None], w / c[:, None], p)
        if i >= 0:
            at = torch.where(on, k, T)
            filt[at], inc[at] = p, torch.log(c)
    b = torch.ones(len(blocks), K, device=DEV, dtype=F64)
    for i in range(chunk + lead - 1, -1, -1):
        k = s0 + i
        b1 = (b * lik[(k + 1).clamp(max=T - 1)]) @ Pi.T
        b = torch.where((k + 1 < T)[:, None], b1 / b1.sum(1, keepdim=True), b)
        if i < chunk:
            w = filt[k.clamp(max=T - 1)] * b
            smooth[torch.where(k < T, k, T)] = w / w.sum(1, keepdim=True)
    return [filt[:T], smooth[:T], torch.cumsum(inc[:T], 0)]
