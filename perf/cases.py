"""The timed workloads of the library: what its users run, over the sizes they run it at.

Each case is one call (or one short run of calls) through the public Python
binding: steps of single systems in every precision form and initial guess,
the batched ensemble, the training of the learned guess, and the energy.
``listed()`` names them, ``draw(rng)`` gives others of the same ranges,
``prepare`` builds the inputs a program holds before the call, ``run`` makes
the call and ``exact`` computes the same results in plain 64-bit PyTorch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1402_3325_gb300 import ics, learned
from paper_1402_3325_gb300 import sakura as sk

GUESS = {"standard": sk.GUESS_STANDARD, "learned": sk.GUESS_LEARNED,
         "taylor": sk.GUESS_TAYLOR, "fp32": sk.GUESS_FP32}
PRECISION = {"fp64": sk.PREC_FP64, "mixed": sk.PREC_MIXED, "df64": sk.PREC_DF64}
RULE = {"literal": sk.MIXED_RULE_LITERAL, "hyp": sk.MIXED_RULE_HYP}


def _steps(name, system, n, *, form="fp64", guess="fp32", rule="hyp", order=2, steps=1,
           host=False):
    return {"name": name, "kind": "steps", "system": system, "n": n, "form": form,
            "guess": guess, "rule": rule, "order": order, "steps": steps, "host": host}


def listed():
    return [
        # a planetary system followed for many steps per call: the smallest
        # systems, where one launch runs every step
        _steps("planets_9", "planetary", 9, steps=100),
        # the 128-body cluster with a central black hole, stepped one call at
        # a time as the accuracy experiments do: launches and latency
        _steps("black_hole_128", "plummer_bh", 128, guess="taylor"),
        # an ordinary cluster run, several steps per call
        _steps("plummer_1024", "plummer", 1024, steps=8),
        # a C or numpy program's call on host arrays: default options, a
        # composed fourth-order step, a size that fills no tile evenly
        _steps("host_order4_2999", "plummer", 2999, guess="standard", order=4, host=True),
        # the large cluster around a black hole in each precision form
        _steps("black_hole_16384", "bh", 16384),
        _steps("black_hole_16384_mixed", "bh", 16384, form="mixed"),
        # the default class rule of the mixed form, which keeps nearly every
        # pair of such a cluster in 64 bits; a ragged size
        _steps("black_hole_5003_literal", "bh", 5003, form="mixed", rule="literal"),
        # a cluster with close binaries in double-word arithmetic
        _steps("binaries_16384_df64", "binaries", 16384, form="df64"),
        # the same kind of cluster with the trained initial guess
        _steps("binaries_8192_learned", "binaries", 8192, guess="learned"),
        # many planetary systems in one launch
        {"name": "ensemble_4096", "kind": "ensemble", "nsys": 4096, "n_lo": 3, "n_hi": 64,
         "sizes": 1, "guess": "fp32", "order": 2, "steps": 50},
        # training the initial-guess network: minibatches of the size its
        # training program uses
        {"name": "train_guess", "kind": "train", "samples": 131072, "batch": 8192, "epochs": 1},
        # the energy check between runs
        {"name": "energy_16384", "kind": "energy", "system": "bh", "n": 16384},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "small", "fp64", "fp64", "fp64", "mixed", "mixed", "df64", "df64",
                       "learned", "host", "ensemble", "train", "energy"])
    if kind == "small":
        c = _steps("", "planetary", rng.randint(2, 20), form=rng.choice(["fp64", "fp64", "df64"]),
                   guess=rng.choice(["fp32", "taylor", "standard"]), order=rng.choice([2, 2, 4]),
                   steps=_log_int(rng, 1, 120))
    elif kind == "ensemble":
        c = {"kind": "ensemble", "nsys": _log_int(rng, 16, 4096), "n_lo": 3,
             "n_hi": rng.randint(8, 64), "sizes": rng.randint(2, 99),
             "guess": rng.choice(["fp32", "fp32", "standard"]), "order": 2,
             "steps": _log_int(rng, 5, 50)}
    elif kind == "train":
        batch = _log_int(rng, 256, 8192)
        c = {"kind": "train", "samples": batch * rng.randint(2, 16) + rng.randint(0, batch - 1),
             "batch": batch, "epochs": 1}
    elif kind == "energy":
        c = {"kind": "energy", "system": rng.choice(["plummer", "bh"]),
             "n": _log_int(rng, 9, 16384)}
    else:
        n = _log_int(rng, 21, 16384)
        system = rng.choice(["plummer", "bh", "binaries"]) if n > 512 else \
            rng.choice(["plummer", "plummer_bh"])
        steps = rng.randint(1, 8) if n < 2048 else 1
        if kind == "host":
            n = min(n, 6000)
            c = _steps("", system, n, guess=rng.choice(["standard", "fp32"]),
                       order=rng.choice([2, 4]), steps=1, host=True)
        elif kind == "learned":
            c = _steps("", system, n, guess="learned", steps=steps)
        elif kind == "mixed":
            c = _steps("", system, n, form="mixed", rule=rng.choice(["hyp", "hyp", "literal"]),
                       steps=steps)
        elif kind == "df64":
            c = _steps("", system, n, form="df64", steps=steps)
        else:
            c = _steps("", system, n, guess=rng.choice(["fp32", "fp32", "taylor", "standard"]),
                       steps=steps)
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# inputs

def _binaries(n, seed):
    """A Plummer cluster in N-body units with a tenth of its particles in
    binaries (the orbits of ics.plummer_binaries; its exact virialisation,
    quadratic in n on the host, is left to the analytic scales)."""
    rng = np.random.default_rng(seed)
    nb = int(round(0.1 * n)) // 2
    c = ics.plummer(n - nb, seed, virial=False)
    r, v = c.r * _RSCALE, c.v * _VSCALE
    a = np.exp(rng.uniform(math.log(1e-4), math.log(1e-2), nb))
    e = np.minimum(np.sqrt(rng.uniform(0.0, 1.0, nb)), 0.999)
    inc = np.arccos(rng.uniform(-1.0, 1.0, nb))
    Om, om, Mn = rng.uniform(0.0, 2 * math.pi, (3, nb))
    rr, vv = ics.elements_to_cartesian(2.0 / n, a, e, inc, Om, om, Mn)
    r = np.concatenate([r[:nb] + 0.5 * rr, r[:nb] - 0.5 * rr, r[nb:]])
    v = np.concatenate([v[:nb] + 0.5 * vv, v[:nb] - 0.5 * vv, v[nb:]])
    p = rng.permutation(n)
    return ics.System(np.full(n, 1.0 / n), r[p], v[p], 2.0 ** -10)


_RSCALE = 3.0 * math.pi / 16.0            # Plummer scale length in N-body units
_VSCALE = math.sqrt(16.0 / (3.0 * math.pi))


def _system(case, seed):
    kind, n = case["system"], int(case["n"])
    if kind == "planetary":
        return ics.planetary(seed, n - 1)
    if kind == "plummer_bh":
        return ics.plummer_bh(n, 1e6, seed)
    if kind == "bh":
        return ics.bh_cluster(n, seed)
    if kind == "binaries":
        return _binaries(n, seed)
    s = ics.plummer(n, seed, virial=False)
    return ics.System(s.m, s.r * _RSCALE, s.v * _VSCALE, s.dt)


def _ensemble(case, seed):
    """Planetary systems packed end to end: their sizes, uniform in [n_lo,
    n_hi], belong to the case, their orbits and masses to the seed."""
    nsys = int(case["nsys"])
    sizes = np.random.default_rng(int(case["sizes"])).integers(
        int(case["n_lo"]), int(case["n_hi"]) + 1, nsys)
    seeds = np.random.default_rng(seed).integers(0, 2 ** 31 - 1, nsys)
    parts = [ics.planetary(int(a), int(b) - 1) for a, b in zip(seeds, sizes)]
    offsets = np.zeros(nsys + 1, dtype=np.int64)
    offsets[1:] = np.cumsum(sizes)
    return ics.Ensemble(np.concatenate([s.m for s in parts]),
                        np.concatenate([s.soa() for s in parts], 1), offsets,
                        np.array([s.dt for s in parts]), seeds)


def _training_set(case, seed):
    """Dimensionless pair variables as close and distant pairs of a cluster
    have them, the network's features of them, and smooth standardised
    targets with the spread of the solver's own."""
    rng = np.random.default_rng(seed)
    k = int(case["samples"])
    tp = np.exp(rng.normal(-3.0, 1.5, k))
    ep = np.sinh(rng.normal(0.0, 1.5, k))
    bp = 2.0 - np.exp(rng.normal(0.5, 1.5, k))
    q = tp * tp * (1.0 + ep * ep + np.abs(bp))
    f = np.stack([np.log(tp), np.arcsinh(ep), np.arcsinh(bp), np.tanh(ep * tp),
                  np.tanh(bp * tp * tp), q / (1.0 + q)], 1)
    t = -0.6 * f[:, 3] + 0.4 * f[:, 4] * f[:, 3] + 0.3 * np.sin(f[:, 0]) * f[:, 5] \
        + 0.05 * rng.normal(size=k)
    t = np.clip((t - t.mean()) / t.std(), -4.0, 4.0)
    params = np.concatenate([rng.normal(0, 1 / math.sqrt(6), 384), np.zeros(64),
                             rng.normal(0, 1 / 8, 4096), np.zeros(64), rng.normal(0, 1 / 8, 64),
                             np.zeros(1)])
    norm = np.concatenate([f.mean(0), f.std(0)])
    return [np.ascontiguousarray(x, dtype=np.float32) for x in (params, norm, f, t)]


def _init(case):
    stream = torch.cuda.current_stream().cuda_stream
    sk.init(torch.cuda.current_device(), stream=stream,
            precision=PRECISION[case.get("form", "fp64")],
            mixed_rule=RULE[case.get("rule", "hyp")], guess=GUESS[case.get("guess", "fp32")])
    if case.get("guess") == "learned":
        learned.load_default()


def prepare(case, seed):
    _init(case)
    kind = case["kind"]
    if kind == "train":
        return case, [torch.tensor(x, device="cuda") for x in _training_set(case, seed)]
    if kind == "ensemble":
        e = _ensemble(case, seed)
        return case, [torch.tensor(e.state, device="cuda"), torch.tensor(e.m, device="cuda"),
                      torch.tensor(e.offsets, device="cuda"), e.offsets,
                      torch.tensor(e.dt, device="cuda"),
                      torch.empty(e.state.shape, dtype=torch.float64, device="cuda")]
    s = _system(case, seed)
    if case.get("host"):
        return case, [s.soa(), np.ascontiguousarray(s.m), s.dt]
    return case, [torch.tensor(s.soa(), device="cuda"), torch.tensor(s.m, device="cuda"), s.dt]


# ---------------------------------------------------------------------------
# one pass

def run(state):
    case, d = state
    kind = case["kind"]
    if kind == "energy":
        return sk.energy(d[0], d[1])
    if kind == "train":
        params = d[0].clone()
        losses = sk.mlp_train(params, d[1], d[2], d[3], int(case["batch"]), int(case["epochs"]),
                              2e-3)
        return {"params": params, "losses": losses}
    if kind == "ensemble":
        work = d[5].copy_(d[0])  # the program's state buffer, advanced in place
        sk.step_batched(work, d[1], d[2], d[3], d[4], int(case["order"]), int(case["steps"]))
        return work
    if case["host"]:
        x = d[0].copy()
        sk.evolve_host(x, d[1], d[2], int(case["order"]), int(case["steps"]))
        return x
    x = d[0].clone()
    if case["steps"] == 1:
        sk.step(x, d[1], d[2], int(case["order"]))
    else:
        sk.evolve(x, d[1], d[2], int(case["order"]), int(case["steps"]))
    return x


def _maps(order):
    """Second-order maps in a step of this order."""
    return 1 if abs(order) <= 2 else 3 ** (order // 2 - 1)


# Operations of one pair solve: the relative state and its drift (19), r0, its
# reciprocal, r.v, v^2, beta and zeta (25), one evaluation of the four Stumpff
# functions and of F, F' and F'' (40), the correction (25), the increments
# (22) and their sums over both particles (24).
_SOLVE = 155


def work(case):
    kind = case["kind"]
    if kind == "train":
        used = (case["samples"] // case["batch"]) * case["batch"] * case["epochs"]
        return {"bytes": 28.0 * used + 8.0 * 4673, "flops": 6.0 * 4673 * used}
    if kind == "ensemble":
        lo, hi = case["n_lo"], case["n_hi"]
        sizes = range(lo, hi + 1)
        pairs = sum(n * (n - 1) / 2 for n in sizes) / len(sizes) * case["nsys"]
        total = (lo + hi) / 2 * case["nsys"]
        return {"bytes": 104.0 * total, "flops": _SOLVE * pairs * case["steps"]}
    n = case["n"]
    if kind == "energy":
        return {"bytes": 56.0 * n, "flops": 13.0 * n * (n - 1) / 2}
    return {"bytes": 104.0 * n,
            "flops": _SOLVE * n * (n - 1) / 2 * case["steps"] * _maps(case["order"])}


# ---------------------------------------------------------------------------
# the same results in 64 bits, by plain PyTorch

def _stumpff(x):
    """c0..c3 by series at the quartered argument and the doubling formulas."""
    k = int(max(0.0, math.ceil(math.log(max(float(x.abs().max()), 1e-300) / 0.1, 4.0))))
    y = x / 4.0 ** k
    c2 = torch.zeros_like(x)
    c3 = torch.zeros_like(x)
    for j in range(8, -1, -1):
        c2 = 1.0 / math.factorial(2 * j + 2) - y * c2
        c3 = 1.0 / math.factorial(2 * j + 3) - y * c3
    c0, c1 = 1.0 - y * c2, 1.0 - y * c3
    for _ in range(k):
        c3 = 0.25 * (c2 + c0 * c3)
        c2 = 0.5 * c1 * c1
        c1 = c0 * c1
        y = 4.0 * y
        c0 = 1.0 - y * c2
    return c0, c1, c2, c3


def _universal(t, r0, eta, beta, zeta):
    """Root s of r0 s + eta G2 + zeta G3 = t by safeguarded Laguerre steps;
    finished entries leave the working set."""
    s_all = t / r0
    act = torch.nonzero(t != 0).flatten()
    s = s_all[act]
    inf = torch.full_like(s, math.inf)
    pos = t[act] > 0
    lo, hi = torch.where(pos, 0.0 * s, -inf), torch.where(pos, inf, 0.0 * s)
    t, r0, eta, beta, zeta = (q[act] for q in (t, r0, eta, beta, zeta))
    for _ in range(100):
        if act.numel() == 0:
            break
        c0, c1, c2, c3 = _stumpff(beta * s * s)
        G1, G2, G3 = s * c1, s * s * c2, s * s * s * c3
        F = zeta * G3 - t + eta * G2 + r0 * s
        Fp = r0 + eta * G1 + zeta * G2
        Fpp = eta * c0 + zeta * G1
        q = F / Fp
        ds = 5.0 * q / (1.0 + 4.0 * torch.sqrt((1.0 - 1.25 * q * Fpp / Fp).abs()))
        lo, hi = torch.where(F < 0, s, lo), torch.where(F < 0, hi, s)
        sn = s - ds
        mid = torch.where(torch.isinf(hi), 2.0 * torch.maximum(lo, s),
                          torch.where(torch.isinf(lo), 2.0 * torch.minimum(hi, s),
                                      0.5 * (lo + hi)))
        fin = ds.abs() <= 4.5e-16 * s.abs()
        sn = torch.where(((sn > lo) & (sn < hi)) | fin, sn, mid)
        s_all[act] = sn
        keep = torch.nonzero(~fin).flatten()
        if keep.numel() < act.numel():
            act, s, lo, hi, t, r0, eta, beta, zeta = (
                v[keep] for v in (act, sn, lo, hi, t, r0, eta, beta, zeta))
        else:
            s = sn
    return s_all


def _pair_map(rr, vv, m, tau):
    """Increments of the second-order pair map over m (flat pair arrays)."""
    x = [a - 0.5 * tau * b for a, b in zip(rr, vv)]
    r0 = torch.sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2])
    eta = x[0] * vv[0] + x[1] * vv[1] + x[2] * vv[2]
    beta = 2.0 * m / r0 - (vv[0] * vv[0] + vv[1] * vv[1] + vv[2] * vv[2])
    zeta = m - beta * r0
    tau = tau + 0.0 * r0
    P = 2.0 * math.pi * m / beta.clamp(min=1e-300) ** 1.5
    t = torch.where((beta > 0) & (tau.abs() > P), torch.fmod(tau, P), tau)
    s = _universal(t, r0, eta, beta, zeta)
    c0, c1, c2, c3 = _stumpff(beta * s * s)
    G1, G2, G3 = s * c1, s * s * c2, s * s * s * c3
    r = r0 + eta * G1 + zeta * G2
    fm1, gmt = -G2 / r0, (t - tau) / m - G3
    fd, gdm1 = -G1 / (r0 * r), -G2 / r
    A, B = fm1 - 0.5 * tau * fd, gmt - 0.5 * tau * gdm1
    return [A * a + B * b for a, b in zip(x, vv)] + [fd * a + gdm1 * b for a, b in zip(x, vv)]


def _one_map(X, m, tau, ij=None):
    """One second-order map of state X [6, n]; tau per particle; ij: the
    ordered pairs of an ensemble, or None for all pairs of one system."""
    n = X.shape[1]
    X = X.clone()
    X[:3] += 0.5 * tau * X[3:]
    D = torch.zeros_like(X)
    if ij is not None:
        i, j = ij
        d = _pair_map([X[q][i] - X[q][j] for q in range(3)],
                      [X[q][i] - X[q][j] for q in range(3, 6)], m[i] + m[j], tau[i])
        for q in range(6):
            D[q].index_add_(0, i, m[j] * d[q])
    else:
        rows = max(1, (1 << 24) // n)
        col = torch.arange(n, device=X.device)
        for a in range(0, n, rows):
            row = torch.arange(a, min(n, a + rows), device=X.device)
            off = (row[:, None] != col[None, :]).flatten()
            i = row.repeat_interleave(n)[off]
            j = col.repeat(row.numel())[off]
            d = _pair_map([X[q][i] - X[q][j] for q in range(3)],
                          [X[q][i] - X[q][j] for q in range(3, 6)], m[i] + m[j], tau[i])
            for q in range(6):
                D[q, row] = (m[j] * d[q]).reshape(row.numel(), n - 1).sum(1) if n > 1 else 0.0
    X += D
    X[:3] += 0.5 * tau * X[3:]
    return X


def _weights(order):
    w = [1.0]
    for k in range(4, order + 1, 2):
        x1 = 1.0 / (2.0 - 2.0 ** (1.0 / (k - 1)))
        w = [x * y for x in (x1, 1.0 - 2.0 * x1, x1) for y in w]
    return w


def _exact_train(case, seed):
    params, norm, f, t = (x.astype(np.float64) for x in _training_set(case, seed))
    x = (f - norm[:6]) / norm[6:]
    W1, b1 = params[:384].reshape(64, 6).copy(), params[384:448].copy()
    W2, b2 = params[448:4544].reshape(64, 64).copy(), params[4544:4608].copy()
    W3, b3 = params[4608:4672].copy(), params[4672:].copy()
    P = [W1, b1, W2, b2, W3, b3]
    M = [np.zeros_like(p) for p in P]
    V = [np.zeros_like(p) for p in P]
    B, losses, k = int(case["batch"]), [], 0
    for _ in range(int(case["epochs"])):
        for a in range(0, x.shape[0] - B + 1, B):
            xb, tb = x[a:a + B], t[a:a + B]
            h1 = np.tanh(xb @ W1.T + b1)
            h2 = np.tanh(h1 @ W2.T + b2)
            res = h2 @ W3 + b3 - tb
            losses.append(float((res * res).mean()))
            g = 2.0 * res / B
            d2 = g[:, None] * W3 * (1.0 - h2 * h2)
            d1 = (d2 @ W2) * (1.0 - h1 * h1)
            k += 1
            for p, m, v, gr in zip(P, M, V, (d1.T @ xb, d1.sum(0), d2.T @ h1, d2.sum(0),
                                             h2.T @ g, np.array([g.sum()]))):
                m += 0.1 * (gr - m)
                v += 0.001 * (gr * gr - v)
                p -= 2e-3 * (m / (1.0 - 0.9 ** k)) / (np.sqrt(v / (1.0 - 0.999 ** k)) + 1e-8)
    return {"params": np.concatenate([p.ravel() for p in P]), "losses": np.array(losses)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    big = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if kind == "ensemble":
        e = _ensemble(case, seed)
        X, m = torch.tensor(e.state, device=big), torch.tensor(e.m, device=big)
        sizes = np.diff(e.offsets)
        i = np.repeat(np.arange(X.shape[1]), np.repeat(sizes, sizes))
        first = np.repeat(np.repeat(e.offsets[:-1], sizes), np.repeat(sizes, sizes))
        start = np.concatenate([[0], np.cumsum(np.repeat(sizes, sizes))])[:-1]
        j = np.arange(i.size) - np.repeat(start, np.repeat(sizes, sizes)) + first
        ij = [torch.tensor(q[i != j], device=big) for q in (i, j)]
        tau = torch.tensor(np.repeat(e.dt, sizes), device=big)
        for _ in range(int(case["steps"])):
            X = _one_map(X, m, tau, ij)
        return X
    s = _system(case, seed)
    n = int(case["n"])
    if n > 4096 and big.type == "cpu":
        return None
    dev = big if n > 64 else torch.device("cpu")
    X, m = torch.tensor(s.soa(), device=dev), torch.tensor(s.m, device=dev)
    if kind == "energy":
        T = 0.5 * (m * (X[3:] * X[3:]).sum(0)).sum()
        U = [torch.zeros((), dtype=torch.float64, device=dev)]
        for a in range(0, n, 1024):
            b = min(n, a + 1024)
            d = torch.sqrt(((X[:3, a:b, None] - X[:3, None, :]) ** 2).sum(0))
            w = torch.where(torch.arange(n, device=dev)[None, :] >
                            torch.arange(a, b, device=dev)[:, None], m[a:b, None] * m / d,
                            torch.zeros_like(d))
            U.append(w.sum())
        return float(T - torch.stack(U).sum())
    one = torch.ones(n, dtype=torch.float64, device=dev)
    for _ in range(int(case["steps"])):
        for w in _weights(int(case["order"])):
            X = _one_map(X, m, w * s.dt * one)
    return X.cpu().numpy() if case["host"] else X
