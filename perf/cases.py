"""Performance cases: the calls a user of the library makes, from one small
estimate to a greedy step over fifty processes.

``listed()`` names twelve of them, ``draw(rng)`` gives more of the same ranges.
Every call goes through the package's public functions with its default
context, as a program that infers a network does.  Inputs are device tensors
made from the seed alone, except the screen's training data, which its entry
point takes from host memory.

Sizes come from the repository's own workloads (``bench.py``, ``synth.py``,
``screen_train.py``) and tests: the Gaussian problem at N = 10^3 and 10^4, the
10-node VAR(5) and 50-node VAR(3) networks, the uneven batch, the logistic
chain of 50 x 1997 samples, batches of 256 rows for the screen.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_1807_10459_gb300 as idtx
from paper_1807_10459_gb300 import synth

DEV = "cuda:0"


# ------------------------------------------------------------------ cases
def listed():
    return [
        # One estimate without surrogates: an exploratory call, where latency counts.
        dict(name="cmi_one", kind="cmi", n=1000, dx=1, dy=1, dz=2, k=4, n_surr=0),
        # The same problem tested against 100 surrogates (the small Gaussian workload).
        dict(name="cmi_1k", kind="cmi", n=1000, dx=1, dy=1, dz=2, k=4, n_surr=100),
        # The same at N = 10^4: one link of a network tested on its own.
        dict(name="cmi_10k", kind="cmi", n=10000, dx=1, dy=1, dz=2, k=4, n_surr=100),
        # No condition: mutual information of two variables against surrogates.
        dict(name="mi_3k", kind="cmi", n=3001, dx=1, dy=1, dz=0, k=4, n_surr=200),
        # Two-dimensional source, another k, per-sample eps and counts wanted.
        dict(name="cmi_counts_k7", kind="cmi", n=2503, dx=2, dy=1, dz=3, k=7, n_surr=20),
        # The first greedy step of a target in the 10-node network (the headline workload).
        dict(name="step_var10", kind="step", net="var10", T=10000, past=3, lags=5, chosen=0,
             n_surr=200, screened=False),
        # A late greedy step in the 50-node network: three parents chosen, six conditions.
        dict(name="step_var50_late", kind="step", net="var50", T=5000, past=3, lags=3, chosen=3,
             n_surr=200, screened=False),
        # The same network's first step with the shipped screen.
        dict(name="step_var50_screened", kind="step", net="var50", T=5000, past=3, lags=3,
             chosen=0, n_surr=200, screened=True),
        # Pruning a selected parent set: every parent given the others, one batch per round.
        dict(name="prune_var10", kind="prune", T=10000, past=3, lags=5, parents=5, n_surr=200),
        # Many uneven problems in one call.
        dict(name="batch_uneven", kind="batch", problems=16, n_min=2000, n_max=50000, dz_max=8,
             n_surr=100),
        # Many replications of a nonlinear system, joint dimension 12, N near 10^5.
        dict(name="logistic_100k", kind="logistic", reps=50, length=2000, dz=10, n_surr=200,
             rep_level=False),
        # Two epochs of the screen's training (forward, backward and update per batch).
        dict(name="screen_train", kind="train", rows=4096, batch=256, epochs=2, quantile=0.99),
    ]


def _logint(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    kind = rng.choice(["cmi", "cmi", "cmi", "step", "step", "prune", "batch", "logistic",
                       "train"])
    if kind == "cmi":
        n = _logint(rng, 300, 20000)
        return dict(kind=kind, n=n, dx=rng.choice([1, 1, 1, 2]), dy=rng.choice([1, 1, 2]),
                    dz=rng.randint(0, 8), k=rng.choice([4, 4, 4, 3, 7]),
                    n_surr=min(_logint(rng, 1, 300), 2000000 // n))
    if kind == "step":
        net = rng.choice(["var10", "var50"])
        return dict(kind=kind, net=net, T=_logint(rng, 900, 10000 if net == "var10" else 5000),
                    past=rng.randint(1, 3), lags=rng.randint(2, 5 if net == "var10" else 3),
                    chosen=rng.randint(0, 3), n_surr=rng.randint(40, 200),
                    screened=rng.random() < 0.4)
    if kind == "prune":
        return dict(kind=kind, T=_logint(rng, 900, 10000), past=rng.randint(1, 3),
                    lags=rng.randint(3, 5), parents=rng.randint(2, 5),
                    n_surr=rng.randint(40, 200))
    if kind == "batch":
        return dict(kind=kind, problems=rng.randint(2, 16), n_min=_logint(rng, 300, 2000),
                    n_max=_logint(rng, 3000, 50000), dz_max=rng.randint(2, 8),
                    n_surr=rng.randint(20, 100))
    if kind == "logistic":
        return dict(kind=kind, reps=rng.randint(5, 50), length=rng.randint(300, 2000),
                    dz=rng.randint(4, 10), n_surr=rng.randint(20, 200),
                    rep_level=rng.random() < 0.4)
    return dict(kind=kind, rows=_logint(rng, 700, 8000), batch=rng.choice([64, 100, 256, 512]),
                epochs=rng.randint(1, 2), quantile=rng.choice([0.0, 0.99]))


# ------------------------------------------------------------------ inputs
def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _gaussian(n, dx, dy, dz, seed):
    """Jointly Gaussian columns with a random covariance, standardised."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    d = dx + dy + dz
    a = torch.from_numpy(np.random.default_rng(seed).standard_normal((d, d))).to(DEV)
    chol = torch.linalg.cholesky(a @ a.T + 0.5 * torch.eye(d, dtype=torch.float64, device=DEV))
    s = chol @ torch.randn(d, n, generator=gen, dtype=torch.float64, device=DEV)
    s = ((s - s.mean(1, keepdim=True)) / s.std(1, keepdim=True)).float()
    return s[:dx].contiguous(), s[dx:dx + dy].contiguous(), s[dx + dy:].contiguous()


# (map, lag) of the logistic chain's conditioning columns, in order of use
_CHAIN_Z = [(3, 1), (3, 2), (0, 1), (1, 2), (2, 2), (0, 2), (0, 3), (3, 3), (1, 3), (2, 3)]


def _logistic(n_reps, length, dx, dy, dz, seed):
    """Four noisy logistic maps coupled along a chain, embedded and with their
    replications concatenated: N = n_reps * (length - 3)."""
    rng = np.random.default_rng(seed)
    x = rng.uniform(0.05, 0.95, (n_reps, 4))
    out = np.empty((length, n_reps, 4))
    for t in range(-200, length):
        f = 4.0 * x * (1.0 - x)
        nxt = 0.9 * f + 0.1 * np.concatenate([f[:, :1], f[:, :3]], axis=1)
        nxt = np.abs(nxt + 0.01 * rng.standard_normal((n_reps, 4)))
        x = np.clip(np.where(nxt > 1.0, 2.0 - nxt, nxt), 0.0, 1.0)
        if t >= 0:
            out[t] = x
    maps = torch.from_numpy(out).to(DEV)

    def take(cols):
        c = torch.stack([maps[3 - lag:length - lag, :, m].T.reshape(-1) for m, lag in cols])
        return ((c - c.mean(1, keepdim=True)) / c.std(1, keepdim=True)).float().contiguous()

    return take([(2, 1), (1, 1)][:dx]), take([(3, 0), (2, 0)][:dy]), take(_CHAIN_Z[:dz])


def _network(net, T, lags, seed):
    if net == "var10":
        return synth.var_network(n_nodes=10, order=lags, T=T, burn=200, seed=seed)
    return synth.var_network_indegree(n_nodes=50, order=lags, indegree=3, T=T, burn=200, seed=seed)


def _parents(net, target, n_proc, lags, past, count, rng):
    """`count` candidate ids a selection could have made: the target's drivers
    first, then other variables."""
    ids = [p * lags + lag - 1 for p, q, lag in net.edges if q == target and lag <= lags]
    rest = [c for c in range(n_proc * lags) if c // lags != target and c not in ids]
    ids = ids + [int(c) for c in rng.permutation(rest)]
    return ids[:count]


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    st = dict(case=case, seed=int(rng.integers(0, 2**62)))
    if kind == "cmi":
        st["xyz"] = _gaussian(case["n"], case["dx"], case["dy"], case["dz"], seed)
    elif kind == "logistic":
        st["xyz"] = _logistic(case["reps"], case["length"], 1, 1, case["dz"], seed)
    elif kind in ("step", "prune"):
        name = case.get("net", "var10")
        net = _network(name, case["T"], case["lags"], seed)
        count = case["chosen"] if kind == "step" else case["parents"]
        # the node with the most drivers: the target whose inference goes furthest
        deg = np.bincount([q for _, q, _ in net.edges], minlength=len(net.series))
        st["target"] = int(np.argmax(deg))
        st["ids"] = _parents(net, st["target"], len(net.series), case["lags"], case["past"], count,
                             rng)
        st["series"] = _gpu(net.series)
        if case.get("screened"):
            path = os.path.join(os.path.dirname(idtx.__file__), "screen_weights.bin")
            idtx.screen_load(path)
    elif kind == "batch":
        st["problems"] = []
        for p in range(case["problems"]):
            # the first problem has the largest N, the second the smallest, the rest are spread
            n = (case["n_max"], case["n_min"])[p] if p < 2 else int(
                math.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"]))))
            dx, dy, dz = 1 + p % 2, 1 + (p // 2) % 2, 1 + p % case["dz_max"]
            pseed = int(rng.integers(0, 2**62))
            if p % 2 == 0:
                x, y, z = _gaussian(n, dx, dy, dz, pseed)
            else:
                x, y, z = (c[:, :n].contiguous()
                           for c in _logistic(-(-n // 497), 500, dx, dy, dz, pseed))
            st["problems"].append(dict(x=x, y=y, z=z, n_surr=case["n_surr"],
                                       seed=int(rng.integers(0, 2**62))))
    else:
        # the screen's features as a collection run gives them: estimate, ln N, dims, k,
        # mean / sd / maximum of the cheap surrogates, ln S; target: the excess over the maximum
        r = case["rows"]
        sd = rng.uniform(0.003, 0.02, r)
        mean = rng.normal(0.0, 0.01, r)
        top = mean + sd * (1.4 + 0.4 * rng.standard_normal(r))
        f = np.stack([mean + sd * 3 * rng.exponential(1.0, r),
                      np.log(rng.choice([3997.0, 4997.0, 9995.0], r)), np.ones(r), np.ones(r),
                      rng.integers(2, 7, r), np.full(r, 4.0), mean, sd, top,
                      np.full(r, math.log(200.0))], axis=1).astype(np.float32)
        t = np.maximum(sd * (1.3 + 0.5 * rng.standard_normal(r)), 0.0).astype(np.float32)
        s = f.std(0)
        st["feats"], st["targets"] = f, t
        st["norm"] = (f.mean(0), np.where(s > 1e-6, 1.0 / np.maximum(s, 1e-6), 1.0))
        st["params"] = idtx.Screen(seed=seed).params
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "cmi":
        x, y, z = st["xyz"]
        want = case["k"] != 4
        return idtx.cmi_ksg(x, y, z if case["dz"] else None, k=case["k"], n_surr=case["n_surr"],
                            seed=st["seed"], want_eps=want, want_counts=want)
    if kind == "logistic":
        x, y, z = st["xyz"]
        return idtx.cmi_ksg(x, y, z, k=4, n_surr=case["n_surr"], seed=st["seed"],
                            n_reps=case["reps"] if case["rep_level"] else 0)
    if kind == "step":
        res, est = idtx.mte_step(
            st["series"], st["target"], case["past"], 1, case["lags"], selected=st["ids"],
            step_index=case["chosen"], k=4, n_surr=case["n_surr"], seed=st["seed"],
            want_estimates=True,
            mode=idtx.MODE_SCREENED if case["screened"] else idtx.MODE_BATCHED)
        return [tuple(res), est]
    if kind == "prune":
        r = idtx.mte_prune(st["series"], st["target"], case["past"], 1, case["lags"],
                           st["ids"], k=4, n_surr=case["n_surr"], seed=st["seed"])
        # as many rounds as there could have been, and as many survivors
        rest = case["parents"] - len(r["rounds"])
        return dict(kept=r["kept"] + [-1] * (case["parents"] - len(r["kept"])),
                    rounds=r["rounds"] + [(-1, False, 0.0, 0.0)] * rest)
    if kind == "batch":
        return idtx.cmi_batch(st["problems"], k=4)
    sc = idtx.Screen(params=st["params"], feat_mean=st["norm"][0], feat_scale=st["norm"][1])
    loss = idtx.screen_train(sc, st["feats"], st["targets"], epochs=case["epochs"],
                             batch=case["batch"], lr=1e-3, seed=st["seed"],
                             quantile=case["quantile"])
    return [loss, sc.params]


# ------------------------------------------------------------------ least work
def _least(n, dx, dy, dz, k, estimates):
    """An estimate needs at least the joint distances of every sample to its k
    neighbours (a difference and a maximum per column) and three counts, whatever
    the search; each column is read once and each estimate written once."""
    return (n * (dx + dy + dz) * 4 + estimates * 8,
            float(estimates) * n * (2 * k * (dx + dy + dz) + 3))


def work(case):
    kind = case["kind"]
    if kind == "cmi":
        n, jobs = case["n"], 1 + case["n_surr"]
        b, f = _least(n, case["dx"], case["dy"], case["dz"], case["k"], jobs)
        return dict(bytes=b + (jobs * n * 16 if case["k"] != 4 else 0), flops=f)
    if kind == "logistic":
        b, f = _least(case["reps"] * (case["length"] - 3), 1, 1, case["dz"], 4, 1 + case["n_surr"])
        return dict(bytes=b, flops=f)
    if kind == "step":
        n_proc = 10 if case["net"] == "var10" else 50
        cand = n_proc * case["lags"] - min(case["past"], case["lags"]) - case["chosen"]
        # a screened step can get by with every candidate's estimate and eight surrogates
        jobs = cand * (1 + (8 if case["screened"] else case["n_surr"]))
        n = case["T"] - max(case["lags"], case["past"])
        b, f = _least(n, 1, 1, case["past"] + case["chosen"], 4, jobs)
        return dict(bytes=n_proc * case["T"] * 4 + jobs * 8, flops=f)
    if kind == "prune":
        jobs = case["parents"] * (1 + case["n_surr"])  # one round
        _, f = _least(case["T"] - max(case["lags"], case["past"]), 1, 1,
                      case["past"] + case["parents"] - 1, 4, jobs)
        return dict(bytes=(1 + case["parents"]) * case["T"] * 4, flops=f)
    if kind == "batch":
        lo, hi = case["n_min"], case["n_max"]
        mean = (hi - lo) / math.log(hi / lo) if hi > lo else lo  # of N spread over its logarithm
        by, fl = 0.0, 0.0
        for p in range(case["problems"]):
            b, f = _least((hi, lo)[p] if p < 2 else mean, 1 + p % 2, 1 + (p // 2) % 2,
                          1 + p % case["dz_max"], 4, 1 + case["n_surr"])
            by, fl = by + b, fl + f
        return dict(bytes=by, flops=fl)
    # forward, input gradients and weight gradients of the three layers, and the last loss
    layer = 2 * (10 * 64 + 64 * 64 + 64)
    rows = case["rows"]
    return dict(bytes=rows * 44 + 2 * idtx.SCREEN_NPARAMS * 4,
                flops=float(rows) * layer * (3 * case["epochs"] + 1))


# ------------------------------------------------------------------ 64 bits
_M = np.uint64(0xFFFFFFFF)


def _mix64(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _perms(n, streams, seed):
    """Fisher-Yates shuffles of [0, n) driven by SplitMix64, one per stream."""
    streams = np.asarray(streams, np.uint64)
    a = np.tile(np.arange(n), (len(streams), 1))
    base = np.uint64(seed) ^ _mix64(streams)
    rows = np.arange(len(streams))
    for s in range(n - 1):
        i = n - 1 - s
        r = _mix64(base + np.uint64((s + 1) * 0x9E3779B97F4A7C15 & 0xFFFFFFFFFFFFFFFF))
        m = np.uint64(i + 1)  # below 2^32: the high word of r * m from 32-bit halves
        j = (((r >> np.uint64(32)) * m + ((r & _M) * m >> np.uint64(32))) >> np.uint64(32)).astype(
            np.int64)
        at = a[rows, j]
        a[rows, j] = a[:, i]
        a[:, i] = at
    return a


def _dist(cols, q0, q1):
    d = torch.zeros(q1 - q0, cols.shape[1], dtype=torch.float64, device=DEV)
    for c in cols:
        d = torch.maximum(d, (c[q0:q1, None] - c[None, :]).abs())
    return d


def _estimates(xs, y, z, k):
    """KSG estimates in 64 bits of every x [d][n] in xs given the same y, z;
    with them eps of every estimate."""
    xs = [x.double() for x in xs]
    y, z = y.double(), z.double()
    n = y.shape[1]
    step = max(1, 20000000 // n)
    total = torch.zeros(len(xs), dtype=torch.float64, device=DEV)
    eps_all = torch.zeros(len(xs), n, dtype=torch.float64, device=DEV)
    for q0 in range(0, n, step):
        q1 = min(n, q0 + step)
        dz = _dist(z, q0, q1)
        own = torch.arange(q0, q1, device=DEV)
        dz[own - q0, own] = math.inf
        dyz = torch.maximum(dz, _dist(y, q0, q1))
        for e, x in enumerate(xs):
            dx = _dist(x, q0, q1)
            eps = torch.topk(torch.maximum(dx, dyz), k, largest=False).values[:, -1:]
            in_z = dz < eps
            nz, nyz = in_z.sum(1), (dyz < eps).sum(1)
            nxz = (in_z & (dx < eps)).sum(1)
            total[e] += (torch.digamma(nz.double() + 1.0) - torch.digamma(nxz.double() + 1.0)
                         - torch.digamma(nyz.double() + 1.0)).sum()
            eps_all[e, q0:q1] = eps[:, 0]
    psi_k = torch.digamma(torch.tensor(float(k), dtype=torch.float64))
    return (psi_k.to(DEV) + total / n), eps_all


def _train64(case, st):
    """The training in 64 bits, the weight matrices rounded to bfloat16 in every pass."""
    F, H = idtx.SCREEN_F, idtx.SCREEN_H
    p = torch.from_numpy(st["params"]).double()
    f = (torch.from_numpy(st["feats"]).double() - torch.from_numpy(np.float32(st["norm"][0])).double()
         ) * torch.from_numpy(np.float32(st["norm"][1])).double()
    t = torch.from_numpy(st["targets"]).double()
    cuts = np.cumsum([H * F, H, H * H, H, H, 1])[:-1]
    q, lr, n = case["quantile"], float(np.float32(1e-3)), case["rows"]
    q = float(np.float32(q))

    def loss_of(p, rows):
        w1, b1, w2, b2, w3, b3 = torch.tensor_split(p, cuts.tolist())
        r16 = lambda w: w + (w.detach().float().bfloat16().double() - w.detach())  # noqa: E731
        h = torch.relu(f[rows] @ r16(w1).view(H, F).T + b1)
        h = torch.relu(h @ r16(w2).view(H, H).T + b2)
        d = (h @ r16(w3) + b3) - t[rows]
        if q > 0.0:
            return (-d * (q - (d.detach() > 0).double())).sum()
        return (d * d).sum()

    m, v, step = torch.zeros_like(p), torch.zeros_like(p), 0
    for ep in range(case["epochs"]):
        order = torch.from_numpy(_perms(n, [ep], st["seed"])[0])
        for at in range(0, n, case["batch"]):
            rows = order[at:at + case["batch"]]
            p = p.detach().requires_grad_(True)
            g, = torch.autograd.grad(loss_of(p, rows) / len(rows), p)
            step += 1
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            p = p.detach() - lr * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step))
                                                             + 1e-8)
    return [float(loss_of(p.detach(), torch.arange(n))) / n, p]


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("cmi", "step", "prune", "train") or case.get("screened"):
        return None  # hours of brute force, or a choice of what to compute
    st = prepare(case, seed)
    if kind == "train":
        return _train64(case, st)
    with torch.no_grad(), np.errstate(over="ignore"):
        if kind == "cmi":
            n, s = case["n"], case["n_surr"]
            if float(n) * n * (1 + s) * (3 + sum(case[d] for d in ("dx", "dy", "dz"))) > 1.2e11:
                return None
            x, y, z = st["xyz"]
            perm = torch.from_numpy(_perms(n, range(s), st["seed"])).to(DEV) if s else []
            est, eps = _estimates([x] + [x[:, p] for p in perm], y, z, case["k"])
            return [est, eps, None] if case["k"] != 4 else est
        # the greedy step's largest estimate; the pruning's smallest one in its first round
        ser, lags, past = st["series"], case["lags"], case["past"]
        first = max(lags, past)
        T = ser.shape[1]

        def col(p, lag):
            return ser[p, first - lag:T - lag]

        def var(c):
            return col(c // lags, 1 + c % lags)

        tgt = st["target"]
        y = col(tgt, 0)[None, :]
        z = [col(tgt, lag) for lag in range(1, past + 1)]
        if kind == "prune":
            stat = min(float(_estimates([var(c)[None, :]], y, torch.stack(
                z + [var(o) for o in st["ids"] if o != c]), 4)[0][0]) for c in st["ids"])
            return dict(kept=None, rounds=[(None, None, stat, None)])
        cands = [c for c in range(ser.shape[0] * lags)
                 if c not in st["ids"] and not (c // lags == tgt and c % lags < past)]
        est, _ = _estimates([var(c)[None, :] for c in cands], y,
                            torch.stack(z + [var(o) for o in st["ids"]]), 4)
        return [(None, None, float(est.max()), None), None]
