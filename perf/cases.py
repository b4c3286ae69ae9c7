"""The work that a user of this engine has it do, as cases that can be timed.

A case is one call (or one short run of calls) of ``paper_0908_0681_gb300.engine`` on one of the
repository's three models (``workloads.three_orbital``, ``five_orbital``, ``seven_orbital``, the
five-orbital one at other temperatures for the Markov chains):

* ``trace``, ``ratio``, ``measure``: a batch of walkers through kt_trace, kt_trace_ratio (one
  insertion or removal per walker) and kt_measure (the observables at beta/2);
* ``cached``: the partial-state cache of fixed configurations built once, then ``rounds`` sets
  of proposals evaluated against it;
* ``sweep``, ``da``: Metropolis steps of independent CT-HYB chains, plain or with multi-try delayed
  acceptance, with and without the partial-state cache;
* ``train``: one pass of Adam over recorded proposals, the surrogate's training.

Precisions: ``f64``, ``f32`` (FP32 Krylov vectors) and ``tri64`` (the same with
KT_FP32_TRIDIAG64). On the FP32 path the ratios and the observables are kept as float32, as a
sampler keeps them: the path computes them to FP32 accuracy. log|T|, which runs to thousands,
stays in float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0908_0681_gb300 import engine, kt, workloads

PRECISION = {"f64": (kt.KT_FP64, 0), "f32": (kt.KT_FP32_KRYLOV, 0),
             "tri64": (kt.KT_FP32_KRYLOV, kt.KT_FP32_TRIDIAG64)}
ORBITALS = {3: "three_orbital", 5: "five_orbital", 7: "seven_orbital"}
FEATURES = 35 * 10 + 3 + 15  # the surrogate's inputs for ten flavors, rounded up to a multiple of 16
N_IN = FEATURES // 16 * 16


def listed():
    return [
        # a smoke-sized call: launches and latency, an odd batch, mostly structural zeros
        {"name": "trace 3 orbitals f64", "do": "trace", "orb": 3, "prec": "f64", "n": 37},
        # the sampler's inner call on the headline model, the default precision
        {"name": "ratio 5 orbitals f32", "do": "ratio", "orb": 5, "prec": "f32", "n": 4096},
        # the same where the user asks for FP64 throughout
        {"name": "ratio 5 orbitals f64", "do": "ratio", "orb": 5, "prec": "f64", "n": 4096},
        # the FP64-accurate tridiagonal option, a ragged batch
        {"name": "ratio 5 orbitals tri64", "do": "ratio", "orb": 5, "prec": "tri64", "n": 777},
        # f-shell model: large blocks, 63 kept states, few walkers
        {"name": "ratio 7 orbitals f32", "do": "ratio", "orb": 7, "prec": "f32", "n": 256},
        {"name": "ratio 7 orbitals f64", "do": "ratio", "orb": 7, "prec": "f64", "n": 101},
        # a measurement of a batch of configurations
        {"name": "measure 5 orbitals f64", "do": "measure", "orb": 5, "prec": "f64", "n": 1000},
        # fixed configurations against several sets of proposals
        {"name": "cached 5 orbitals f32", "do": "cached", "orb": 5, "prec": "f32", "n": 4096, "rounds": 4},
        # production sampling: chains at beta = 50, from scratch and with the partial-state cache
        {"name": "sweep f32", "do": "sweep", "beta": 50.0, "prec": "f32", "n": 1024, "steps": 16, "cache": 0},
        {"name": "sweep f32 cached", "do": "sweep", "beta": 50.0, "prec": "f32", "n": 1024, "steps": 16, "cache": 512},
        # the same chains behind the surrogate, eight tries a step
        {"name": "sweep f32 delayed cached", "do": "da", "beta": 50.0, "prec": "f32", "n": 1024, "steps": 8,
         "tries": 8, "cache": 512},
        # fitting the surrogate to recorded proposals
        {"name": "surrogate epoch", "do": "train", "rows": 32768, "batch": 4096},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["trace", "ratio", "ratio", "ratio", "measure", "cached", "sweep", "sweep", "da", "train"])
    if do == "train":
        batch = 16 * _log(rng, 4, 256)
        return {"do": do, "rows": batch * rng.randint(2, 8) + rng.randint(0, 15), "batch": batch}
    if do in ("sweep", "da"):
        prec = rng.choice(["f32", "f32", "f64"])
        c = {"do": do, "beta": rng.choice([10.0, 50.0]) if prec == "f64" else 50.0, "prec": prec,
             "n": _log(rng, 2, 1024 if prec == "f32" else 64), "steps": rng.randint(3, 12 if prec == "f32" else 4),
             "cache": rng.choice([0, 512])}
        if do == "da":
            c["tries"] = rng.randint(1, 8)
        return c
    if do == "trace":
        orb, prec = rng.choice([(3, "f64"), (5, "f64"), (5, "f32"), (7, "f64")])
    elif do == "measure":
        orb, prec = rng.choice([(3, "f64"), (5, "f64"), (5, "f32"), (5, "tri64")])
    elif do == "cached":
        orb, prec = rng.choice([(3, "f64"), (3, "f32"), (5, "f32"), (5, "tri64")])
    else:
        orb, prec = rng.choice([3, 5, 5, 7]), rng.choice(["f64", "f32", "tri64"])
    most = {3: 4096, 5: 4096 if prec != "f64" else 1024, 7: 192 if prec != "f64" else 64}[orb]
    c = {"do": do, "orb": orb, "prec": prec, "n": _log(rng, {3: 24, 5: 2, 7: 2}[orb], most)}
    if do == "cached":
        c["rounds"] = rng.randint(1, 4)
    elif orb == 3 and rng.random() < 0.4:
        c["eps"] = 0.0   # the untruncated trace: every eigenstate kept
        c["n"] = min(c["n"], 512)
    elif orb == 7 and rng.random() < 0.4:
        c["eps"] = 1e-4  # the wider energy window
    return c


def _workload(case):
    if case["do"] in ("sweep", "da"):
        w = workloads.five_orbital()
        w.model = workloads.five_orbital_sweep(case["beta"]).model
        w.lam = 6.0 * case["beta"] / 50.0
        return w
    w = getattr(workloads, ORBITALS[case["orb"]])()
    if "eps" in case:
        w.model.trunc_eps = case["eps"]
    return w


def _model(case, w):
    prec, flags = PRECISION[case["prec"]]
    return engine.model_from_spec(w.model, precision=prec, flags=flags)


def _rows(case, seed):
    """Recorded proposals: features as sparse and as small as the sweep's, smooth targets."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.rand((case["rows"], N_IN), device="cuda", generator=g)
    X = torch.where(X < 0.3, X / 0.3, torch.zeros_like(X)).to(torch.bfloat16)
    a = torch.randn(N_IN, device="cuda", generator=g)
    return X, torch.clamp(X.float() @ a, -25.0, 10.0)


def _weights(seed, out=1.0):
    rng = np.random.default_rng(seed)
    H = kt.KT_MLP_HIDDEN
    return np.concatenate([rng.normal(0, np.sqrt(2.0 / N_IN), H * N_IN), np.zeros(H),
                           rng.normal(0, np.sqrt(2.0 / H), H * H), np.zeros(H),
                           rng.normal(0, out * np.sqrt(2.0 / H), H), np.zeros(1)]).astype(np.float32)


def prepare(case, seed):
    s = {"case": case}
    if case["do"] == "train":
        s["X"], s["t"] = _rows(case, seed)
        s["net"] = engine.Surrogate(N_IN, max_batch=case["batch"], params=_weights(seed))
        return s
    w = _workload(case)
    m = s["model"] = _model(case, w)
    seqs = workloads.generate_sequences(w, case["n"], seed)
    if case["do"] in ("sweep", "da"):
        hyb = workloads.semicircular_hybridization(case["beta"], 10, n_quad=512)
        sw = engine.Sweep(m, hyb, case["beta"], case["n"], k_cap=64, n_bins=100, cache_ops=case["cache"])
        sw.set_configs(seqs)
        s["sweep"] = sw
        s["rng"] = torch.Generator(device="cuda").manual_seed(seed)
        if case["do"] == "da":  # small outputs: a surrogate that leaves most of the decision to stage 2
            s["net"] = engine.Surrogate(N_IN, max_batch=max(16, (case["n"] * case["tries"] + 15) // 16 * 16),
                                        params=_weights(seed, 0.1))
            sw.set_surrogate(s["net"])
        return s
    s["seqs"] = engine.DeviceSeqs.from_host(seqs)
    if case["do"] in ("ratio", "cached"):
        s["moves"] = [engine.DeviceMoves.from_host(workloads.generate_moves(w, seqs, seed + 1000 + r))
                      for r in range(case.get("rounds", 1))]
        # the current weights, which a sampler carries along: here in 64 bits for every precision
        m64 = m if case["prec"] == "f64" else _model({**case, "prec": "f64"}, w)
        s["sign"], s["log"], _ = engine.trace(m64, s["seqs"])
    if case["do"] == "cached":
        s["cache"] = engine.RatioCache(m, case["n"], max_ops=256)
    else:
        nobs = case["do"] == "measure"
        size = (kt.kt_measure_workspace_size if nobs else kt.kt_workspace_size)(m, case["n"])
        s["ws"] = torch.empty(max(size, 1), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    case = s["case"]
    do, f32 = case["do"], case.get("prec") != "f64"
    if do == "trace":
        sign, log, status = engine.trace(s["model"], s["seqs"], ws=s["ws"])
        return {"sign": sign, "log": log, "status": status}
    if do == "ratio":
        sign, lr, status = engine.trace_ratio(s["model"], s["seqs"], s["sign"], s["log"], s["moves"][0], ws=s["ws"])
        return {"sign": sign, "logratio": lr.float() if f32 else lr, "status": status}
    if do == "measure":
        sign, log, obs, status = engine.measure(s["model"], s["seqs"], ws=s["ws"])
        return {"sign": sign, "log": log, "obs": obs.float() if f32 else obs, "status": status}
    if do == "cached":
        s["cache"].build(s["seqs"])
        out = []
        for mv in s["moves"]:
            sign, lr, status = s["cache"].ratio(s["seqs"], s["sign"], s["log"], mv)
            out.append({"sign": sign, "logratio": lr.float() if f32 else lr, "status": status})
        return out
    if do == "train":
        loss = s["net"].train(s["X"], s["t"], epochs=1, batch=case["batch"])
        return {"loss": loss, "params": s["net"].params()}
    sw, shape = s["sweep"], (case["steps"], case["n"])
    if do == "sweep":
        sw.run(torch.rand(shape + (6,), dtype=torch.float64, device="cuda", generator=s["rng"]),
               meas_every=max(1, case["steps"] // 2))
    else:
        sw.run_da_multi(torch.rand(shape + (case["tries"], 7), dtype=torch.float64, device="cuda", generator=s["rng"]),
                        meas_every=max(1, case["steps"] // 2))
    st, acc = sw.state(), sw.accumulators()
    inside = torch.arange(sw.capacity, device="cuda")[None, :] < st["lens"][:, None]  # past its end a slot holds nothing
    for k in ("tau", "flavor", "dagger"):
        st[k] = st[k] * inside
    del acc["obs_sum"]  # not asked for
    return {"state": st, "acc": acc}


def _blocks(n):
    """Sizes of the invariant blocks: (n_up, n_dn) and the set of singly occupied orbitals."""
    x = np.arange(4 ** n)
    up = [(x >> 2 * a) & 1 for a in range(n)]
    dn = [(x >> 2 * a + 1) & 1 for a in range(n)]
    mask = sum((up[a] ^ dn[a]) << a for a in range(n))
    key = (sum(up) * (n + 1) + sum(dn)) * 2 ** n + mask
    return np.unique(key, return_inverse=True, return_counts=True)[1:]


def work(case):
    """Every operator, move and uniform read once, every result written once. Arithmetic: a
    propagation and an operator of one surviving kept state per walker and operator, as a
    dense block-to-block product."""
    if case["do"] == "train":
        per_row = 2 * 3 * (N_IN * 256 + 256 * 256 + 256)
        n_par = 256 * N_IN + 256 * 256 + 3 * 256 + 1
        steps = case["rows"] // case["batch"]
        return {"bytes": case["rows"] * (2 * N_IN + 4) + n_par * 4 * (1 + 6 * steps), "flops": steps * case["batch"] * per_row}
    w = _workload(case)
    n, nf = w.model.n_orb, 2 * w.model.n_orb
    d = _blocks(n)[1]
    K = nf * (8.0 if w.order == "uniform8" else 2 * w.lam)
    per_walker = K * 2.0 * float((d * d).sum()) / len(d)
    nw = case["n"]
    if case["do"] in ("sweep", "da"):
        evals = case["steps"] * nw
        u = evals * 8 * (6 if case["do"] == "sweep" else 7 * case["tries"])
        order = K / 2 / nf
        state = nw * (10 * K + 8 * nf * order * order + 100 * nf * 8)
        mlp = evals * case.get("tries", 0) * 2 * (N_IN * 256 + 256 * 256 + 256)
        return {"bytes": u + 2 * state, "flops": evals * (per_walker + 4 * order * order) + mlp}
    rounds = case.get("rounds", 1) if case["do"] != "measure" else 1
    nobs = kt.measure_nobs(n) if case["do"] == "measure" else 0
    moves = 30 * rounds if case["do"] in ("ratio", "cached") else 0
    return {"bytes": nw * (10 * K + 4 + moves + rounds * 13 + 8 * nobs), "flops": nw * per_walker * rounds}


# ---------------------------------------------------------------------------
# The same results in 64 bits, from dense block exponentials in plain torch and numpy.
# ---------------------------------------------------------------------------
class _Dense:
    """H_loc block by block, diagonalised, with the c / c^+ maps between the blocks."""

    def __init__(self, spec, dev):
        n, nf = spec.n_orb, 2 * spec.n_orb
        N = 4 ** n
        x = np.arange(N)
        bit = lambda y, f: (y >> f) & 1  # noqa: E731
        sgn = np.array([[1 - 2 * (bin(int(y) & ((1 << f) - 1)).count("1") & 1) for f in range(nf)] for y in x])
        blk, dim = _blocks(n)
        B, D = len(dim), int(dim.max())
        order = np.argsort(blk, kind="stable")
        first = np.concatenate([[0], np.cumsum(dim)[:-1]])
        rank = np.empty(N, np.int64)
        rank[order] = np.arange(N) - first[blk[order]]
        H = np.zeros((B, D, D))
        e = np.zeros(N)
        for a in range(n):
            u, d = bit(x, 2 * a), bit(x, 2 * a + 1)
            e += -(spec.mu + spec.delta[a]) * (u + d) + spec.U * u * d
            for b in range(a):
                bu, bd = bit(x, 2 * b), bit(x, 2 * b + 1)
                e += spec.up * (u * bd + d * bu) + (spec.up - spec.J) * (u * bu + d * bd)
        H[blk, rank, rank] = e
        S2 = np.zeros((B, D, D))
        nu, nd = sum(bit(x, 2 * a) for a in range(n)), sum(bit(x, 2 * a + 1) for a in range(n))
        sz = 0.5 * (nu - nd)
        S2[blk, rank, rank] = sz * sz + sz + sum(bit(x, 2 * a + 1) * (1 - bit(x, 2 * a)) for a in range(n))

        def string(ops):  # the image of every bitstring under a string of operators, right to left
            y, s, ok = x.copy(), np.ones(N, np.int64), np.ones(N, bool)
            for f, dag in ops:
                ok &= bit(y, f) != dag
                s *= sgn[y, f]
                y = y ^ (1 << f)
            return y[ok], x[ok], s[ok]

        for a in range(n):
            for b in range(n):
                if a != b:
                    y, z, s = string([(2 * a, 0), (2 * b + 1, 0), (2 * b, 1), (2 * a + 1, 1)])
                    np.add.at(H, (blk[y], rank[y], rank[z]), -spec.J * s)
                    np.add.at(S2, (blk[y], rank[y], rank[z]), s)
                    y, z, s = string([(2 * a + 1, 0), (2 * a, 0), (2 * b + 1, 1), (2 * b, 1)])
                    np.add.at(H, (blk[y], rank[y], rank[z]), -spec.J * s)
        E, V = np.full((B, D), 1e6), np.zeros((B, D, D))
        for b in range(B):
            E[b, :dim[b]], V[b, :dim[b], :dim[b]] = np.linalg.eigh(H[b, :dim[b], :dim[b]])
        self.E0 = E.min()
        lv = sorted((E[b, k], b, k) for b in range(B) for k in range(dim[b]))
        kept = []
        for i, l in enumerate(lv):  # whole multiplets
            if i and l[0] - lv[i - 1][0] > spec.deg_tol * max(1.0, abs(l[0])) and spec.trunc_eps > 0 and \
                    math.exp(-spec.beta * (l[0] - self.E0)) < spec.trunc_eps:
                break
            kept.append(l)
        self.kept_b = np.array([b for _, b, _ in kept])
        self.kept_e = np.array([k[0] - self.E0 for k in kept])
        self.kept_v = np.array([V[b][:, k] for _, b, k in kept])
        # row r of block b under flavor f: source rank and sign if the row's bit f equals dag
        src, sg = np.zeros((B, nf, D), np.int64), np.zeros((B, nf, D))
        occ = np.zeros((B, nf, D), np.int64)
        target = np.full((B, nf, 2), -1)
        for f in range(nf):
            src[blk, f, rank], sg[blk, f, rank], occ[blk, f, rank] = rank[x ^ (1 << f)], sgn[:, f], bit(x, f)
            target[blk, f, 1 - bit(x, f)] = blk[x ^ (1 << f)]
        real = np.zeros((B, D))
        real[blk, rank] = 1.0
        self.sector = np.zeros(B, np.int64)
        self.sector[blk] = nu * (n + 1) + nd
        self.target, self.beta, self.n, self.nf, self.D, self.dev = target, spec.beta, n, nf, D, dev
        t = lambda v: torch.as_tensor(v, device=dev)  # noqa: E731
        self.E, self.V, self.S2 = t(E - self.E0), t(V), t(S2)
        self.src, self.sg, self.occ, self.real = t(src), t(sg), t(occ), t(real)

    def alive(self, seqs):
        """(walker, kept state) pairs whose block path closes."""
        w, q = [], []
        for i, (_, fl, dg) in enumerate(seqs):
            b = self.kept_b.copy()
            for f, d in zip(fl, dg):
                b = np.where(b >= 0, self.target[b, f, d], -1)
            k = np.nonzero(b == self.kept_b)[0]
            w += [i] * len(k)
            q += k.tolist()
        return np.array(w, np.int64), np.array(q, np.int64)

    def push(self, q, steps, t_end, backward):
        """The kept states q through their operators (a list per item, in the order they act; from
        beta downwards if backward) up to t_end: normalised vectors, blocks, log-weights."""
        dev, n = self.dev, len(q)
        K = max((len(s[0]) for s in steps), default=0)
        tau, fl, dg, real = np.zeros((n, K)), np.zeros((n, K), np.int64), np.zeros((n, K), np.int64), np.zeros((n, K), bool)
        for i, (a, b, c) in enumerate(steps):
            k = len(a)
            tau[i, :k], fl[i, :k], dg[i, :k], real[i, :k] = a, b, c, True
        blk = self.kept_b[q]
        x = torch.as_tensor(self.kept_v[q], device=dev)
        log = torch.zeros(n, dtype=torch.float64, device=dev)
        t = np.full(n, self.beta if backward else 0.0)

        def flow(x, log, blk, dt, on):
            b, dt = torch.as_tensor(blk, device=dev), torch.as_tensor(np.where(on, dt, 0.0), device=dev)
            c = torch.einsum("nrk,nr->nk", self.V[b], x)
            e = self.E[b]
            c = c * torch.exp(-dt[:, None] * (e - e[:, :1]))
            y = torch.einsum("nrk,nk->nr", self.V[b], c)
            nrm = y.norm(dim=1)
            y, l = y / torch.where(nrm > 0, nrm, torch.ones_like(nrm))[:, None], log + torch.log(nrm) - dt * e[:, 0]
            on = torch.as_tensor(on & (dt.cpu().numpy() > 0), device=dev)
            return torch.where(on[:, None], y, x), torch.where(on, l, log)

        for k in range(K):
            on = real[:, k]
            x, log = flow(x, log, blk, (t - tau[:, k]) if backward else (tau[:, k] - t), on)
            t = np.where(on, tau[:, k], t)
            d = 1 - dg[:, k] if backward else dg[:, k]
            nb = np.where(on, self.target[blk, fl[:, k], d], blk)
            b2, f2 = torch.as_tensor(nb, device=dev), torch.as_tensor(fl[:, k], device=dev)
            y = torch.gather(x, 1, self.src[b2, f2]) * self.sg[b2, f2] * self.real[b2]
            y = y * (self.occ[b2, f2] == torch.as_tensor(d, device=dev)[:, None])
            x = torch.where(torch.as_tensor(on, device=dev)[:, None], y, x)
            blk = nb
        x, log = flow(x, log, blk, (t - t_end) if backward else (t_end - t), np.ones(n, bool))
        return x, blk, log

    def halves(self, seqs):
        """Both halves of every live item, meeting at beta/2."""
        w, q = self.alive(seqs)
        h = 0.5 * self.beta
        cut = [int(np.searchsorted(s[0], h)) for s in seqs]
        f = self.push(q, [tuple(v[:cut[i]] for v in seqs[i]) for i in w], h, False)
        b = self.push(q, [tuple(v[cut[i]:][::-1] for v in seqs[i]) for i in w], h, True)
        return w, f, b

    def total(self, n, w, val, log):
        """sum over the items of a walker of val exp(log): sign and log of each."""
        val, log = val.cpu().numpy(), log.cpu().numpy()
        top = np.full(n, -np.inf)
        np.maximum.at(top, w, log)
        s = np.zeros(n)
        np.add.at(s, w, val * np.exp(log - top[w]))
        with np.errstate(divide="ignore", invalid="ignore"):
            return s, np.where(s != 0, np.log(np.abs(s)) + top - self.beta * self.E0, -np.inf), top

    def trace(self, seqs):
        w, (fx, fb, fl), (bx, _, bl) = self.halves(seqs)
        s, log, _ = self.total(len(seqs), w, (fx * bx).sum(1), fl + bl)
        return np.sign(s).astype(np.int8), log

    def measure(self, seqs):
        n, nf, nl = self.n, self.nf, self.nf + self.n + 1
        w, (fx, fb, fl), (bx, _, bl) = self.halves(seqs)
        b = torch.as_tensor(fb, device=self.dev)
        p = fx * bx
        s, log, top = self.total(len(seqs), w, p.sum(1), fl + bl)
        obs = np.zeros((len(seqs), kt.measure_nobs(n)))
        occ = self.occ[b].double()
        cols = [(p * occ[:, f]).sum(1) for f in range(nf)]
        cols += [(p * occ[:, 2 * a] * occ[:, 2 * a + 1]).sum(1) for a in range(n)]
        cols.append((bx * torch.einsum("nrs,ns->nr", self.S2[b], fx)).sum(1))
        e = np.exp((fl + bl).cpu().numpy() - top[w])
        for k, v in enumerate(cols):
            np.add.at(obs[:, k], w, v.cpu().numpy() * e)
        np.add.at(obs, (w, nl + self.sector[fb]), p.sum(1).cpu().numpy() * e)
        with np.errstate(divide="ignore", invalid="ignore"):
            obs = np.where(s[:, None] != 0, obs / s[:, None], np.nan)
        return np.sign(s).astype(np.int8), log, obs


def _edited(seqs, mv):
    """Every walker's sequence after its proposed update."""
    out = []
    for i in range(seqs.n):
        tau, fl, dg = seqs.walker(i)
        f = int(mv.flavor[i])
        if mv.kind[i] == 0:
            new = sorted([(mv.t_dag[i], 1), (mv.t_ann[i], 0)])
            at = np.searchsorted(tau, [t for t, _ in new], side="right")
            out.append((np.insert(tau, at, [t for t, _ in new]), np.insert(fl, at, f), np.insert(dg, at, [d for _, d in new])))
        else:
            r = int(mv.rem_idx[i])
            mine = np.nonzero(fl == f)[0]
            pair = [r, int(mine[(int(np.nonzero(mine == r)[0][0]) + 1) % len(mine)])]
            out.append(tuple(np.delete(v, pair) for v in (tau, fl, dg)))
    return out


def _exact_training(case, seed):
    """Mean squared error and Adam in 64 bits on the same rows in the same order."""
    X, t = _rows(case, seed)
    p = torch.as_tensor(_weights(seed), device="cuda").double()
    H, n = kt.KT_MLP_HIDDEN, N_IN
    cuts = [H * n, H, H * H, H, H, 1]
    m, v, losses, batch = torch.zeros_like(p), torch.zeros_like(p), [], case["batch"]
    g = torch.Generator(device="cuda").manual_seed(0)
    steps = case["rows"] // batch
    perm = torch.randperm(X.shape[0], device="cuda", generator=g)[:steps * batch]
    for k in range(steps):
        idx = perm[k * batch:(k + 1) * batch]
        q = p.clone().requires_grad_(True)
        W1, b1, W2, b2, w3, b3 = torch.split(q, cuts)
        h = torch.relu(X[idx].double() @ W1.view(H, n).T + b1)
        h = torch.relu(h @ W2.view(H, H).T + b2)
        loss = ((h @ w3 + b3 - t[idx].double()) ** 2).mean()
        grad, = torch.autograd.grad(loss, q)
        m, v = 0.9 * m + 0.1 * grad, 0.999 * v + 0.001 * grad * grad
        p = p - 1e-3 * (m / (1 - 0.9 ** (k + 1))) / (torch.sqrt(v / (1 - 0.999 ** (k + 1))) + 1e-8)
        losses.append(float(loss))
    return {"loss": [sum(losses) / max(steps, 1)], "params": p.cpu().numpy()}


def exact(case, seed):
    if case["do"] in ("sweep", "da"):
        return None  # a Markov chain's decisions have no value of their own
    if case["do"] == "train":
        return _exact_training(case, seed)
    w = _workload(case)
    D = _Dense(w.model, "cuda" if torch.cuda.is_available() else "cpu")
    host = workloads.generate_sequences(w, case["n"], seed)
    seqs = [host.walker(i) for i in range(host.n)]
    if case["do"] == "measure":
        sign, log, obs = D.measure(seqs)
        return {"sign": sign, "log": log, "obs": obs, "status": None}
    sign, log = D.trace(seqs)
    if case["do"] == "trace":
        return {"sign": sign, "log": log, "status": None}
    out = []
    for r in range(case.get("rounds", 1)):
        s, l = D.trace(_edited(host, workloads.generate_moves(w, host, seed + 1000 + r)))
        with np.errstate(invalid="ignore"):
            l = np.where(sign == 0, np.nan, l - log)
        out.append({"sign": (s * sign).astype(np.int8), "logratio": l, "status": None})
    return out if case["do"] == "cached" else out[0]
