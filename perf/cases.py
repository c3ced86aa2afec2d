"""The work that a user of the PSGLD library has it do, as measurable cases.

A case is one kind of call on one kind of data:

* ``sweep``    -- psgld_sweep on a chain past its burn-in (the posterior sums
                  are taken), then the factors read back to device tensors;
* ``step``     -- one psgld_part_step, then the factors read back;
* ``load``     -- new entries and factors into a context, one part-step, the
                  factors read back;
* ``evaluate`` -- log-likelihood, RMSE of the sample and of the posterior mean;
* ``readout``  -- posterior means and variances into host arrays;
* ``batch``    -- psgld_batch_sweep over uneven dense chains, every chain's
                  factors read back.

Data: ``ratings`` (sparse, Zipf degrees, values 1..5), ``poisson``,
``compound`` (compound Poisson-gamma, exact zeros) and ``gamma`` (dense).
``exact`` states one iteration from the paper's equations in FP64 torch.
"""
import math
import random

import numpy as np
import torch

from paper_1506_01418_gb300 import datagen
from paper_1506_01418_gb300 import psgld as P

DEV = "cuda"
GAUSS, EXPON = P.PSGLD_PRIOR_GAUSSIAN, P.PSGLD_PRIOR_EXPONENTIAL


def _sparse(name, kind, I, J, nnz, K, B, **kw):
    c = dict(kind=kind, data="ratings", I=I, J=J, nnz=nnz, K=K, B=B, p=0.0, prior=GAUSS, zipf_row=1.1,
             zipf_col=1.1, eps=2e-5, init=0.3, sweeps=1)
    c.update(kw)
    return dict(c, name=name) if name else c


def _dense(name, data, I, J, K, B, p, **kw):
    c = dict(kind="sweep", data=data, I=I, J=J, K=K, B=B, p=p, prior=EXPON, K_true=8, eps=1e-4, init=0.5,
             dense_path=1, sweeps=1)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest chain: dense Poisson counts on the FP32 path, where a
        # sweep is a few launches on next to no data
        _dense("sweep_counts_256x256_K8", "poisson", 256, 256, 8, 4, 1.0, init=1.0, dense_path=0),
        # one iteration at a time, as a program does that looks at every
        # sample: ragged pieces, odd K, a non-integer power, decaying step
        _sparse("step_counts_6997x1013_K13", "step", 6997, 1013, 100_000, 13, 7, p=1.5, prior=EXPON,
                init=0.6, eps_a=1e-5, eps_b=0.75),
        # a MovieLens-10M-shaped ratings chain: the ordinary sparse sweep
        _sparse("sweep_ratings_10M_K50", "sweep", 70000, 10000, 10_000_000, 50, 32),
        # the largest sparse chain, factors beyond L2
        _sparse("sweep_ratings_100M_K100", "sweep", 480000, 18000, 100_000_000, 100, 64, zipf_row=1.2,
                zipf_col=0.0, eps=5e-6, init=0.25),
        # the same recipe with fewer entries and the BF16-gathered factors
        _sparse("sweep_ratings_30M_K100_bf16", "sweep", 480000, 18000, 30_000_000, 100, 64, zipf_row=1.2,
                zipf_col=0.0, eps=5e-6, init=0.25, gather_bf16=1),
        # a new ratings slice arrives: data and factors in, the first iteration
        _sparse("load_ratings_10M_K50", "load", 70000, 10000, 10_000_000, 50, 32),
        # convergence checks of the ratings chain
        _sparse("evaluate_ratings_10M_K50", "evaluate", 70000, 10000, 10_000_000, 50, 32),
        # the answer of a chain: posterior means and variances on the host
        _sparse("readout_70000x10000_K50", "readout", 70000, 10000, 100_000, 50, 32),
        # one spectrogram alone: a job's sweeps replayed from its graph
        _dense("sweep_spectrogram_513x4000_K32", "gamma", 513, 4000, 32, 8, 1.0, K_true=16, sweeps=20),
        # the standing chain: tensor-core blocks, BF16 V, 10^9 entries a sweep
        _dense("sweep_counts_32768_K256", "poisson", 32768, 32768, 256, 16, 1.0, K_true=16, eps=2e-5,
               init=0.25, dense_path=2, dense_v_bf16=1),
        # many uneven spectrograms advancing together
        _dense("batch_256_spectrograms_K32", "gamma", 513, 0, 32, 8, 0.0, kind="batch", chains=256, J_lo=200,
               J_hi=5000, K_true=16, mix="alternate", sweeps=2, dense_path=2),
        # one turn of a serving loop: the jobs in flight, each one sweep on
        _dense("batch_serving_12_jobs", "mixed", 0, 0, 0, 8, 0.0, kind="batch", chains=12, J_lo=500,
               J_hi=20000, mix="serving", dense_path=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: any kind, sizes log-uniform, odd ones too."""
    kind = rng.choice(["sweep", "sweep", "step", "load", "evaluate", "readout", "dense", "dense", "batch"])
    if kind == "batch":
        if rng.random() < 0.5:
            return _dense(None, "gamma", rng.choice([129, 257, 513]), 0, rng.choice([16, 24, 32, 50, 64]),
                          rng.choice([4, 7, 8]), 0.0, kind="batch", chains=_log_int(rng, 8, 128), J_lo=200,
                          J_hi=5000, K_true=16, mix="alternate", sweeps=rng.randint(1, 4), dense_path=2,
                          list_seed=rng.randint(0, 999))
        return _dense(None, "mixed", 0, 0, 0, 8, 0.0, kind="batch", chains=_log_int(rng, 3, 24), J_lo=500,
                      J_hi=20000, mix="serving", dense_path=2, list_seed=rng.randint(0, 999))
    if kind == "dense":
        path = rng.choice([0, 1, 1, 2])
        top = 1200 if path == 0 else 12000
        I, J = _log_int(rng, 96, top), _log_int(rng, 96, top)
        # K <= 256: one pass of the tensor-core path; the FP32 path takes any
        K = _log_int(rng, 4, 256 if path else 64)
        p, data = rng.choice([(1.0, "poisson"), (1.5, "compound"), (2.0, "gamma")])
        c = _dense(None, data, I, J, K, rng.randint(1, 16), p, dense_path=path, sweeps=rng.randint(1, 4),
                   init=round(math.sqrt(8.0 / K), 4), eps=float("%.2e" % (0.1 / max(I, J))))
        if path == 2 and rng.random() < 0.5:
            c["dense_v_bf16"] = 1
        return c
    nnz = _log_int(rng, 20_000, 30_000_000)
    # at most one entry in 60 observed, as in the ratings workloads
    J = _log_int(rng, max(200, nnz // 8000), 20000)
    I = max(_log_int(rng, 300, 480000), 60 * nnz // J + 1)
    counts = kind == "step" or rng.random() < 0.3
    K = _log_int(rng, 4, 200)
    c = _sparse(None, kind, I, J, nnz, K, rng.randint(1, 64), zipf_row=rng.choice([1.05, 1.1, 1.2]),
                zipf_col=rng.choice([0.0, 1.05, 1.1]), eps=float("%.2e" % (0.05 / max(I, J))),
                init=round(0.3 if not counts else math.sqrt(3.0 / K), 4))
    if counts:
        c.update(p=rng.choice([1.0, 1.5, 2.0]), prior=EXPON)
    elif kind == "sweep" and rng.random() < 0.3:
        c["gather_bf16"] = 1
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _entries(case, seed):
    """(i, j, v) of sparse data on the device."""
    return datagen.sparse_ratings(case["I"], case["J"], case["nnz"], 20, seed, zipf_row=case["zipf_row"],
                                  zipf_col=case["zipf_col"] or None, device=DEV)


def _matrix(case, seed):
    I, J, kt, data = case["I"], case["J"], case["K_true"], case["data"]
    if data == "poisson":
        return datagen.dense_poisson_device(I, J, kt, seed, DEV)
    if data == "compound":
        return datagen.dense_compound_poisson_device(I, J, kt, seed, DEV, p=case["p"])
    return datagen.dense_gamma_device(I, J, kt, seed, DEV)


def _factors(case, seed):
    """Initial W (I x K) and H^T (J x K): Uniform(0.5, 1.5) or normal, scaled."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 7919)
    out = []
    for n in (case["I"], case["J"]):
        if case["prior"] == EXPON:
            x = torch.rand((n, case["K"]), generator=g, device=DEV).add_(0.5)
        else:
            x = torch.randn((n, case["K"]), generator=g, device=DEV)
        out.append(x.mul_(case["init"]))
    return out


def _sums(case, seed):
    """Posterior sums of 25 earlier samples, as a checkpoint holds them."""
    g = np.random.Generator(np.random.Philox(seed))
    K, n, out = case["K"], 25, []
    for rows in (case["I"], case["J"]):
        mean = g.standard_normal((rows, K)) * 0.4
        out += [mean * n, (mean * mean + 0.01 * g.random((rows, K))) * n]
    return (*out, np.array([n * case["B"], n, n], np.int64))


def _members(case):
    """The chains of a batch: what each is, from the case's own list."""
    rng = random.Random(case.get("list_seed", 0))
    out = []
    for k in range(case["chains"]):
        if case["mix"] == "alternate":
            m = dict(case, J=rng.randint(case["J_lo"], case["J_hi"]), p=1.0 + k % 2)
        else:
            p = rng.choice([1.0, 1.5])
            m = dict(case, I=rng.choice([257, 513, 1025]), J=_log_int(rng, case["J_lo"], case["J_hi"]),
                     K=rng.choice([16, 64]), p=p, data="poisson" if p == 1.0 else "compound")
        out.append(m)
    return out


_OPTIONS = ("dense_path", "dense_v_bf16", "gather_bf16")


def _chain(case, seed):
    opts = {k: case[k] for k in _OPTIONS if k in case}
    if "eps_a" in case:
        opts.update(eps_mode=P.PSGLD_EPS_POLY, eps_a=case["eps_a"], eps_b=case["eps_b"])
    return P.PSGLD(case["I"], case["J"], case["K"], case["B"], case["p"], 1.0, prior_kind=case["prior"],
                   seed=seed, eps=case["eps"], **opts)


def _with_data(case, seed):
    ch = _chain(case, seed)
    if case["data"] == "ratings":
        ch.set_data_coo(*_entries(case, seed))
    else:
        ch.set_data_dense(_matrix(case, seed))
    ch.set_factors(*_factors(case, seed))
    return ch


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        members = _members(case)
        state = {"kind": kind, "sweeps": case["sweeps"],
                 "chains": [_with_data(m, seed + 17 * k) for k, m in enumerate(members)]}
        # one buffer for all the factors, each chain's a contiguous piece
        state["out"] = torch.empty(sum((m["I"] + m["J"]) * m["K"] for m in members), device=DEV)
        state["views"], at = [], 0
        for m in members:
            pair = []
            for n in (m["I"], m["J"]):
                pair.append(state["out"][at:at + n * m["K"]].view(n, m["K"]))
                at += n * m["K"]
            state["views"].append(pair)
    elif kind == "load":
        state = {"kind": kind, "chain": _chain(case, seed), "entries": _entries(case, seed),
                 "factors": _factors(case, seed)}
    else:
        state = {"kind": kind, "chain": _with_data(case, seed), "sweeps": case["sweeps"], "t": 0}
        if kind in ("evaluate", "readout"):
            state["chain"].set_state(_sums(case, seed))
    torch.cuda.synchronize()
    return state


def run(state):
    kind = state["kind"]
    if kind == "batch":
        P.psgld_batch_sweep(state["chains"], state["sweeps"])
        for ch, (W, Ht) in zip(state["chains"], state["views"]):
            P.psgld_get_factors(ch.ctx, W, Ht)
        return state["out"]
    ch = state["chain"]
    if kind == "sweep":
        ch.sweep(state["sweeps"])
    elif kind == "step":
        state["t"] += 1
        ch.part_step(state["t"])
    elif kind == "load":
        ch.set_data_coo(*state["entries"])
        ch.set_factors(*state["factors"])
        ch.part_step(1)
    elif kind == "evaluate":
        return ch.log_lik(), ch.rmse(), ch.rmse(use_posterior_mean=True)
    elif kind == "readout":
        return ch.posterior_mean()
    return ch.get_factors()


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Entries once (8 bytes with their index, or the dense V's 4 or 2), the
    factors read and written once per part-step; three products of 2 K per
    entry."""
    if case["kind"] == "batch":
        parts = [work(dict(m, kind="sweep")) for m in _members(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    I, J, K, B, kind = case["I"], case["J"], case["K"], case["B"], case["kind"]
    sparse = case["data"] == "ratings"
    n = case["nnz"] if sparse else I * J
    per = 8 if sparse else 2 if case.get("dense_v_bf16") else 4
    fac = 8 * (I + J) * K
    if kind == "sweep":
        s = case["sweeps"]
        # each sweep's sample: the factors into two FP64 sums, read and written
        return {"bytes": s * (per * n + B * fac + 4 * fac), "flops": 6 * n * K * s}
    if kind == "step":
        return {"bytes": per * n // B + fac, "flops": 6 * n * K // B}
    if kind == "load":
        return {"bytes": 12 * n + fac + per * n // B + fac, "flops": 6 * n * K // B}
    if kind == "evaluate":
        # three passes over the entries, the sample twice and the sums once
        return {"bytes": 3 * per * n + 2 * fac, "flops": 6 * n * K}
    return {"bytes": 4 * fac, "flops": 6 * (I + J) * K}


# ---------------------------------------------------------------------------
# FP64 restatement (Sec. 3 Eq. psgld_w and psgld_h, Algorithm 1; Philox4x32-10
# normals by Box-Muller)
# ---------------------------------------------------------------------------

_M32 = 0xFFFFFFFF


def _normals(t, K, segments):
    """The n x K normals at iteration t of each segment (seed, matrix, n)."""
    groups, z = (K + 3) // 4, []

    def per_item(values):
        return torch.cat([torch.full((n * groups,), v, device=DEV, dtype=torch.int64)
                          for v, (_, _, n) in zip(values, segments)])

    rows = torch.cat([torch.arange(n, device=DEV) for _, _, n in segments])
    k0, k1 = (per_item([(seed >> b) & _M32 for seed, _, _ in segments]) for b in (0, 32))
    x = [torch.arange(groups, device=DEV).repeat(len(rows)), rows.repeat_interleave(groups),
         torch.full_like(k0, t & _M32), per_item([((t >> 32) << 1) | mat for _, mat, _ in segments])]
    for _ in range(10):
        a, b = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57          # 64-bit products, modulo 2^64
        x = [((b >> 32) & _M32) ^ x[1] ^ k0, b & _M32, ((a >> 32) & _M32) ^ x[3] ^ k1, a & _M32]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    u = [((w >> 9).double() + 0.5) * 2.0 ** -23 for w in x]
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        r = torch.sqrt(-2.0 * torch.log(a))
        z += [r * torch.cos(2 * math.pi * b), r * torch.sin(2 * math.pi * b)]
    return torch.stack(z, 1).view(len(rows), 4 * groups)[:, :K].split([n for _, _, n in segments])


def _residual(case, v, mu):
    p = case["p"]
    if p == 0.0:
        return v - mu
    return (v - mu) * mu.clamp(min=1e-10) ** -p


class _Exact:
    """One chain in FP64: data, factors, iteration counter."""

    def __init__(self, case, seed):
        self.case, self.seed, self.t = case, seed, 0
        self.W, self.H = (x.double() for x in _factors(case, seed))
        I, J, B = case["I"], case["J"], case["B"]
        self.rs = [(r * I) // B for r in range(B + 1)]
        self.cs = [(r * J) // B for r in range(B + 1)]
        if case["data"] == "ratings":
            i, j, v = _entries(case, seed)
            i, j = i.long(), j.long()
            part = (((j + 1) * B - 1) // J - ((i + 1) * B - 1) // I) % B
            order = torch.argsort(part, stable=True)
            self.i, self.j, self.v = i[order], j[order], v[order]
            self.first = [0] + torch.bincount(part, minlength=B).cumsum(0).tolist()
        else:
            self.V = _matrix(case, seed)

    def segments(self):
        return [(self.seed, 0, self.case["I"]), (self.seed, 1, self.case["J"])]

    def step(self, normals=None):
        c, self.t = self.case, self.t + 1
        I, J, B = c["I"], c["J"], c["B"]
        s, W, H = (self.t - 1) % B, self.W, self.H
        z = normals or _normals(self.t, c["K"], self.segments())
        GW, GH, n = torch.zeros_like(W), torch.zeros_like(H), 0
        if c["data"] == "ratings":
            n, N = self.first[s + 1] - self.first[s], len(self.v)
            for a in range(self.first[s], self.first[s + 1], 1 << 20):
                at = slice(a, min(a + (1 << 20), self.first[s + 1]))
                i, j = self.i[at], self.j[at]
                w, h = W[i], H[j]
                e = _residual(c, self.v[at].double(), (w * h).sum(1)).unsqueeze(1)
                GW.index_add_(0, i, e * h)
                GH.index_add_(0, j, e * w)
        else:
            N = I * J
            for r in range(B):
                q = (r + s) % B
                a, b, x, y = self.rs[r], self.rs[r + 1], self.cs[q], self.cs[q + 1]
                e = _residual(c, self.V[a:b, x:y].double(), W[a:b] @ H[x:y].T)
                n += (b - a) * (y - x)
                GW[a:b] = e @ H[x:y]
                GH[x:y] = e.T @ W[a:b]
        eps = (c["eps_a"] / self.t) ** c["eps_b"] if "eps_a" in c else c["eps"]
        S = N / n if n else 0.0
        out = []
        for x, g, zx in ((W, GW, z[0]), (H, GH, z[1])):
            prior = -1.0 if c["prior"] == EXPON else -x
            y = x + eps * (S * g + prior) + math.sqrt(2 * eps) * zx
            out.append(y.abs() if c["prior"] == EXPON else y)
        self.W, self.H = out


def _evaluate(x, n):
    """(log-likelihood, RMSE of the sample, RMSE of the mean) of sparse data."""
    c, sums = x.case, _sums(x.case, x.seed)
    mean = [torch.from_numpy(s).to(DEV) / n for s in (sums[0], sums[2])]
    ll = ss = sm = 0.0
    for a in range(0, len(x.v), 1 << 21):
        i, j, v = (y[a:a + (1 << 21)] for y in (x.i, x.j, x.v))
        v = v.double()
        mu = (x.W[i] * x.H[j]).sum(1)
        ss += float(((v - mu) ** 2).sum())
        sm += float(((v - (mean[0][i] * mean[1][j]).sum(1)) ** 2).sum())
        m, b = mu.clamp(min=1e-10) if c["p"] else mu, 2.0 - c["p"]
        if b == 2.0:
            d = 0.5 * (v - m) ** 2
        elif b == 1.0:
            d = torch.xlogy(v, v / m) - v + m
        elif b == 0.0:
            d = v / m - torch.log(v / m) - 1.0
        else:
            d = v ** b / (b * (b - 1)) - v * m ** (b - 1) / (b - 1) + m ** b / b
        ll -= float(d.sum())
    return ll, math.sqrt(ss / len(x.v)), math.sqrt(sm / len(x.v))


def exact(case, seed):
    kind = case["kind"]
    if kind == "readout":
        sW, sW2, sH, sH2, (_, _, n) = _sums(case, seed)
        out = []
        for s, s2 in ((sW, sW2), (sH, sH2)):
            m = s / n
            out += [m, s2 / n - m * m]
        return (*out, int(n))
    if kind == "batch":
        chains = [_Exact(m, seed + 17 * k) for k, m in enumerate(_members(case))]
        for t in range(1, case["sweeps"] * case["B"] + 1):
            for K in sorted({x.case["K"] for x in chains}):      # one K's normals together
                mine = [x for x in chains if x.case["K"] == K]
                z = _normals(t, K, [q for x in mine for q in x.segments()])
                for k, x in enumerate(mine):
                    x.step(z[2 * k:2 * k + 2])
        return torch.cat([f.reshape(-1) for x in chains for f in (x.W, x.H)])
    x = _Exact(case, seed)
    if kind == "evaluate":
        return _evaluate(x, 25)
    for _ in range(case["sweeps"] * case["B"] if kind == "sweep" else 1):
        x.step()
    return x.W, x.H
