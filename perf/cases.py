"""The work a user of this library has it do, as measurable cases.

Every case goes through a public entry point of ``paper_1606_08281_gb300.pf``
on one of the repository's own networks (``workloads.py``): the particle-filter
likelihood (`pf_loglik`), the exact finite-state-projection likelihood
(`pf_fsp_loglik`), the deterministic Erk-model likelihood (`pf_erk_loglik`) and
the batching context (`pf_ctx_run_batch`).  Sizes are those of the workloads,
of the request mixes in ``workloads.py`` and of the tests, or parts of them
that one GPU finishes in well under two seconds.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1606_08281_gb300 import pf
from paper_1606_08281_gb300 import workloads as W

# Work of one SSA event in FP64 operations: for R reactions R propensity
# products, R - 1 prefix sums, u2 a0, t + tau, one Exp(1) variate and one
# division (multiply-adds count two): 21 for R = 4, 53 for R = 20.
EVENT_FLOPS = {"birth_death": 17, "telegraph": 21, "gene_expression": 21, "cascade": 53, "lac_gfp": 49}
# Mean events per particle and unit of time over the workload's parameter
# prior (lac_gfp: over the neighbourhood of theta*).
EVENT_RATE = {"birth_death": 9.0, "telegraph": 0.006, "gene_expression": 3.5, "cascade": 110.0, "lac_gfp": 3500.0}


def listed():
    return [
        # the sampler scores one candidate theta from host memory: the smallest call, all latency
        {"name": "one_theta", "kind": "filter", "net": "birth_death", "M": 1, "T": 1, "K": 20, "N": 100, "host": True},
        # the birth-death workload as benchmarked: few filters, each split over a 4-block cluster
        {"name": "birth_death", "kind": "filter", "net": "birth_death", "M": 200, "T": 1, "K": 20, "N": 100, "cluster": 4},
        # the RNA model's whole batch with its diagnostics: many cheap filters, few events each
        {"name": "telegraph", "kind": "filter", "net": "telegraph", "M": 4096, "T": 1, "K": 25, "N": 200, "diagnostics": True},
        # the main workload: gene expression at full size per theta, prior draws, a quarter of its rows
        {"name": "gene_expression", "kind": "filter", "net": "gene_expression", "M": 1024, "T": 10, "K": 50, "N": 1000},
        # a later level set with early rejection against its threshold; odd sizes
        {"name": "gene_reject", "kind": "filter", "net": "gene_expression", "M": 333, "T": 3, "K": 23, "N": 777, "reject": -4.5},
        # ten species and twenty reactions at full size per filter, population on chip
        {"name": "cascade", "kind": "filter", "net": "cascade", "M": 64, "T": 16, "K": 60, "N": 512},
        # the same network with 4096 particles: populations beyond shared memory
        {"name": "cascade_large", "kind": "filter", "net": "cascade", "M": 38, "T": 8, "K": 10, "N": 4096},
        # the paper's Lac-Gfp network with its model extensions, near theta*, split over clusters
        {"name": "lac_gfp", "kind": "filter", "net": "lac_gfp", "M": 24, "T": 4, "K": 12, "N": 200, "cluster": 4, "spread": 0.5},
        # the exact likelihood of the RNA model for its whole batch
        {"name": "fsp_telegraph", "kind": "fsp", "net": "telegraph", "M": 4096, "K": 25},
        # the exact likelihood of birth-death on its 1201-state box
        {"name": "fsp_birth_death", "kind": "fsp", "net": "birth_death", "M": 200, "K": 20},
        # the deterministic Erk model for a level set near theta-bar
        {"name": "erk", "kind": "erk", "M": 4096, "K": 60, "patterns": 6},
        # requests of a serving window, mixed networks and sizes, in one batch
        {"name": "batch", "kind": "batch", "requests": 24, "N": 256},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["filter"] * 7 + ["fsp", "fsp", "erk", "erk", "batch"])
    if kind == "batch":
        return {"kind": "batch", "requests": rng.randint(2, 32), "N": rng.choice([128, 200, 256, 333, 512])}
    if kind == "erk":
        return {"kind": "erk", "M": _log(rng, 16, 4096), "K": rng.randint(5, 60), "patterns": rng.randint(1, 6)}
    if kind == "fsp":
        net = rng.choice(["telegraph", "birth_death"])
        return {"kind": "fsp", "net": net, "M": _log(rng, 8, 4096 if net == "telegraph" else 200),
                "K": rng.randint(3, 25 if net == "telegraph" else 20)}
    net = rng.choice(["birth_death", "telegraph", "gene_expression", "gene_expression", "cascade", "cascade", "lac_gfp"])
    w = W.get(net)
    c = {"kind": "filter", "net": net, "T": rng.randint(1, w.T), "K": rng.randint(max(1, w.K // 5), w.K)}
    if net == "lac_gfp":
        c |= {"N": _log(rng, 64, 400), "K": rng.randint(3, 12), "spread": 0.5}
    else:
        c["N"] = _log(rng, 64, 4096)
    if net == "cascade":
        c["K"] = rng.randint(5, 60)
    if rng.random() < 0.4:
        c["cluster"] = rng.choice([2, 4])
        if c["N"] > 2048:
            c["N"] -= 2048
    if net != "telegraph" and net != "lac_gfp" and rng.random() < 0.3:
        c["reject"] = -4.5 if net != "cascade" else -12.0
    if rng.random() < 0.3:
        c["diagnostics"] = True
    # no more work than the largest listed case of its network (the prior's
    # heaviest rows set the time of a small draw, so the bound is on events)
    most = {"birth_death": 4e8, "telegraph": 4e8, "gene_expression": 4e9, "cascade": 3e9, "lac_gfp": 6e8}[net]
    per_theta = c["T"] * c["N"] * float(w.obs_times[c["K"] - 1]) * EVENT_RATE[net]
    top = max(1, min(w.M, int(most / max(per_theta, 1.0))))
    c["M"] = _log(rng, 1, top)
    if rng.random() < 0.15:
        c["host"] = True
    return c


class _Context:
    """A batching context with the problems loaded, destroyed with the state."""

    def __init__(self, problems):
        self.h = pf.pf_ctx_create(0, 1, 1024)
        self.ids = {}
        for name in problems:
            w = W.get(name)
            self.ids[name] = pf.pf_ctx_load_problem(self.h, w.net, len(w.prior_lo), w.x0, w.obs_times,
                                                    w.observations(), w.C, w.sigma, model=w.model)

    def __del__(self):
        h, self.h = self.h, None
        if h is not None:
            pf.pf_ctx_destroy(h)


def _thetas(w, M, seed, spread=None):
    rng = np.random.default_rng([seed, w.theta_seed])
    lo, hi = w.prior_lo, w.prior_hi
    if spread is not None:
        lo = np.maximum(lo, w.theta_star * np.exp(-spread))
        hi = np.minimum(hi, w.theta_star * np.exp(spread))
    return W.log_uniform(rng, lo, hi, M)


def _erk_thetas(e, M, seed):
    rng = np.random.default_rng([seed, e.theta_seed])
    return W.log_uniform(rng, np.maximum(e.prior_lo, e.theta_bar / math.e),
                         np.minimum(e.prior_hi, e.theta_bar * math.e), M)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        rng = np.random.default_rng([case["requests"], case["N"]])     # the mix's sizes; its values come from `seed`
        reqs = []
        for i in range(case["requests"]):
            # the serving stream's sizes: level-set batches of two networks, and birth-death
            name = ["gene_expression", "cascade", "birth_death"][int(rng.integers(3))]
            hi = {"gene_expression": 512, "cascade": 32, "birth_death": 512}[name]
            K = {"gene_expression": 10, "cascade": 5, "birth_death": 20}[name]
            M = int(np.exp(rng.uniform(np.log(1), np.log(hi + 1))))
            reqs.append((name, _thetas(W.get(name), M, seed * 1000 + i), case["N"], K, seed * 1000 + i))
        return {"kind": kind, "ctx": _Context(["gene_expression", "cascade", "birth_death"]), "reqs": reqs}
    if kind == "erk":
        e = W.erk()
        return {"kind": kind, "patterns": e.patterns[:case["patterns"]], "times": e.obs_times[:case["K"]],
                "y": _dev(e.observations()[:case["patterns"], :case["K"]]), "theta": _dev(_erk_thetas(e, case["M"], seed))}
    w = W.get(case["net"])
    T, K = case.get("T", 1), case["K"]
    y = w.observations()[:T, :K]
    theta = _thetas(w, case["M"], seed, case.get("spread"))
    if not case.get("host"):
        y, theta = _dev(y), _dev(theta)
    st = {"kind": kind, "w": w, "times": w.obs_times[:K], "y": y, "theta": theta}
    if kind == "filter":
        st |= {"N": case["N"], "seed": w.filter_seed + seed, "options": {}}
        if case.get("cluster"):
            st["options"]["cluster_blocks"] = case["cluster"]
        if case.get("diagnostics"):
            st["options"]["diagnostics"] = True
        if case.get("reject") is not None:
            st["options"]["reject_below"] = case["reject"] * T * K
    return st


def run(state):
    kind = state["kind"]
    if kind == "batch":
        ctx = state["ctx"]
        reqs = [pf.Request(ctx.ids[name], th, N, s, K_use=K) for name, th, N, K, s in state["reqs"]]
        pf.pf_ctx_run_batch(ctx.h, reqs)
        return [{"loglik": r.loglik, "status": r.status} for r in reqs]
    if kind == "erk":
        return pf.pf_erk_loglik(state["theta"], state["patterns"], state["times"], state["y"])
    w = state["w"]
    if kind == "fsp":
        return pf.pf_fsp_loglik(w.net, state["theta"], w.x0, w.fsp_box, state["times"], state["y"], w.C, w.sigma)
    return pf.pf_loglik(w.net, state["theta"], w.x0, state["times"], state["y"], w.C, w.sigma, state["N"],
                        state["seed"], model=w.model, **state["options"])


def work(case):
    """Input and output bytes, and the FP64 operations of the method as it is
    defined (expected SSA events; Poisson terms of the uniformisation over the
    reachable states; Dormand-Prince steps)."""
    kind = case["kind"]
    if kind == "batch":
        flops = nbytes = 0
        for name, hi, K in (("gene_expression", 512, 10), ("cascade", 32, 5), ("birth_death", 512, 20)):
            n = case["requests"] / 3 * (hi / math.log(hi + 1))     # mean rows of a log-uniform draw
            w = W.get(name)
            flops += n * w.T * case["N"] * float(w.obs_times[K - 1]) * EVENT_RATE[name] * EVENT_FLOPS[name]
            nbytes += n * (8 * len(w.prior_lo) + 9)
        return {"bytes": int(nbytes), "flops": int(flops)}
    M, K = case["M"], case["K"]
    if kind == "erk":
        # about 1450 steps of 1618 operations over the full 120 minutes
        return {"bytes": M * (36 * 8 + 9) + 8 * K * case["patterns"],
                "flops": int(M * case["patterns"] * 1450 * (K / 60) * 1618)}
    w = W.get(case["net"])
    T = case.get("T", 1)
    nbytes = M * (8 * len(w.prior_lo) + 9) + 8 * T * K * w.P
    if kind == "fsp":
        S = 122 if case["net"] == "telegraph" else 1201
        terms = K * (20 if case["net"] == "telegraph" else 900)
        return {"bytes": nbytes, "flops": int(M * S * terms * 2 * (w.R + 2))}
    if case.get("diagnostics"):
        nbytes += M * T * 24
    events = M * T * case["N"] * float(w.obs_times[K - 1]) * EVENT_RATE[case["net"]]
    return {"bytes": nbytes, "flops": int(events * EVENT_FLOPS[case["net"]])}


# ----------------------------------------------------------------------------
# the same values in 64 bits by plain torch
# ----------------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind == "fsp":
        w = W.get(case["net"])
        ll = _exact_fsp(w, _thetas(w, case["M"], seed), w.obs_times[:case["K"]], w.observations()[0, :case["K"]])
        return {"loglik": ll, "status": None}
    if kind == "erk" and case["M"] * case["patterns"] <= 4096 * 6:
        e = W.erk()
        ll = _exact_erk(_erk_thetas(e, case["M"], seed), e.patterns[:case["patterns"]], e.obs_times[:case["K"]],
                        e.observations()[:case["patterns"], :case["K"]])
        return {"loglik": ll, "status": None}
    # The filter's value is a Monte Carlo estimate along the library's random
    # stream: one network is restated here in full; the others' event counts
    # put a plain evaluation beyond its time.
    if (kind == "filter" and case["net"] == "birth_death" and not case.get("reject") and
            case["M"] * case["T"] * case["N"] <= 2_000_000 and case["M"] * case["T"] <= 2000):
        w = W.get("birth_death")
        ll = _exact_birth_death(w, _thetas(w, case["M"], seed), w.obs_times[:case["K"]],
                                w.observations()[:case["T"], :case["K"], 0], case["N"], w.filter_seed + seed)
        out = {"loglik": ll.sum(1), "status": None}
        if case.get("diagnostics"):
            out |= {"ll_traj": ll, "events": None, "digest": None}
        return out
    return None


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _exact_fsp(w, thetas, times, y):
    """Forward algorithm on the box by uniformisation with a far longer series
    than 64 bits need: only sums of non-negative terms, so every state's
    probability is accurate to its own last places."""
    dev = _device()
    box = [int(b) for b in w.fsp_box]
    shape = [b + 1 for b in box]
    S = int(np.prod(shape))
    x = torch.stack(torch.meshgrid(*[torch.arange(n, device=dev) for n in shape], indexing="ij"), -1).reshape(S, -1)
    th = torch.from_numpy(thetas).to(dev)
    M = th.shape[0]
    reac = torch.from_numpy(np.asarray(w.net["reactants"], np.int64)).to(dev)
    nu = torch.from_numpy(np.asarray(w.net["products"], np.int64)).to(dev) - reac
    strides = torch.tensor([int(np.prod(shape[u + 1:])) for u in range(len(shape))], device=dev)
    # first-order and zero-order reactions only (both networks)
    h = torch.where(reac[None] > 0, x[:, None, :], torch.ones_like(x)[:, None, :]).prod(-1).double()   # [S][R]
    a0 = th @ h.T
    lam = a0.max(1).values[:, None]
    stay = (lam - a0) / lam
    flows = []
    for r in range(reac.shape[0]):
        z = x - nu[r]
        ok = ((z >= 0) & (z <= torch.tensor(box, device=dev))).all(-1)
        src = torch.where(ok, (z * strides).sum(-1), torch.zeros_like(ok, dtype=torch.long))
        flows.append((src, th[:, r:r + 1] / lam * torch.where(ok, h[src, r], torch.zeros(S, device=dev, dtype=torch.float64))))
    p = torch.zeros(M, S, dtype=torch.float64, device=dev)
    p[:, int((torch.from_numpy(w.x0.astype(np.int64)).to(dev) * strides).sum())] = 1.0
    C = torch.from_numpy(w.C[0]).to(dev)
    mu = x.double() @ C
    sigma = float(w.sigma[0])
    ll = torch.zeros(M, dtype=torch.float64, device=dev)
    t = 0.0
    for k, tk in enumerate(times):
        lh = lam[:, 0] * (tk - t)
        top = float(lh.max())
        n = int(math.ceil(top + 12.0 * math.sqrt(top) + 60.0))
        lg = torch.log(lh)
        acc = torch.exp(-lh)[:, None] * p
        for j in range(1, n + 1):
            q = stay * p
            for src, c in flows:
                q = q + c * p[:, src]
            p = q
            acc = acc + torch.exp(j * lg - lh - math.lgamma(j + 1.0))[:, None] * p
        le = -0.5 * ((float(y[k, 0]) - mu) / sigma) ** 2 - math.log(sigma) - 0.5 * math.log(2.0 * math.pi)
        m = torch.where(acc > 0, le[None].expand(M, S), torch.full((), -math.inf, device=dev, dtype=torch.float64)).max(1).values
        v = acc * torch.exp(le[None] - m[:, None])
        v = torch.where(acc > 0, v, torch.zeros_like(v))
        c = v.sum(1)
        ll = ll + m + torch.log(c)
        p = v / c[:, None]
        t = float(tk)
    return ll.cpu().numpy()


def _exact_erk(thetas, patterns, times, y):
    """Every (theta, pattern) by extrapolated modified-midpoint steps of at
    most a tenth of a minute, all together: an error near 1e-13."""
    dev = _device()
    th = torch.from_numpy(thetas).to(dev)
    M, NP = th.shape[0], len(patterns)
    th = th[:, None, :].expand(M, NP, 36).reshape(M * NP, 36).T.contiguous()
    a = math.log10(2.0) / 90.0
    k = th
    pack = lambda rows: torch.stack(rows)  # noqa: E731
    one = torch.ones_like(k[0])
    kA = pack([k[2], k[6] * k[8] ** 2, k[11], k[15], k[19]])
    KA = pack([k[3], k[7], k[12], k[16], k[20]])
    kB = pack([k[4], k[9], k[13], k[17], k[22]])
    KB = pack([k[5], k[10], k[14], k[18], k[23]])
    hill = k[8] ** 2

    def f(x, u):
        act = x[[1, 3, 5, 7, 9]]
        sub, prod = x[[2, 4, 6, 8, 10]], x[[3, 5, 7, 9, 11]]
        up = kA * act * sub / (KA + sub)
        dn = kB * prod / (KB + prod)
        e2, n2, r2 = x[1] ** 2, x[11] ** 2, x[9] ** 2
        v3 = up[1] / (hill + n2) - dn[1]
        v6 = up[4] * e2 / (k[21] ** 2 + e2) - dn[4]
        v1 = k[0] * u * x[0] - k[1] * x[1]
        v2, v4, v5 = up[0] - dn[0], up[2] - dn[2], up[3] - x[13] * dn[3]
        d12 = a * (k[24] * (1.0 + k[25] * r2 / (k[26] + r2)) - x[12])
        return torch.stack([-v1, v1, -v2, v2, -v3, v3, -v4, v4, -v5, v5, -v6, v6, d12, a * (x[12] - x[13])])

    seq = [2, 4, 6, 8, 10, 12]

    def step(x, u, H):
        tab = []
        f0 = f(x, u)
        for i, n in enumerate(seq):
            h = H / n
            z0, z1 = x, x + h * f0
            for _ in range(1, n):
                z0, z1 = z1, z0 + 2.0 * h * f(z1, u)
            row = [0.5 * (z1 + z0 + h * f(z1, u))]
            for q in range(i):
                row.append(row[q] + (row[q] - tab[i - 1][q]) / ((seq[i] / seq[i - 1 - q]) ** 2 - 1.0))
            tab.append(row)
        return tab[-1][-1]

    zero = torch.zeros_like(one)
    x = torch.stack([k[27], zero, 0.1 * one, zero, 0.7 * one, zero, 0.68 * one, zero, 0.26 * one, zero, k[28], zero, k[29], k[29]])
    stops = sorted(set(float(t) for t in times) | {float(s) for st, _ in patterns for s in st if 0.0 < s < times[-1]})
    ll = torch.zeros(M * NP, dtype=torch.float64, device=dev)
    where = {float(t): i for i, t in enumerate(times)}
    t = 0.0
    for s in stops:
        u = torch.tensor([float(sv[np.searchsorted(st, t, side="right") - 1]) if t >= st[0] else 0.0
                          for st, sv in patterns], dtype=torch.float64, device=dev).repeat(M)
        n = int(math.ceil((s - t) / 0.1 - 1e-9))
        for _ in range(n):
            x = step(x, u, (s - t) / n)
        t = s
        if s in where:
            R = k[31] * (x[9] * k[33] * k[34] / ((x[8] + (1.0 - k[33]) * x[9]) * k[35]) + k[30])
            yk = torch.from_numpy(np.ascontiguousarray(y[:, where[s]])).to(dev).repeat(M)
            ll = ll - 0.5 * ((yk - R) / k[32]) ** 2 - torch.log(k[32]) - 0.5 * math.log(2.0 * math.pi)
    return ll.reshape(M, NP).sum(1).cpu().numpy()


_M32 = 0xFFFFFFFF


def _mulhilo(c, v):
    lo16, hi16 = v & 0xFFFF, v >> 16
    p0, p1 = c * lo16, c * hi16
    return ((p0 >> 16) + p1) >> 16, (p0 + ((p1 & 0xFFFF) << 16)) & _M32


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors of 32-bit words."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for i in range(10):
        ha, la = _mulhilo(0xD2511F53, c0)
        hb, lb = _mulhilo(0xCD9E8D57, c2)
        c0, c1, c2, c3 = hb ^ c1 ^ k0, lb, ha ^ c3 ^ k1, la
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _u53(hi, lo):
    return (hi << 21) | (lo >> 11)


def _ziggurat(dev):
    r, v, n = 10.02289706840504086041, 0.0004891103607436302956561, 2048
    x = [v / math.exp(-r), r]
    for i in range(1, n - 1):
        x.append(-math.log(v / x[i] + math.exp(-x[i])))
    x.append(0.0)
    return torch.tensor(x, dtype=torch.float64, device=dev), r


def _exp1(hi, lo, draw, part, lane, row, seed, zx, r):
    """Exp(1) variates by the 2048-layer ziggurat (Marsaglia & Tsang 2000)."""
    E = torch.zeros(hi.shape, dtype=torch.float64, device=hi.device)
    todo = torch.arange(hi.numel(), device=hi.device)
    s, words = 0, None
    while todo.numel():
        i = lo & 0x7FF
        xi = zx[i]
        x = (_u53(hi, lo).double() * 2.0 ** -53) * xi
        fast = x < zx[i + 1]
        E[todo[fast]] = x[fast]
        keep = ~fast
        todo, i, xi, x = todo[keep], i[keep], xi[keep], x[keep]
        if not todo.numel():
            break
        s += 1
        w0, w1, w2, w3 = _philox(draw[todo], part[todo] | (s << 16), lane[todo], row[todo], seed)
        U = _u53(w1, w0)
        tail = i == 0
        E[todo[tail]] = r - torch.log((U[tail] + 1).double() * 2.0 ** -53)
        f, f1 = torch.exp(-xi), torch.exp(-zx[i + 1])
        ok = ~tail & (f + (U.double() * 2.0 ** -53) * (f1 - f) < torch.exp(-x))
        E[todo[ok]] = x[ok]
        keep = ~(tail | ok)
        todo, hi, lo = todo[keep], w3[keep], w2[keep]
    return E


def _exact_birth_death(w, thetas, times, y, N, seed):
    """The bootstrap filter of 0 -> X, X -> 0 along the library's stream."""
    dev = _device()
    M, T = thetas.shape[0], y.shape[0]
    F = M * T
    zx, r = _ziggurat(dev)
    th = torch.from_numpy(thetas).to(dev).repeat_interleave(T, 0)
    m_f = torch.arange(M, device=dev).repeat_interleave(T)
    t_f = torch.arange(T, device=dev).repeat(M)
    x = torch.full((F, N), int(w.x0[0]), dtype=torch.int64, device=dev)
    ll = torch.zeros(F, dtype=torch.float64, device=dev)
    sigma = float(w.sigma[0])
    q, prev = None, 0.0
    for k, tk in enumerate(times):
        lane_f = (t_f << 20) | k
        if q is not None:
            Q = torch.cumsum(q, 1)
            Wt = Q[:, -1]
            ones = torch.zeros_like(lane_f)
            w0, w1, _, _ = _philox(ones, ones + _M32, lane_f, m_f, seed)
            u = torch.tensor([(((int(b) << 32) | int(c)) * int(v)) >> 64 for b, c, v in zip(w1.cpu(), w0.cpu(), Wt.cpu())],
                             dtype=torch.int64, device=dev)
            point = u[:, None] + torch.arange(N, device=dev)[None] * Wt[:, None]
            x = torch.gather(x, 1, torch.searchsorted(N * Q, point, right=True))
        flat = x.reshape(-1).clone()
        act = torch.arange(F * N, device=dev)
        now = torch.full((F * N,), prev, dtype=torch.float64, device=dev)
        draws = 0
        while act.numel():
            f = act // N
            part = act - f * N
            d = torch.full_like(act, draws)
            w0, w1, w2, w3 = _philox(d, part, lane_f[f], m_f[f], seed)
            a1 = th[f, 0]
            a0 = a1 + th[f, 1] * flat[act].double()
            nxt = now[act] + _exp1(w1, w0, d, part, lane_f[f], m_f[f], seed, zx, r) / a0
            go = nxt <= tk
            up = (_u53(w3, w2).double() * 2.0 ** -53) * a0 < a1
            act, nxt, up = act[go], nxt[go], up[go]
            flat[act] += torch.where(up, 1, -1)
            now[act] = nxt
            draws += 1
        x = flat.reshape(F, N)
        e = -0.5 * ((torch.from_numpy(np.ascontiguousarray(y[:, k])).to(dev)[t_f][:, None] - x.double()) / sigma) ** 2
        top = e.max(1).values
        g = torch.exp(e - top[:, None])
        q = (g * 2.0 ** 32).long()
        ll = ll + top + torch.log(g.sum(1)) - math.log(N) - math.log(sigma) - 0.5 * math.log(2.0 * math.pi)
        prev = float(tk)
    return ll.reshape(M, T).cpu().numpy()
