"""Performance cases of the TNVAN library: what a user's program has it do, over the range it is used in.

A case is a plain dict:
  op      "step"      one iteration of Algorithm 1 (TNVAN.train_step, or a replay of TNVAN.capture_train_step)
          "sample"    sampling with log q and log Z_R (TNVAN.sample)
          "log_prob"  log q of given configurations (Context.log_prob)
          "contract"  log Z_R of given configurations, optionally with d/dbeta (Context.contract)
          "backward"  the gradient of F_q from given samples, optionally with d/dbeta and d/dJ (Context.backward)
          "moments"   conditional magnetisation and its averages (Context.magnetisation)
          "observables"  internal energy and bond correlations (Context.observables)
  graph   "lattice" (L x L, the columns c with c % period == period - 1 in W), "mixed" (lattices of several L),
          "sk" (n spins, the last `rest` left to the contraction), "rrg" (n spins of degree `degree`, W found for
          elimination width `width`)
  dist    couplings: "gauss", "pm1" or "ferro"
  inst    instances, each with couplings and an inverse temperature of its own
  hidden  the network's hidden widths, as "128,128"
  prec    "fp32", "tf32" or "bf16"
  batch   samples per instance
"""
import functools
import math

import numpy as np
import torch

from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

PREC = {"fp32": tv.FP32, "tf32": tv.TF32, "bf16": tv.BF16}
MIXED = (8, 12, 16, 24, 32)
BASE = {"graph": "lattice", "dist": "gauss", "inst": 1, "hidden": "128,128", "prec": "bf16", "adjoint": False,
        "capture": False, "period": 4, "L": 16, "n": 64, "rest": 16, "degree": 3, "width": 8}


def listed():
    cases = [
        # the smallest problem in use: a 4x4 lattice's training step, launched call by call (launch latency)
        {"name": "step_4x4", "op": "step", "dist": "pm1", "L": 4, "period": 3, "hidden": "16", "batch": 1024},
        # the benchmark's training step: five temperatures of a 16x16 lattice, captured once and replayed
        {"name": "step_ea16", "op": "step", "inst": 5, "batch": 16384, "adjoint": True, "capture": True},
        # many instances of different sizes trained side by side
        {"name": "step_mixed", "op": "step", "graph": "mixed", "inst": 64, "batch": 1024, "capture": True},
        # drawing samples of the fully connected model with the wider network
        {"name": "sample_sk64", "op": "sample", "graph": "sk", "inst": 3, "hidden": "256,256", "batch": 4096},
        # samples in single precision, a ragged batch (the final estimates of a run)
        {"name": "sample_ea16_fp32", "op": "sample", "inst": 5, "prec": "fp32", "batch": 4099},
        # log q of given configurations, the largest network input (256 spins), a ragged batch
        {"name": "log_prob_ea32", "op": "log_prob", "L": 32, "inst": 3, "batch": 5003},
        # exact contraction of many given configurations with the conditional energy (estimates after training)
        {"name": "contract_ea16", "op": "contract", "inst": 5, "batch": 65536, "adjoint": True},
        # the 40x40 ferromagnet at six temperatures: strips of 12 columns
        {"name": "contract_ferro40", "op": "contract", "dist": "ferro", "L": 40, "period": 13, "inst": 6,
         "hidden": "256,256", "batch": 1000},
        # the gradient of the wider network in reduced precision
        {"name": "backward_sk64", "op": "backward", "graph": "sk", "inst": 3, "hidden": "256,256", "batch": 4096},
        # the gradient in single precision, the full batch of the benchmark
        {"name": "backward_ea16_fp32", "op": "backward", "inst": 5, "prec": "fp32", "batch": 16384},
        # a random regular graph with a found width set: gradient with d/dbeta and d/dJ through the elimination
        {"name": "backward_rrg500", "op": "backward", "graph": "rrg", "dist": "pm1", "n": 500, "batch": 4096,
         "adjoint": True},
        # magnetisation and susceptibility from samples
        {"name": "moments_ea16", "op": "moments", "inst": 5, "batch": 2048},
    ]
    return [{**BASE, **c} for c in cases]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    op = rng.choice(("step", "step", "sample", "sample", "log_prob", "contract", "contract", "backward", "backward",
                     "moments", "observables"))
    c = dict(BASE, op=op)
    c["graph"] = rng.choice(("lattice", "lattice", "lattice", "sk", "rrg"))
    c["dist"] = "pm1" if c["graph"] == "rrg" else rng.choice(("gauss", "gauss", "pm1"))
    c["inst"] = rng.choice((1, 1, 2, 3, 4, 5))
    c["hidden"] = rng.choice(("16", "64", "32,48", "64,64", "128,128", "128,128", "256,256"))
    c["prec"] = rng.choice(("bf16", "bf16", "fp32", "tf32" if op == "backward" else "bf16"))
    small = c["prec"] == "fp32" or c["graph"] != "lattice"
    most = {"step": 8192, "sample": 8192, "log_prob": 16384, "contract": 65536, "backward": 16384, "moments": 2048,
            "observables": 4096}[op]
    c["batch"] = _log_int(rng, 64, most // 2 if small else most)
    if c["graph"] == "lattice":
        c["L"] = rng.randint(4, 24)
        c["period"] = rng.randint(2, min(5, c["L"]))
        if op == "contract" and rng.random() < 0.3:  # wide strips
            c["L"], c["period"] = rng.randint(13, 40), rng.randint(6, 13)
            c["batch"] = _log_int(rng, 64, 1000)
            c["dist"] = rng.choice(("ferro", "gauss", "pm1"))
    elif c["graph"] == "sk":
        c["rest"] = rng.randint(10, 16)
        c["n"] = c["rest"] + rng.randint(8, 64)
        c["dist"] = "gauss"
    else:
        c["degree"] = rng.choice((3, 3, 4))
        c["n"] = 2 * rng.randint(32, 250 if c["degree"] == 3 else 120)
        c["width"] = rng.randint(1, 8)
        c["batch"] = min(c["batch"], 4096)
    if op in ("step", "contract", "backward"):
        c["adjoint"] = c["period"] <= 5 and rng.random() < 0.5
    if op == "step":
        c["capture"] = rng.random() < 0.5
    return c


# ---------------------------------------------------------------------------
# Problems: graphs, width sets and orders are fixed by the case (as a study of
# one ensemble fixes them), couplings and all values by the seed.
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=16)
def _rrg(n, degree, width):
    g = wl.random_regular(n, degree, 1)
    W, order, _, _ = tv.find_width_set(n, g.ei, g.ej, width, 1, 0, tv.SLICE_GREEDY)
    return g, W, order


def _problem(case, seed):
    graphs, Ws, orders = [], [], []
    for k in range(case["inst"]):
        s = 1000 * seed + k
        if case["graph"] == "sk":
            g = wl.sk(case["n"], s)
            graphs.append(g)
            Ws.append(np.arange(case["n"] - case["rest"], dtype=np.int32))
            orders.append(None)
        elif case["graph"] == "rrg":
            g, W, order = _rrg(case["n"], case["degree"], case["width"])
            J = np.random.default_rng(s).choice(np.array([-1.0, 1.0]), size=g.m)
            graphs.append(wl.Graph(g.n, g.ei, g.ej, J))
            Ws.append(W)
            orders.append(order)
        else:
            L = MIXED[k % len(MIXED)] if case["graph"] == "mixed" else case["L"]
            g = wl.lattice(L, L, case["dist"], s)
            cols = wl.every_kth_column(L, case["period"])
            W = wl.width_columns(L, L, cols)
            graphs.append(g)
            Ws.append(W)
            wset = set(W.tolist())
            orders.append(np.asarray([v for v in range(L * L) if v not in wset], np.int32)
                          if case["period"] > 5 else None)
    n = case["inst"]
    if case["dist"] == "ferro" and case["graph"] == "lattice":
        temps = [1.0, 2.0, 2.0 / math.log(1.0 + math.sqrt(2.0)), 3.0, 4.0, 5.0]
        betas = [1.0 / temps[k % 6] for k in range(n)]
    elif case["graph"] == "mixed":
        betas = [0.8] * n
    else:
        betas = [(k + 1) / n for k in range(n)]
    hidden = [int(h) for h in case["hidden"].split(",")]
    return graphs, Ws, orders, hidden, betas


def _params(Ws, hidden, seed):
    return np.concatenate([wl.made_params(len(W), hidden, 77 + 1000 * seed + k) for k, W in enumerate(Ws)])


def _values(case, Ws, seed, device="cuda"):
    """Seeded configurations and per-sample values: log q near that of an untrained network, log Z_R with the
    spread of a batch (a few units around its mean)."""
    B, n = case["batch"], len(Ws)
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    D = [len(W) for W in Ws]
    spins = (torch.randint(0, 2, (B * sum(D),), generator=gen, device=device, dtype=torch.int8) * 2 - 1)
    logq = torch.cat([-d * math.log(2.0) + torch.randn(B, generator=gen, device=device) for d in D])
    logZR = 100.0 + 2.0 * torch.randn(n * B, generator=gen, device=device, dtype=torch.float64)
    return spins, logq, logZR


def prepare(case, seed):
    case = {**BASE, **case}
    graphs, Ws, orders, hidden, betas = _problem(case, seed)
    B, op, prec = case["batch"], case["op"], PREC[case["prec"]]
    model = TNVAN(graphs, Ws, hidden, betas, params=_params(Ws, hidden, seed),
                  elim_orders=orders if any(o is not None for o in orders) else None)
    model.ctx.reserve(B)
    n, dev = model.n, model.device
    s = {"op": op, "model": model, "batch": B, "prec": prec, "seed": seed, "pass": 0}
    f64 = dict(dtype=torch.float64, device=dev)
    s["dbeta"] = torch.zeros(n * B, **f64) if case["adjoint"] else None
    s["dJ"] = torch.zeros(sum(model.n_edges), **f64) if case["adjoint"] else None
    if op in ("step", "sample"):
        s["out"] = model.buffers(B)
    else:
        s["spins"], s["logq"], s["logZR"] = _values(case, Ws, seed)
    if op == "step":
        # a run resumed from a checkpoint in mid-training: Adam moments of the gradients' size
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed + 1)
        p = model.params
        model.m.copy_(0.01 * torch.randn(p.shape, generator=gen, device=dev))
        model.v.copy_(1e-3 * (0.5 + torch.rand(p.shape, generator=gen, device=dev)))
        model.t = 1000
        s["live"] = [model.params, model.m, model.v]
        s["saved"] = [t.clone() for t in s["live"]]
        s["stats"] = torch.zeros(8 * n, **f64)
        if case["capture"]:
            s["step"] = model.capture_train_step(B, seed, prec, 0.01, s["out"], s["dbeta"], s["dJ"])
    elif op == "log_prob":
        s["logq"] = torch.empty(n * B, dtype=torch.float32, device=dev)
    elif op == "contract":
        s["logZR"] = torch.empty(n * B, **f64)
    elif op == "moments":
        s["mean"], s["var"] = torch.empty(n * B, **f64), torch.empty(n * B, **f64)
    elif op == "observables":
        s["corr"] = torch.empty(sum(model.n_edges), **f64)
    return s


def _some(d):
    return {k: v for k, v in d.items() if v is not None}


def run(s):
    m, B, prec, op = s["model"], s["batch"], s["prec"], s["op"]
    if op == "step":
        # every pass takes one step from the checkpoint (with samples of its own), as a scan over step sizes does
        s["pass"] += 1
        torch._foreach_copy_(s["live"], s["saved"])
        if "step" in s:
            s["step"].replay()
            stats = s["step"].stats
        else:
            m.t = 1000
            m.train_step(B, s["seed"], s["pass"], prec, 0.01, s["out"], s["dbeta"], s["dJ"])
            stats = m.step_stats(s["stats"])
        spins, logq, logZR = s["out"]
        return _some({"spins": spins, "logq": logq, "logZR": logZR, "dbeta": s["dbeta"], "dJ": s["dJ"], "stats": stats,
                      "grad": m.grad, "params": m.params, "m": m.m, "v": m.v})
    if op == "sample":
        s["pass"] += 1
        spins, logq, logZR = m.sample(B, s["seed"], s["pass"], prec, s["out"])
        return {"spins": spins, "logq": logq, "logZR": logZR}
    if op == "log_prob":
        m.ctx.log_prob(B, s["spins"], s["logq"], prec)
        return {"logq": s["logq"]}
    if op == "contract":
        m.ctx.contract(m.betas, B, s["spins"], prec, s["logZR"], s["dbeta"])
        return _some({"logZR": s["logZR"], "dbeta": s["dbeta"]})
    if op == "backward":
        m.ctx.backward(m.betas, B, s["spins"], s["logZR"], s["logq"], prec, m.grad, s["dbeta"], s["dJ"])
        return _some({"grad": m.grad, "dbeta": s["dbeta"], "dJ": s["dJ"]})
    if op == "moments":
        avg = m.ctx.magnetisation(m.betas, B, s["spins"], s["logZR"], s["logq"], s["mean"], s["var"])
        return {"averages": avg, "mean": s["mean"], "var": s["var"]}
    avg = m.ctx.observables(m.betas, B, s["spins"], s["logZR"], s["logq"], s["corr"])
    return {"averages": avg, "corr": s["corr"]}


# ---------------------------------------------------------------------------
# Work: what the path cannot do without (masked network products counted once,
# each input read once and each output written once).
# ---------------------------------------------------------------------------

def _degrees(D, hidden):
    cyc = max(D - 1, 1)
    return [np.arange(1, D + 1)] + [np.arange(H) % cyc + 1 for H in hidden] + [np.arange(1, D + 1)]


def _masks(D, hidden):
    deg = _degrees(D, hidden)
    last = len(deg) - 2
    return [(deg[l + 1][:, None] > deg[l][None, :]) if l == last else (deg[l + 1][:, None] >= deg[l][None, :])
            for l in range(last + 1)]


def _contraction_flops(case, g, W):
    """Multiply-adds of one sample's forward contraction."""
    if case["graph"] == "sk":
        return 2.0 * 2.0 ** case["rest"]
    if case["graph"] == "rrg":
        _, W, order = _rrg(case["n"], case["degree"], case["width"])
        wset = set(W.tolist())
        adj = [set() for _ in range(g.n)]
        for a, b in zip(g.ei.tolist(), g.ej.tolist()):
            if a not in wset and b not in wset:
                adj[a].add(b)
                adj[b].add(a)
        total = 0.0
        for v in order.tolist():
            nb = adj[v]
            total += 4.0 * 2.0 ** (len(nb) + 1)
            for a in nb:
                adj[a].discard(v)
                adj[a].update(u for u in nb if u != a)
        return total
    L = g.Lx
    cols = sorted(set((W % L).tolist()))
    bands = np.diff([-1] + cols + [L]) - 1
    return float(sum(L * (2.0 * w * 2 ** w + 2.0 * 2 ** w) for w in bands if w > 0))


def work(case):
    case = {**BASE, **case}
    graphs, Ws, _, hidden, _ = _problem(case, 1)
    op, B = case["op"], case["batch"]
    flops = nbytes = 0.0
    for g, W in zip(graphs, Ws):
        D = len(W)
        macs = float(sum(m.sum() for m in _masks(D, hidden)))
        P = wl.made_param_count(D, hidden)
        con = _contraction_flops(case, g, W)
        adj = 3.0 * con if case["adjoint"] else 0.0
        nbytes += D * B
        if op in ("step", "sample", "log_prob"):
            flops += 2.0 * macs * B
            nbytes += 4 * P + 4 * B
        if op in ("step", "sample", "contract"):
            flops += con * B
            nbytes += 8 * B
        if op == "step":
            flops += 4.0 * macs * B
            nbytes += 4 * P + 20 * P
        if op == "backward":
            flops += 6.0 * macs * B
            nbytes += 4 * P + 4 * P + 12 * B
        if case["adjoint"]:
            flops += (con if op == "backward" else 0.0) * B + adj * B
            nbytes += 8 * B
        if op in ("moments", "observables"):
            flops += 3.0 * con * B
            nbytes += 12 * B + (16 * B if op == "moments" else 8 * g.m)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# The same values in 64 bits, in plain torch.
# ---------------------------------------------------------------------------

def _log_q(theta, D, hidden, s):
    """log q of configurations s [B, D] (float64), differentiable in theta."""
    sizes = [D] + hidden + [D]
    h, off = s, 0
    masks = _masks(D, hidden)
    for l, m in enumerate(masks):
        nin, nout = sizes[l], sizes[l + 1]
        Wl = theta[off:off + nin * nout].view(nout, nin) * torch.as_tensor(m, dtype=theta.dtype, device=theta.device)
        off += nin * nout
        h = h @ Wl.T + theta[off:off + nout]
        off += nout
        h = torch.relu(h) if l < len(masks) - 1 else h
    return -torch.nn.functional.softplus(-s * h).sum(1)


def _uniforms(seed, step, inst, B, D, device):
    """24-bit uniforms of Philox4x32-10 (Salmon et al., SC 2011): counter (b, i >> 2, step, instance), word i & 3."""
    lo = 0xFFFFFFFF
    nq = (D + 3) // 4
    c = [torch.arange(B, device=device).repeat_interleave(nq), torch.arange(nq, device=device).repeat(B),
         torch.full((B * nq,), step & lo, device=device), torch.full((B * nq,), inst, device=device)]
    k0, k1 = seed & lo, (seed >> 32) & lo

    def mul(a, x):  # 32 x 32 -> (high, low), without overflow in 64 signed bits
        low = a * (x & 0xFFFF)
        t = a * (x >> 16) + (low >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (low & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & lo, (k1 + 0xBB67AE85) & lo
    words = torch.stack(c, 1).view(B, nq * 4)[:, :D]
    return (words >> 8).double() * 2.0 ** -24


def _draw_samples(theta, D, hidden, u):
    sizes = [D] + hidden + [D]
    masks = [torch.as_tensor(m, dtype=theta.dtype, device=theta.device) for m in _masks(D, hidden)]
    layers, off = [], 0
    for l, m in enumerate(masks):
        nin, nout = sizes[l], sizes[l + 1]
        layers.append((theta[off:off + nin * nout].view(nout, nin) * m, theta[off + nin * nout:off + nin * nout + nout]))
        off += nin * nout + nout
    s = torch.zeros_like(u)
    for i in range(D):
        h = s
        for l, (Wl, bl) in enumerate(layers[:-1]):
            h = torch.relu(h @ Wl.T + bl)
        x = h @ layers[-1][0][i] + layers[-1][1][i]
        s[:, i] = torch.where(u[:, i] < torch.sigmoid(x), 1.0, -1.0)
    return s


def _sign_table(k, device):
    x = torch.arange(2 ** k, device=device)
    return torch.stack([1.0 - 2.0 * ((x >> c) & 1).double() for c in range(k)], 1)  # [2^k, k], first spin fastest


class _Exact:
    """log Z_R of configurations s [B, D] of one instance, differentiable in J [m], beta [B] and field [B] (a uniform
    field on the spins of R, in units of beta)."""

    def __init__(self, g, W, device):
        self.g, self.W, self.dev = g, [int(v) for v in W], device
        self.pos = {v: k for k, v in enumerate(self.W)}
        self.ei, self.ej = g.ei.tolist(), g.ej.tolist()

    def ww(self, J, s):
        idx = [(k, self.pos[a], self.pos[b]) for k, (a, b) in enumerate(zip(self.ei, self.ej))
               if a in self.pos and b in self.pos]
        if not idx:
            return 0.0
        k, a, b = (torch.tensor(v, device=self.dev) for v in zip(*idx))
        return (s[:, a] * s[:, b]) @ J[k]

    def fields(self, J, s, R):
        """h [B, len(R)]: couplings to W's spins."""
        at = {v: k for k, v in enumerate(R)}
        M = torch.zeros(len(self.W), len(R), dtype=torch.float64, device=self.dev)
        e, r, c = [], [], []
        for k, (a, b) in enumerate(zip(self.ei, self.ej)):
            if a in at and b in self.pos:
                a, b = b, a
            if a in self.pos and b in at:
                e.append(k)
                r.append(self.pos[a])
                c.append(at[b])
        if e:
            M = M.index_put((torch.tensor(r, device=self.dev), torch.tensor(c, device=self.dev)),
                            J[torch.tensor(e, device=self.dev)], accumulate=True)
        return s @ M

    def log_z(self, J, beta, s, field=None):
        R = [v for v in range(self.g.n) if v not in self.pos]
        h = beta[:, None] * self.fields(J, s, R)
        if field is not None:
            h = h + field[:, None]
        total = beta * self.ww(J, s)
        if self.g.topology == wl.DENSE:
            return total + self._dense(J, beta, h, R)
        if self.g.topology == wl.LATTICE2D:
            return total + self._strips(J, beta, h, R)
        return total + self._eliminate(J, beta, h, R)

    def _dense(self, J, beta, h, R):
        at = {v: k for k, v in enumerate(R)}
        t = _sign_table(len(R), self.dev)
        e = sum(J[k] * t[:, at[a]] * t[:, at[b]] for k, (a, b) in enumerate(zip(self.ei, self.ej))
                if a in at and b in at)
        return torch.logsumexp(h @ t.T + beta[:, None] * e[None, :], 1)

    def _strips(self, J, beta, h, R):
        L, Ly = self.g.Lx, self.g.Ly
        cols = sorted(set(v % L for v in self.W))
        at = {v: k for k, v in enumerate(R)}
        edge = {(a, b): k for k, (a, b) in enumerate(zip(self.ei, self.ej))}
        out = torch.zeros_like(beta)
        for c0, c1 in zip([-1] + cols, cols + [L]):
            w = c1 - c0 - 1
            if w <= 0:
                continue
            t = _sign_table(w, self.dev)
            v = None
            for y in range(Ly):
                site = [y * L + c0 + 1 + c for c in range(w)]
                d = h[:, [at[i] for i in site]] @ t.T
                for c in range(w - 1):
                    d = d + beta[:, None] * J[edge[(site[c], site[c + 1])]] * (t[:, c] * t[:, c + 1])[None, :]
                if v is None:
                    v = torch.ones_like(d)
                else:
                    for c in range(w):
                        K = beta * J[edge[(site[c] - L, site[c])]]
                        x = v.view(-1, 2 ** (w - 1 - c), 2, 2 ** c)
                        v = (torch.exp(K).view(-1, 1, 1, 1) * x
                             + torch.exp(-K).view(-1, 1, 1, 1) * x.flip(2)).reshape(v.shape)
                top = d.amax(1).detach()
                v = v * torch.exp(d - top[:, None])
                big = v.amax(1).detach()
                v = v / big[:, None]
                out = out + top + torch.log(big)
            out = out + torch.log(v.sum(1))
        return out

    def _eliminate(self, J, beta, h, R):
        at = {v: k for k, v in enumerate(R)}
        sgn = torch.tensor([1.0, -1.0], dtype=torch.float64, device=self.dev)
        factors = {}  # id -> (scope, table [B, 2, ...])
        of = {v: set() for v in R}
        adj = {v: set() for v in R}

        def add(scope, t):
            k = 1 + max(factors, default=0)
            factors[k] = (scope, t)
            for v in scope:
                of[v].add(k)

        for k, (a, b) in enumerate(zip(self.ei, self.ej)):
            if a in at and b in at:
                add((a, b), torch.exp((beta * J[k])[:, None, None] * sgn[:, None] * sgn[None, :]))
                adj[a].add(b)
                adj[b].add(a)
        out = torch.zeros_like(beta)
        left = set(R)
        while left:
            v = min(left, key=lambda u: (len(adj[u]), u))
            left.discard(v)
            scope = sorted(adj[v]) + [v]
            hv = h[:, at[v]]
            t = torch.exp(hv[:, None] * sgn[None, :] - hv.abs().detach()[:, None])
            out = out + hv.abs().detach()
            t = t.view([-1] + [1] * (len(scope) - 1) + [2])
            for k in sorted(of[v]):
                sc, f = factors.pop(k)
                for u in sc:
                    if u != v:
                        of[u].discard(k)
                order = sorted(range(len(sc)), key=lambda i: scope.index(sc[i]))
                f = f.permute([0] + [i + 1 for i in order])
                t = t * f.reshape([f.shape[0]] + [2 if u in sc else 1 for u in scope])
            t = t.sum(-1)
            nb = scope[:-1]
            big = t.reshape(t.shape[0], -1).amax(1).detach()
            out = out + torch.log(big)
            t = t / big.view([-1] + [1] * (t.dim() - 1))
            if nb:
                add(tuple(nb), t)
                for a in nb:
                    adj[a].discard(v)
                    adj[a].update(u for u in nb if u != a)
            else:
                out = out + torch.log(t)
        return out


def exact(case, seed):
    case = {**BASE, **case}
    op, B = case["op"], case["batch"]
    if op == "step" or (op == "sample" and case["prec"] != "fp32"):
        return None  # the samples themselves depend on the rounding of the network
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    graphs, Ws, _, hidden, betas = _problem(case, seed)
    theta_all = torch.as_tensor(_params(Ws, hidden, seed)).double().to(dev)
    spins = logq = logZR = None
    if op != "sample":
        spins, logq, logZR = _values(case, Ws, seed, dev)
    got, at, off = {}, 0, 0

    def put(name, v):
        got.setdefault(name, []).append(v)

    for k, (g, W) in enumerate(zip(graphs, Ws)):
        D = len(W)
        P = wl.made_param_count(D, hidden)
        theta = theta_all[off:off + P].clone()
        off += P
        J = torch.as_tensor(g.J, dtype=torch.float64, device=dev)
        ex = _Exact(g, W, dev)
        if op == "sample":
            s = _draw_samples(theta, D, hidden, _uniforms(seed, 1, k, B, D, dev))
        else:
            s = spins[at:at + B * D].view(B, D).double()
        at += B * D
        if op in ("sample", "log_prob"):
            put("logq", torch.cat([_log_q(theta, D, hidden, x) for x in s.split(16384)]))
        if op in ("sample", "contract") or case["adjoint"]:
            dJ = torch.zeros_like(J)
            for x in s.split(1024 if g.topology != wl.LATTICE2D or case["period"] > 5 else 16384):
                Jx = J.clone().requires_grad_(case["adjoint"])
                b = torch.full((x.shape[0],), betas[k], dtype=torch.float64, device=dev)
                b.requires_grad_(case["adjoint"])
                z = ex.log_z(Jx, b, x)
                put("logZR", z.detach())
                if case["adjoint"]:
                    db, dj = torch.autograd.grad(z.sum(), (b, Jx))
                    put("dbeta", db)
                    dJ += dj / B
            put("dJ", dJ)
        if op == "backward":
            l = logZR[k * B:(k + 1) * B] - logq[k * B:(k + 1) * B].double()
            wgt = -(l - l.mean()) / (betas[k] * B)
            grad = torch.zeros_like(theta)
            for x, wx in zip(s.split(16384), wgt.split(16384)):
                th = theta.clone().requires_grad_(True)
                grad += torch.autograd.grad((wx * _log_q(th, D, hidden, x)).sum(), th)[0]
            put("grad", grad)
        if op in ("moments", "observables"):
            l = logZR[k * B:(k + 1) * B] - logq[k * B:(k + 1) * B].double()
            p = torch.softmax(l, 0)
            mean, var, energy = [], [], []
            corr = torch.zeros_like(J)
            for x, px in zip(s.split(1024), p.split(1024)):
                Jx = J.clone().requires_grad_(op == "observables")
                b = torch.full((x.shape[0],), betas[k], dtype=torch.float64, device=dev)
                f = torch.zeros_like(b)
                if op == "observables":
                    b.requires_grad_(True)
                    z = ex.log_z(Jx, b, x)
                    db, = torch.autograd.grad(z.sum(), b, retain_graph=True)
                    energy.append(-db)
                    corr += torch.autograd.grad((px * z).sum(), Jx)[0]
                else:
                    f.requires_grad_(True)
                    z = ex.log_z(Jx, b, x, f)
                    d1, = torch.autograd.grad(z.sum(), f, create_graph=True)
                    d2, = torch.autograd.grad(d1.sum(), f)
                    mean.append(d1.detach() + x.sum(1))
                    var.append(d2)
            ess = 1.0 / (p * p).sum()
            if op == "observables":
                E = torch.cat(energy)
                put("averages", torch.stack([(p * E).sum(), E.mean(), ess]))
                put("corr", corr)
            else:
                mu, v = torch.cat(mean), torch.cat(var)
                m1, m2 = (p * mu).sum(), (p * (mu * mu + v)).sum()
                put("averages", torch.stack([m1, m2, betas[k] * (m2 - m1 * m1) / g.n, mu.mean(), (mu * mu + v).mean(),
                                             ess]))
                put("mean", mu)
                put("var", v)
    v = {name: torch.stack(x) if name == "averages" else torch.cat(x) for name, x in got.items()}
    if op == "sample":
        return {"spins": None, "logq": v["logq"], "logZR": v["logZR"]}
    if op == "log_prob":
        return {"logq": v["logq"]}
    if op == "contract":
        return _some({"logZR": v["logZR"], "dbeta": v.get("dbeta")})
    if op == "backward":
        return _some({"grad": v["grad"], "dbeta": v.get("dbeta"), "dJ": v.get("dJ") if case["adjoint"] else None})
    if op == "moments":
        return {"averages": v["averages"], "mean": v["mean"], "var": v["var"]}
    return {"averages": v["averages"], "corr": v["corr"]}
