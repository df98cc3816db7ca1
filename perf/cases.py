"""The work that a user of this library has it do, as cases that can be timed.

Every case goes through the public entry points of `paper_0903_3053_gb300`: batches of 2D Ising chains in both
storage layouts, batches of 4D SU(2) chains, uneven chains advanced together as a group, and the learned proposal's
log-probability, training step and sampler.  A pass of a Markov-chain case is a stretch of a run as a program
makes it: some sweeps with measurements, the records read back, and the configurations taken out into the
program's own device buffers (layout-free formats).  The chains go on from pass to pass.

`exact` restates the SU(2) heat-bath and the masked network in 64 bits with plain torch; the Ising results and
the sampler's spins are whole numbers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0903_3053_gb300 import mc

BETA_C = 0.4406868
BETAS_ISING = [0.30, 0.40, 0.4406868, 0.50, 0.60]
BETAS_SU2 = [1.5, 2.0, 2.3, 2.6]


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one small chain followed sweep by sweep: latency
        {"name": "ising_64_int8", "kind": "ising", "layout": "int8", "lx": 64, "ly": 64, "chains": 1, "sweeps": 100, "every": 1},
        # the 1024 x 512 lattice of the paper's Ising section, default layout, E and M after every sweep
        {"name": "ising_1024x512_int8", "kind": "ising", "layout": "int8", "lx": 1024, "ly": 512, "chains": 1, "sweeps": 50, "every": 1},
        # the local sweeps between two rounds of the learned proposal: many small int8 chains
        {"name": "ising_4096x64_int8", "kind": "ising", "layout": "int8", "lx": 64, "ly": 64, "chains": 4096, "sweeps": 10, "every": 10},
        # the README's run: four 4096^2 chains at the critical point, 32 spins per word, measured every sweep
        {"name": "ising_4x4096_msc", "kind": "ising", "layout": "msc", "lx": 4096, "ly": 4096, "chains": 4, "sweeps": 20, "every": 1},
        # the benchmark batch: L in {1024, 4096, 16384} x five couplings, 32 spins per word
        {"name": "ising_bench_msc", "kind": "ising", "layout": "msc", "lx": 0, "ly": 0, "chains": 15, "sweeps": 8, "every": 1},
        # small SU(2) lattices at the benchmark's four couplings, plaquette every sweep: latency
        {"name": "su2_8^4_x4", "kind": "su2", "l0": 8, "l1": 8, "l2": 8, "l3": 8, "chains": 4, "overrelax": 0, "sweeps": 20, "every": 1},
        # a lattice of the paper's Table 1 with overrelaxation, measured every five sweeps
        {"name": "su2_4x24^3_or1", "kind": "su2", "l0": 4, "l1": 24, "l2": 24, "l3": 24, "chains": 1, "overrelax": 1, "sweeps": 10, "every": 5},
        # the SU(2) benchmark: 32^4 at four couplings, heat-bath and plaquette every sweep
        {"name": "su2_32^4_x4", "kind": "su2", "l0": 32, "l1": 32, "l2": 32, "l3": 32, "chains": 4, "overrelax": 0, "sweeps": 2, "every": 1},
        # a parameter scan: uneven Ising and SU(2) chains advanced together
        {"name": "group_256_64", "kind": "group", "ising": 256, "su2": 64, "pick": 0, "sweeps": 10, "every": 1},
        # log q of as many configurations as the learned proposal has chains
        {"name": "van_logq_4096x64", "kind": "logq", "L": 64, "n": 4096, "depth": 6},
        # one maximum-likelihood training step
        {"name": "van_train_512x64", "kind": "train", "L": 64, "n": 512, "depth": 6},
        # proposals for every chain: the sequential sampler
        {"name": "van_sample_4096x64", "kind": "sample", "L": 64, "n": 4096, "depth": 6},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(rng, lo, hi):
    return max(lo, 2 * (_log_int(rng, lo, hi) // 2))


def draw(rng):
    kind = rng.choice(["int8", "int8", "msc", "msc", "su2", "su2", "su2", "group", "logq", "train", "sample"])
    if kind in ("int8", "msc"):
        if kind == "msc":
            lx, ly = 64 * _log_int(rng, 1, 128), _even(rng, 16, 8192)
        else:
            lx, ly = _even(rng, 8, 2048), _even(rng, 8, 2048)
        sites = lx * ly
        chains = _log_int(rng, 1, max(1, min(48, (1 << 26) // sites)))
        sweeps = max(4, min(100, int((1 << (30 if kind == "msc" else 28)) / (sites * chains))))
        return {"kind": "ising", "layout": kind, "lx": lx, "ly": ly, "chains": chains, "sweeps": sweeps,
                "every": rng.choice([1, 1, 2])}
    if kind == "su2":
        L = [_even(rng, 4, 24) for _ in range(4)]
        chains = rng.randint(1, 4)
        sweeps = max(2, min(20, int(4e7 / (4 * math.prod(L) * chains))))
        return {"kind": "su2", "l0": L[0], "l1": L[1], "l2": L[2], "l3": L[3], "chains": chains,
                "overrelax": rng.choice([0, 0, 1, 3]), "sweeps": sweeps, "every": rng.choice([1, 2])}
    if kind == "group":
        return {"kind": "group", "ising": _log_int(rng, 8, 256), "su2": _log_int(rng, 2, 64), "pick": rng.randint(1, 999),
                "sweeps": rng.randint(4, 10), "every": rng.choice([1, 2])}
    L = _even(rng, 6, 64)
    most = {"logq": 4096, "train": 512, "sample": 4096}[kind] * 64 * 64
    return {"kind": kind, "L": L, "n": _log_int(rng, 32, max(33, min(4096, most // (L * L)))), "depth": rng.choice([4, 5, 6, 6, 7])}


# ------------------------------------------------------------------ preparation
def _ising_chains(case, seed):
    if case["lx"] == 0:  # the benchmark batch
        return [mc.ising(L, b, seed=seed, chain_id=i) for i, (L, b) in
                enumerate((L, b) for L in (1024, 4096, 16384) for b in BETAS_ISING)]
    return [mc.ising((case["lx"], case["ly"]), BETA_C, seed=seed, chain_id=k) for k in range(case["chains"])]


def _records(case):
    return case["sweeps"] // case["every"] + 1


def _su2_dims(case):
    return case["l0"], case["l1"], case["l2"], case["l3"]


def _su2_start(case, seed):
    """Random links, one canonical float32 tensor [site][mu][4] per chain."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for _ in range(case["chains"]):
        q = torch.randn((math.prod(_su2_dims(case)), 4, 4), generator=g, device="cuda", dtype=torch.float64)
        out.append((q / q.norm(dim=-1, keepdim=True)).float())
    return out


def _group_chains(case, seed):
    """Extents and couplings of an uneven scan: the same lattices for every seed."""
    rng = np.random.default_rng(case["pick"])
    sizes = rng.choice([32, 64, 128, 256, 512, 1024], size=case["ising"])
    betas = rng.uniform(0.35, 0.55, size=case["ising"])
    i8 = [mc.ising(int(L), float(b), seed=seed + i, chain_id=i) for i, (L, b) in enumerate(zip(sizes, betas)) if L % 64]
    msc = [mc.ising(int(L), float(b), seed=seed + i, chain_id=i) for i, (L, b) in enumerate(zip(sizes, betas)) if L % 64 == 0]
    sizes = rng.choice([4, 6, 8, 12, 16], size=case["su2"])
    betas = rng.uniform(1.8, 2.6, size=case["su2"])
    s2 = [mc.su2(int(L), float(b), seed=seed + 1000 + i, chain_id=case["ising"] + i) for i, (L, b) in enumerate(zip(sizes, betas))]
    return i8, msc, s2


def _van_params(case, seed):
    """He-style random weights of the masked network and small biases: [(W[o][i][5][5], b[o]), ...] in float32."""
    rng = np.random.default_rng(seed)
    D, out = case["depth"], []
    for l in range(D):
        cin, cout = (1 if l == 0 else 32), (1 if l == D - 1 else 32)
        W = rng.normal(0.0, 0.7 * math.sqrt(2.0 / (cin * (12 if l == 0 else 13))), size=(cout, cin, 5, 5))
        out.append((W.astype(np.float32), rng.normal(0.0, 0.05, size=cout).astype(np.float32)))
    return out


def _van_spins(case, seed):
    """Configurations with domains, as at the critical coupling: the sign of smoothed noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    L, n = case["L"], case["n"]
    x = torch.randn((n, 1, L, L), generator=g, device="cuda")
    r = min(2, L // 4)
    x = torch.nn.functional.avg_pool2d(torch.nn.functional.pad(x, (r, r, r, r), mode="circular"), 2 * r + 1, stride=1)
    return torch.where(x[:, 0] >= 0, 1, -1).to(torch.int8).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ising":
        chains = _ising_chains(case, seed)
        layout = mc.MC_LAYOUT_INT8 if case["layout"] == "int8" else mc.MC_LAYOUT_MSC32
        b = mc.Batch(chains, layout=layout, series_capacity=_records(case))
        outs = None
        if len(chains) <= 48:
            if layout == mc.MC_LAYOUT_INT8:
                outs = [torch.empty((c.L[1], c.L[0]), dtype=torch.int8, device="cuda") for c in chains]
            else:
                outs = [torch.empty((c.L[1], c.L[0] // 32), dtype=torch.int32, device="cuda") for c in chains]
        return {"case": case, "batch": b, "outs": outs}
    if kind == "su2":
        links = _su2_start(case, seed)
        b = mc.Batch([mc.su2(_su2_dims(case), BETAS_SU2[(k + 2) % 4] if case["chains"] < 4 else BETAS_SU2[k], seed=seed, chain_id=k)
                      for k in range(case["chains"])], series_capacity=_records(case))
        b.set_overrelax(case["overrelax"])
        for k, q in enumerate(links):
            b.set_config_device(k, q)
        return {"case": case, "batch": b, "outs": links}
    if kind == "group":
        i8, msc, s2 = _group_chains(case, seed)
        cap = _records(case)
        batches = []
        if i8:
            batches.append(mc.Batch(i8, layout=mc.MC_LAYOUT_INT8, series_capacity=cap))
        if msc:
            batches.append(mc.Batch(msc, layout=mc.MC_LAYOUT_MSC32, series_capacity=cap))
        batches.append(mc.Batch(s2, series_capacity=cap))
        g = mc.Group(batches)
        g.configure(8, 256, -1.0)  # the shape that the autotuner picks for such scans
        last = []  # the largest chain of each batch, whose configuration the program takes out
        for b in batches:
            k = max(range(len(b.chains)), key=lambda j: math.prod(b.chains[j].L))
            c = b.chains[k]
            if b.kind == mc.MC_KIND_SU2:
                out = torch.empty((math.prod(c.L), 4, 4), dtype=torch.float32, device="cuda")
            else:
                out = torch.empty((c.L[1], c.L[0]), dtype=torch.int8, device="cuda")
            last.append((b, k, out))
        return {"case": case, "group": g, "batches": batches, "last": last}
    net = mc.VAN(case["L"], case["n"], depth=case["depth"], seed=seed)
    net.set_params(mc.van_pack(_van_params(case, seed)))
    return {"case": case, "net": net, "spins": None if kind == "sample" else _van_spins(case, seed)}


# ------------------------------------------------------------------ one pass
def _series(b):
    r = b.read_series()
    if b.kind == mc.MC_KIND_SU2:
        return {"sweep": r["sweep"], "P": r["P"], "Ps": r["Ps"], "Pt": r["Pt"]}
    return {"sweep": r["sweep"], "E": r["E"], "M": r["M"]}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ising":
        b = state["batch"]
        b.sweep(case["sweeps"], case["every"])
        if state["outs"] is None:
            spins = mc.ising_gather(b)
        else:
            spins = state["outs"]
            for k, t in enumerate(spins):
                b.get_config_device(k, t, mc.MC_FMT_INT8 if case["layout"] == "int8" else mc.MC_FMT_BITS)
        return {"series": _series(b), "spins": spins}
    if kind == "su2":
        b = state["batch"]
        b.sweep(case["sweeps"], case["every"])
        for k, t in enumerate(state["outs"]):
            b.get_config_device(k, t)
        return {"series": _series(b), "links": state["outs"]}
    if kind == "group":
        state["group"].sweep(case["sweeps"], case["every"])
        out = {"series": [_series(b) for b in state["batches"]], "last": []}
        for b, k, t in state["last"]:
            b.get_config_device(k, t)
            out["last"].append(t)
        return out
    net = state["net"]
    if kind == "logq":
        return {"logq": net.log_prob(state["spins"])}
    if kind == "train":
        loss = net.train_step(state["spins"], lr=1e-3, apply=True)
        _, grads = net.get_params(grads=True)
        return {"loss": loss, "grads": grads}
    spins, logq = net.sample(case["n"], round=1)
    return {"spins": spins, "logq": logq}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Lattices, weights, inputs and results once each; per site and sweep the random numbers and the update."""
    kind = case["kind"]
    if kind == "ising":
        if case["lx"] == 0:
            sites = 5.0 * sum(L * L for L in (1024, 4096, 16384))
        else:
            sites = float(case["lx"]) * case["ly"] * case["chains"]
        per = 1.0 if case["layout"] == "int8" else 0.125
        return {"bytes": 3 * sites * per, "flops": 18.0 * sites * case["sweeps"]}
    if kind == "su2":
        links = 4.0 * math.prod(_su2_dims(case)) * case["chains"]
        return {"bytes": 3 * 16 * links, "flops": links * case["sweeps"] * (430.0 + 330.0 * case["overrelax"])}
    if kind == "group":
        rng = np.random.default_rng(case["pick"])
        sizes = rng.choice([32, 64, 128, 256, 512, 1024], size=case["ising"]).astype(float)
        rng.uniform(0.35, 0.55, size=case["ising"])
        su2 = 4.0 * float((rng.choice([4, 6, 8, 12, 16], size=case["su2"]).astype(float) ** 4).sum())
        sites = float((sizes ** 2).sum())
        return {"bytes": sites / 4 + 32 * su2, "flops": case["sweeps"] * (18.0 * sites + 430.0 * su2)}
    L, n, D = case["L"], case["n"], case["depth"]
    pos = float(n) * L * L
    macs = pos * (12 * 32 + (D - 2) * 13 * 32 * 32 + 13 * 32)
    if kind == "train":
        return {"bytes": pos + 8.0 * mc.van_param_count(D), "flops": 6 * macs}
    return {"bytes": pos + 8.0 * n + 2.0 * mc.van_param_count(D), "flops": 2 * macs}


# ------------------------------------------------------------------ 64-bit restatements
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # the low 64 bits are right under wrap-around
        c0, c1, c2, c3 = ((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _uniform(r):
    return ((r >> 8) + 1).double() * 2.0 ** -24


def _qmul(a, b):
    a0, a1, a2, a3 = a.unbind(-1)
    b0, b1, b2, b3 = b.unbind(-1)
    return torch.stack((a0 * b0 - a1 * b1 - a2 * b2 - a3 * b3, a0 * b1 + b0 * a1 - a2 * b3 + a3 * b2,
                        a0 * b2 + b0 * a2 - a3 * b1 + a1 * b3, a0 * b3 + b0 * a3 - a1 * b2 + a2 * b1), -1)


def _qdag(a):
    return torch.stack((a[..., 0], -a[..., 1], -a[..., 2], -a[..., 3]), -1)


class _Lattice:
    """One SU(2) chain in float64: U[mu] of shape (L0, L3, L2, L1, 4)."""

    AXIS = {0: 0, 3: 1, 2: 2, 1: 3}

    def __init__(self, links, dims, beta, seed, chain):
        L0, L1, L2, L3 = dims
        self.dims, self.beta, self.seed, self.chain = dims, beta, seed, chain
        q = links.double().reshape(L0, L3, L2, L1, 4, 4)
        self.U = [q[..., mu, :].clone() for mu in range(4)]
        s = torch.arange(L0 * L1 * L2 * L3, device=links.device)
        x1, x2, x3, x0 = s % L1, s // L1 % L2, s // (L1 * L2) % L3, s // (L1 * L2 * L3)
        par = (x0 + x1 + x2 + x3) & 1
        self.sites = [torch.nonzero(par == p)[:, 0] for p in (0, 1)]

    def at(self, U, mu, d):
        return torch.roll(U, -d, dims=self.AXIS[mu])

    def staple(self, mu):
        W = torch.zeros_like(self.U[0])
        for nu in range(4):
            if nu != mu:
                Un, Um = self.U[nu], self.U[mu]
                W = W + _qmul(_qmul(Un, self.at(Um, nu, 1)), _qdag(self.at(Un, mu, 1)))
                W = W + _qmul(_qmul(_qdag(self.at(Un, nu, -1)), self.at(Um, nu, -1)), self.at(self.at(Un, mu, 1), nu, -1))
        return W

    def update(self, p, mu, sweep, reflect):
        idx = self.sites[p]
        W = self.staple(mu).reshape(-1, 4)[idx]
        k = W.norm(dim=-1)
        V = torch.where(k[:, None] > 0, W / k.clamp_min(1e-300)[:, None], torch.tensor([1.0, 0, 0, 0], dtype=W.dtype, device=W.device))
        flat = self.U[mu].reshape(-1, 4)
        old = flat[idx]
        if reflect:
            new = _qmul(_qmul(V, _qdag(old)), V)
            new = torch.where(k[:, None] > 0, new / new.norm(dim=-1, keepdim=True), old)
        else:
            alpha, e = self.beta * k, idx >> 1
            one = torch.ones_like(e)
            sel = (p << 12) | (mu << 8)
            a0, open_ = torch.zeros_like(alpha), torch.arange(e.numel(), device=e.device)
            for t in range(72):
                if open_.numel() == 0:
                    break
                al, eo = alpha[open_], e[open_]
                r = _philox(eo, one[open_] * sweep, one[open_] * (0x12000000 | sel | t), one[open_] * self.chain, self.seed)
                u = [_uniform(v) for v in r]
                if t < 8:
                    lam = -(torch.log(u[0]) + torch.cos(2 * math.pi * u[1]) ** 2 * torch.log(u[2])) / (2 * al)
                    c, ok = 1 - 2 * lam, (u[3] ** 2 <= 1 - lam) & (al > 0)
                else:
                    c = torch.where(al > 0, 1 + torch.log1p((1 - u[0]) * torch.expm1(-2 * al)) / al, 2 * u[0] - 1)
                    ok = u[1] ** 2 <= 1 - c * c
                a0[open_[ok]] = c[ok]
                open_ = open_[~ok]
            r = _philox(e, one * sweep, one * (0x13000000 | sel), one * self.chain, self.seed)
            ct, phi = 2 * _uniform(r[0]) - 1, 2 * math.pi * _uniform(r[1])
            st, rad = (1 - ct * ct).clamp_min(0).sqrt(), (1 - a0 * a0).clamp_min(0).sqrt()
            X = torch.stack((a0, rad * st * torch.cos(phi), rad * st * torch.sin(phi), rad * ct), -1)
            new = _qmul(X, V)
            new = new / new.norm(dim=-1, keepdim=True)
            new[open_] = old[open_]
        flat = flat.clone()
        flat[idx] = new
        self.U[mu] = flat.reshape(self.U[mu].shape)

    def sweep(self, t, n_or):
        for r in range(1 + n_or):
            for p in (1, 0):
                for mu in range(4):
                    self.update(p, mu, t, r > 0)

    def plaquettes(self):
        s = {False: 0.0, True: 0.0}
        for mu in range(4):
            for nu in range(mu + 1, 4):
                A = _qmul(self.U[mu], self.at(self.U[nu], mu, 1))
                B = _qmul(self.U[nu], self.at(self.U[mu], nu, 1))
                s[mu == 0] += float((A * B).sum())
        n = math.prod(self.dims)
        return (s[False] + s[True]) / (6 * n), s[False] / (3 * n), s[True] / (3 * n)

    def canonical(self):
        return torch.stack(self.U, -2).reshape(-1, 4, 4)


_TAPS = [(dy, dx) for dy in (-2, -1, 0) for dx in range(-2, 3) if dy < 0 or dx <= 0]


def _conv(x, W, b, own):
    """Masked 5 x 5 convolution of x [n][L][L][c] with zero padding; `own`: whether the tap at the position itself counts."""
    n, L = x.shape[0], x.shape[1]
    xp = torch.nn.functional.pad(x, (0, 0, 2, 2, 2, 0))
    out = b.expand(n, L, L, b.numel())
    for dy, dx in _TAPS:
        if own or (dy, dx) != (0, 0):
            out = out + xp[:, 2 + dy:2 + dy + L, 2 + dx:2 + dx + L] @ W[:, :, dy + 2, dx + 2].t()
    return out


def _van_logq(spins, params):
    h = spins.double()[..., None]
    s = spins.double()
    for l, (W, b) in enumerate(params):
        h = _conv(h, W, b, l > 0)
        if l + 1 < len(params):
            h = torch.relu(h)
    return torch.nn.functional.logsigmoid(s * h[..., 0]).sum(dim=(1, 2))


def exact(case, seed):
    kind = case["kind"]
    if kind == "su2":
        # a longer chain amplifies the rounding of its first sweeps, and one accept decision that 64 bits take otherwise
        # changes all that follows: two sweeps are what an independent evaluation can follow
        if case["sweeps"] * (1 + case["overrelax"]) > 2:
            return None
        series, links = [], []
        for k, q in enumerate(_su2_start(case, seed)):
            beta = BETAS_SU2[(k + 2) % 4] if case["chains"] < 4 else BETAS_SU2[k]
            lat = _Lattice(q, _su2_dims(case), beta, seed, k)
            rec = []
            for t in range(case["sweeps"]):
                lat.sweep(t, case["overrelax"])
                if (t + 1) % case["every"] == 0:
                    rec.append(lat.plaquettes())
            series.append(rec)
            links.append(lat.canonical())
        s = np.array(series, dtype=np.float64)
        return {"series": {"sweep": None, "P": s[..., 0], "Ps": s[..., 1], "Pt": s[..., 2]}, "links": links}
    if kind not in ("logq", "train"):
        return None
    dev = torch.device("cuda")
    params = [(torch.tensor(W, dtype=torch.float64, device=dev), torch.tensor(b, dtype=torch.float64, device=dev))
              for W, b in _van_params(case, seed)]
    spins = _van_spins(case, seed)
    chunk = max(1, 131072 // case["L"] ** 2)
    if kind == "logq":
        with torch.no_grad():
            return {"logq": torch.cat([_van_logq(s, params) for s in spins.split(chunk)])}
    for W, b in params:
        W.requires_grad_()
        b.requires_grad_()
    loss = 0.0
    for s in spins.split(chunk):
        part = -_van_logq(s, params).sum() / case["n"]
        part.backward()
        loss += float(part.detach())
    grads = torch.cat([torch.cat((W.grad.reshape(-1), b.grad.reshape(-1))) for W, b in params])
    return {"loss": loss, "grads": grads.cpu().numpy()}
