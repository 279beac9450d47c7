"""Cases that measure this package through its public entry points.

Each case is one call, or the short sequence of calls, that a program built on
the package repeats: the pool step of an ADAPT iteration (state, pool gradient,
energy), the energy with its parameter gradient that drives the VQE
optimisation, a state with its energy read back, the screened pool step, a
batch of small instances, and the screening network's inference and gradient.
Sizes are those of the package's own workloads (12/4, 28/8, 52/12, the uneven
batch, the pool of 301,600 operators) and the 46 spin-orbitals of the
cc-pVDZ molecules, from 29 determinants to one million.

``exact`` restates the quantities in 64 bits with plain torch and numpy: gates
as gathers on a sorted list of bitstrings, sigma by enumerating every
Slater-Condon pair, the parameter gradient by torch's autograd.
"""
from __future__ import annotations

import math

import numpy as np
import torch

PAIRS_EXACT = dict(pool_step=4e8, state=1e9, vqe_grad=4e8)  # connected pairs up to which exact() restates a state
GATE_WORK_EXACT = 3e7    # gates x determinants up to which exact() restates the gates


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def listed():
    return [
        # smallest call: a test-sized molecule without truncation, all launches and latency
        dict(name="pool_step_12so_4e", kind="pool_step", n_so=12, n_e=4, gates=10, n_keep=0, eps=0.0),
        # ordinary ADAPT iteration of a mid-sized molecule; the size bound does not bite
        dict(name="pool_step_28so_8e", kind="pool_step", n_so=28, n_e=8, gates=60, n_keep=100_000, eps=0.0),
        # a cc-pVDZ molecule at a ragged determinant budget
        dict(name="pool_step_46so_10e", kind="pool_step", n_so=46, n_e=10, gates=120, n_keep=33_333, eps=0.0),
        # the largest ADAPT iteration: 52 spin-orbitals, 12 electrons, 200 gates, one million determinants
        dict(name="pool_step_52so_12e", kind="pool_step", n_so=52, n_e=12, gates=200, n_keep=1_000_000, eps=0.0),
        # the optimiser's call inside ADAPT: few gates, small budget, made hundreds of times a run
        dict(name="vqe_grad_52so_adapt", kind="vqe_grad", n_so=52, n_e=12, gates=15, n_keep=10_000, eps=0.0, ckpt=20),
        # VQE of a mid-sized molecule with a fixed ansatz
        dict(name="vqe_grad_28so_8e", kind="vqe_grad", n_so=28, n_e=8, gates=60, n_keep=100_000, eps=0.0, ckpt=20),
        # VQE at the largest state: 200 parameters through checkpoints
        dict(name="vqe_grad_52so_12e", kind="vqe_grad", n_so=52, n_e=12, gates=200, n_keep=1_000_000, eps=0.0, ckpt=20),
        # a state, its energy, and the determinants read back for analysis; magnitude criterion on
        dict(name="state_40so_10e", kind="state", n_so=40, n_e=10, gates=150, n_keep=100_000, eps=1e-9),
        # the pool step with the learned screen: features, network, top 5 %, exact gradients of those
        dict(name="screened_52so_12e", kind="screened", n_so=52, n_e=12, gates=120, n_keep=50_000, eps=0.0, frac=0.05),
        # many small independent systems in one launch, every result read back
        dict(name="batch_uneven_12", kind="batch", instances=12, n_so_max=40, keep_max=100_000),
        # the screening network over the whole 52-orbital pool
        dict(name="net_predict_301600", kind="net_predict", rows=301_600, d_in=32, width=256),
        # one minibatch of the network's training
        dict(name="net_grad_8192", kind="net_grad", rows=8_192, d_in=32, width=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pool_step", "pool_step", "pool_step", "vqe_grad", "vqe_grad", "vqe_grad", "state",
                       "screened", "batch", "net_predict", "net_grad"])
    if kind in ("net_predict", "net_grad"):
        return dict(kind=kind, rows=_log_int(rng, 1_000, 301_600 if kind == "net_predict" else 65_536),
                    d_in=rng.choice([32, 32, 64]), width=rng.choice([64, 128, 160, 256, 256]))
    if kind == "batch":
        return dict(kind=kind, instances=rng.randint(4, 16), n_so_max=2 * rng.randint(12, 20),
                    keep_max=_log_int(rng, 3_000, 100_000))
    if kind == "state":  # large enough that the size bound decides how many determinants come back
        return dict(kind=kind, n_so=2 * rng.randint(14, 26), n_e=2 * rng.randint(4, 6), gates=_log_int(rng, 100, 200),
                    n_keep=_log_int(rng, 1_000, 10_000), eps=rng.choice([0.0, 1e-9]))
    n_so = 2 * rng.randint(6, 26)
    n_e = 2 * rng.randint(2, min(6, n_so // 4))
    case = dict(kind=kind, n_so=n_so, n_e=n_e, gates=_log_int(rng, 10, 200), n_keep=_log_int(rng, 1_000, 1_000_000),
                eps=rng.choice([0.0, 0.0, 0.0, 1e-8]))
    if kind == "vqe_grad":
        case["ckpt"] = rng.choice([10, 20, 20, 20, 33])
    if kind == "screened":
        case["frac"] = rng.choice([0.02, 0.05, 0.1])
    return case


# --------------------------------------------------------------------------
# inputs, from the seed alone
# --------------------------------------------------------------------------
def _integrals(n_so, rng):
    """Spin-orbital h[p,q] and <pq||rs> (interleaved spin): sorted orbital energies, small
    couplings, Coulomb integrals that decay with the orbitals' distance."""
    m = n_so // 2
    h = rng.normal(0.0, 0.05, size=(m, m))
    h = np.tril(h, -1) + np.tril(h, -1).T
    h[np.arange(m), np.arange(m)] = np.sort(rng.uniform(-2.0, 1.0, size=m))
    p, q = np.tril_indices(m)
    x = np.exp(-np.abs(p - q)[:, None] - np.abs(p - q)[None, :]) * rng.uniform(0.0, 0.5, size=(len(p), len(p)))
    x = np.tril(x) + np.tril(x, -1).T
    pack = np.zeros((m, m), np.int64)
    pack[p, q] = pack[q, p] = np.arange(len(p))
    eri = x[pack.reshape(-1)][:, pack.reshape(-1)].reshape(m, m, m, m)   # (pq|rs)
    phys = eri.transpose(0, 2, 1, 3)                                       # <pr|qs> = (pq|rs)
    g = np.zeros((n_so,) * 4)
    for s in (0, 1):
        for t in (0, 1):
            g[s::2, t::2, s::2, t::2] += phys
            g[s::2, t::2, t::2, s::2] -= phys.transpose(0, 1, 3, 2)
    hso = np.zeros((n_so, n_so))
    hso[0::2, 0::2] = hso[1::2, 1::2] = h
    return hso, g


def _ansatz(n_so, n_e, gates, rng):
    """Occupied-to-virtual singles and doubles drawn without replacement, angles N(0, 0.05)."""
    occ, vir = np.arange(n_e), np.arange(n_e, n_so)
    i, a = (v.reshape(-1) for v in np.meshgrid(occ, vir, indexing="ij"))
    ok = i % 2 == a % 2
    z = np.zeros(int(ok.sum()), np.int64)
    single = np.stack([z + 1, i[ok], a[ok], z, z], 1)
    oi, oj = np.triu_indices(n_e, 1)
    va, vb = np.triu_indices(n_so - n_e, 1)
    x, y = (v.reshape(-1) for v in np.meshgrid(np.arange(len(oi)), np.arange(len(va)), indexing="ij"))
    i, j, a, b = oi[x], oj[x], va[y] + n_e, vb[y] + n_e
    ok = i % 2 + j % 2 == a % 2 + b % 2
    z = np.zeros(int(ok.sum()), np.int64)
    pool = np.concatenate([single, np.stack([z + 2, i[ok], j[ok], a[ok], b[ok]], 1)]).astype(np.uint8)
    sel = rng.choice(len(pool), size=min(gates, len(pool)), replace=False)
    return np.ascontiguousarray(pool[sel]), rng.normal(0.0, 0.05, size=len(sel))


def _system(case, seed):
    rng = np.random.default_rng([seed, case["n_so"], case["n_e"]])
    h, g = _integrals(case["n_so"], rng)
    ops, theta = _ansatz(case["n_so"], case["n_e"], case["gates"], rng)
    return h, g, ops, theta


def _batch_specs(case):
    """The instances' sizes, by the case alone."""
    rng = np.random.default_rng([case["instances"], case["n_so_max"], case["keep_max"]])
    out = []
    for _ in range(case["instances"]):
        n_so = 2 * int(rng.integers(8, case["n_so_max"] // 2 + 1))
        n_e = min(2 * int(rng.integers(2, 7)), n_so - 2)
        out.append(dict(n_so=n_so, n_e=n_e, gates=int(rng.integers(20, 151)), eps=0.0,
                        n_keep=int(round(10 ** rng.uniform(3.0, math.log10(case["keep_max"]))))))
    return out


def _network(case, seed):
    """Parameters of a screening network that leans on its strongest predictor, as a trained one does."""
    d, w = case["d_in"], case["width"]
    rng = np.random.default_rng([seed, d, w])
    W1, W2 = rng.normal(size=(w, d)) * math.sqrt(2.0 / d), rng.normal(size=(w, w)) * math.sqrt(2.0 / w)
    w3 = rng.normal(size=w) * math.sqrt(1.0 / w)
    b1, b2 = rng.normal(size=w) * 0.1, rng.normal(size=w) * 0.1
    W1[0] = 0.0
    W1[0, 29], b1[0] = 1.0, 3.0
    W2[0] = 0.0
    W2[0, 0], w3[0] = 1.0, 4.0
    return [np.asarray(v, np.float32) for v in (W1, b1, W2, b2, w3, rng.normal(size=1) * 0.1)]


def _net_rows(case, seed):
    """Feature rows in the range of the pool's features (BF16 bits) and log10 |g| targets."""
    gen = torch.Generator().manual_seed(seed)
    x = (torch.randn(case["rows"], case["d_in"], generator=gen) * 0.6).to(torch.bfloat16)
    t = -10.0 * torch.rand(case["rows"], generator=gen)
    return x, t


# --------------------------------------------------------------------------
# what a program has in hand, and one pass
# --------------------------------------------------------------------------
def prepare(case, seed):
    from paper_2411_07920_gb300 import swcs
    kind = case["kind"]
    if kind in ("net_predict", "net_grad"):
        net = swcs.Mlp(case["d_in"], case["width"])
        net.set_params(np.concatenate([v.reshape(-1) for v in _network(case, seed)]))
        x, t = _net_rows(case, seed)
        return dict(kind=kind, net=net, x=x.view(torch.int16).cuda(), t=t.cuda(),
                    y=torch.empty(case["rows"], device="cuda"), grad=torch.empty(net.n_params, device="cuda"),
                    loss=torch.empty(1, dtype=torch.float64, device="cuda"))
    if kind == "batch":
        b = swcs.Batch()
        for i, spec in enumerate(_batch_specs(case)):
            h, g, ops, theta = _system(spec, seed + 1000 * (i + 1))
            b.add(h, g, spec["n_so"], spec["n_e"], ops, theta, spec["n_keep"])
        b.build(autotune=False)
        return dict(kind=kind, batch=b, instances=case["instances"])
    h, g, ops, theta = _system(case, seed)
    ctx = swcs.Context()
    ctx.load_hamiltonian(h, g, case["n_so"], case["n_e"])
    if case["eps"]:
        ctx.set_truncation_threshold(case["eps"])
    state = dict(kind=kind, ctx=ctx, ops=ops, theta=theta, n_keep=case["n_keep"], ckpt=case.get("ckpt", 20))
    if kind == "screened":
        net = swcs.Mlp(32, 256)
        net.set_params(np.concatenate([v.reshape(-1) for v in _network(dict(d_in=32, width=256), seed)]))
        pool = ctx.pool_size()
        state.update(net=net, frac=case["frac"], sub=torch.empty(pool, dtype=torch.int64, device="cuda"),
                     g=torch.zeros(pool, dtype=torch.float64, device="cuda"))
    return state


def run(s):
    kind = s["kind"]
    if kind == "net_predict":
        s["net"].predict_dev(s["x"], s["y"])
        return s["y"]
    if kind == "net_grad":
        s["net"].grad_dev(s["x"], s["t"], s["grad"], s["loss"])
        return dict(grad=s["grad"], loss=s["loss"])
    if kind == "batch":
        s["batch"].run()
        return [s["batch"].results(i) for i in range(s["instances"])]
    ctx = s["ctx"]
    if kind == "vqe_grad":
        e, d = ctx.energy_grad(s["ops"], s["theta"], s["n_keep"], s["ckpt"])
        return dict(e=e, d=d)
    ctx.apply_ansatz(s["ops"], s["theta"], s["n_keep"])
    if kind == "pool_step":
        g = ctx.pool_gradients()
        e, n2 = ctx.sweep_energy()
        return dict(g=g, e=e, n2=n2, dets=ctx.state_size())
    if kind == "state":
        e, n2 = ctx.energy()
        keys, amps = ctx.get_state()
        return dict(e=e, n2=n2, keys=keys.view(np.int64), amps=amps)
    k = ctx.pool_screen_dev(s["net"], s["frac"], s["sub"])
    ctx.pool_gradients_dev(s["g"], s["sub"][:k])
    return dict(g=s["g"], selected=k)


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def _shape(case):
    """(determinants at most, connections of one, pool operators)."""
    m, no = case["n_so"] // 2, case["n_e"] // 2
    nv = m - no
    dim = math.comb(m, no) ** 2
    dets = min(dim, 2 ** min(case["gates"], 60), case["n_keep"] or dim)
    conn = 2 * no * nv + 2 * math.comb(no, 2) * math.comb(nv, 2) + (no * nv) ** 2
    return dets, conn, 2 * math.comb(m, 2) + 6 * math.comb(m, 4) + (m * (m - 1)) ** 2 // 2


def work(case):
    kind = case["kind"]
    if kind in ("net_predict", "net_grad"):
        n, d, w = case["rows"], case["d_in"], case["width"]
        params = w * d + w * w + 3 * w + 1
        flops = 2.0 * n * (d * w + w * w + w)
        if kind == "net_predict":
            return dict(bytes=2.0 * n * d + 4.0 * n + 2.0 * params, flops=flops)
        return dict(bytes=2.0 * n * d + 4.0 * n + 6.0 * params, flops=3.0 * flops - 2.0 * n * d * w)
    if kind == "batch":
        each = [work(dict(spec, kind="pool_step")) for spec in _batch_specs(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    dets, conn, pool = _shape(case)
    n = case["n_so"]
    ham = 8.0 * (n * n + (n * (n - 1) // 2) ** 2)
    gate_flops = 6.0 * dets * case["gates"] / 4  # an operator acts on a fraction of the determinants
    if kind == "pool_step":  # sigma on every connected determinant, then the contraction with each pair
        return dict(bytes=ham + 16.0 * dets + 8.0 * pool, flops=gate_flops + 4.0 * dets * (conn + 1))
    if kind == "screened":
        return dict(bytes=ham + 16.0 * dets + 8.0 * pool, flops=gate_flops + 2.0 * dets * (conn + 1) * (1 + case["frac"]))
    energy_flops = 2.0 * dets * min(conn + 1, dets)
    if kind == "state":
        return dict(bytes=ham + 48.0 * dets, flops=gate_flops + energy_flops)
    return dict(bytes=ham + 16.0 * dets + 29.0 * case["gates"], flops=4 * gate_flops + energy_flops)


# --------------------------------------------------------------------------
# the same quantities in 64 bits
# --------------------------------------------------------------------------
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _parity(x):
    for s in (32, 16, 8, 4, 2, 1):
        x = x ^ (x >> s)
    return x & 1


def _below(d, p):
    return _parity(d & ((1 << p) - 1)) if isinstance(p, int) else _parity(d & (torch.bitwise_left_shift(torch.ones_like(p), p) - 1))


def _bit(p):
    return torch.bitwise_left_shift(torch.ones_like(p), p)


def _phase1(d, a, c):
    return _below(d, a) ^ _below(d ^ _bit(a), c)


def _phase2(d, a0, a1, c2, c3):
    """Sign bit of a+_c2 a+_c3 a_a1 a_a0 on d."""
    par = _below(d, a0)
    x = d ^ _bit(a0)
    par = par ^ _below(x, a1)
    x = x ^ _bit(a1)
    par = par ^ _below(x, c3)
    return par ^ _below(x | _bit(c3), c2)


def _gates(case, ops, theta, keep_zeros):
    """The truncated ansatz: bitstrings ascending, amplitudes (differentiable in theta)."""
    dev = _dev()
    keys = torch.tensor([(1 << case["n_e"]) - 1], dtype=torch.int64, device=dev)
    amps = torch.ones(1, dtype=torch.float64, device=dev)
    for k, op in enumerate(ops.tolist()):
        co, si = torch.cos(theta[k]), torch.sin(theta[k])
        lo, hi = (op[1:2], op[2:3]) if op[0] == 1 else (op[1:3], op[3:5])
        ma, mc = sum(1 << p for p in lo), sum(1 << p for p in hi)
        up, dn = (keys & (ma | mc)) == ma, (keys & (ma | mc)) == mc
        act = up | dn
        partner = torch.where(act, keys ^ (ma | mc), keys)
        new = torch.unique(torch.cat([keys, partner]))
        at = torch.searchsorted(new, keys)
        a0 = torch.zeros(len(new), dtype=torch.float64, device=dev).index_put((at,), amps)
        up, dn = (new & (ma | mc)) == ma, (new & (ma | mc)) == mc
        low = torch.where(up, new, new ^ (ma | mc))  # the lower determinant carries the phase of tau
        one = torch.ones_like(low)
        if op[0] == 1:
            sg = _phase1(low, one * op[1], one * op[2])
        else:
            sg = _phase2(low, one * op[1], one * op[2], one * op[3], one * op[4])
        sg = 1.0 - 2.0 * sg.to(torch.float64)
        act = up | dn
        other = torch.searchsorted(new, torch.where(act, new ^ (ma | mc), new))
        rot = torch.where(up, a0 * co - sg * (a0[other] * si), a0 * co + sg * (a0[other] * si))
        a1 = torch.where(act, rot, a0)
        mag = a1.detach().abs()
        live = mag >= (case["eps"] or 0.0 if keep_zeros else case["eps"] or 5e-324)  # a projector keeps exact zeros
        idx = torch.nonzero(live).reshape(-1)
        if case["n_keep"] and len(idx) > case["n_keep"]:
            order = torch.sort(-mag[idx], stable=True).indices[:case["n_keep"]]  # ties: smaller bitstring first
            idx = idx[torch.sort(order).values]
        keys, amps = new[idx], a1[idx]
    return keys, amps


class _Pairs:
    """Every connected pair (D, E) of a list of determinants, block by block."""

    def __init__(self, case, h, g):
        dev = _dev()
        n = self.n = case["n_so"]
        self.no, self.m = case["n_e"] // 2, n // 2
        self.h = torch.from_numpy(h).to(dev)
        self.g = torch.from_numpy(g).to(dev).reshape(-1)
        self.gdiag = torch.einsum("ijij->ij", torch.from_numpy(g).to(dev))
        self.gs = torch.einsum("rkpk->prk", torch.from_numpy(g).to(dev)).contiguous()  # <rk||pk>
        p, q = np.triu_indices(n, 1)
        same = (p % 2) == (q % 2)
        one = np.full((n, n), -1, np.int64)
        one[p[same], q[same]] = np.arange(int(same.sum()))
        spin = p % 2 + q % 2
        ok = spin[:, None] == spin[None, :]
        ok &= (p[:, None] != p[None, :]) & (p[:, None] != q[None, :]) & (q[:, None] != p[None, :]) & (q[:, None] != q[None, :])
        ok &= np.arange(len(p))[:, None] < np.arange(len(p))[None, :]
        two = np.where(ok.reshape(-1), np.cumsum(ok.reshape(-1)) - 1 + int(same.sum()), -1)
        self.pool = int(same.sum()) + int(ok.sum())
        self.one = torch.from_numpy(one).to(dev).reshape(-1)
        self.two = torch.from_numpy(two).to(dev)
        self.np = len(p)

    def _pair(self, p, q):
        return p * self.n - torch.div(p * (p + 1), 2, rounding_mode="floor") + q - p - 1

    def blocks(self, keys, diagonal, pool):
        """Yields (rows of keys, E, <E|H|D>, operator, sign of its contribution), flattened: E = D where
        diagonal is set, then every excitation; operator and sign only where pool is set."""
        dev, n, no, m = keys.device, self.n, self.no, self.m
        nv = m - no
        step = max(1, int(2e7) // max(1, (no * nv) ** 2))
        for r0 in range(0, len(keys), step):
            d = keys[r0:r0 + step]
            row = torch.arange(r0, r0 + len(d), device=dev)
            bits = (d[:, None] >> torch.arange(n, device=dev)) & 1
            order = torch.sort(1 - bits, dim=1, stable=True).indices
            occ = order[:, :2 * no]
            A, B = (torch.sort(1 - bits[:, s::2], dim=1, stable=True).indices * 2 + s for s in (0, 1))
            if diagonal:
                e = self.h[occ, occ].sum(1) + 0.5 * self.gdiag[occ[:, :, None], occ[:, None, :]].sum((1, 2))
                yield row, d, e, None, None
            for X in (A, B):
                p = X[:, :no, None].expand(-1, no, nv).reshape(len(d), -1)
                r = X[:, None, no:].expand(-1, no, nv).reshape(len(d), -1)
                dd = d[:, None].expand_as(p)
                f = self.h[r, p] + self.gs[p.unsqueeze(-1), r.unsqueeze(-1), occ[:, None, :]].sum(-1)
                sg = 1.0 - 2.0 * _phase1(dd, p, r).to(torch.float64)
                k = self.one[torch.minimum(p, r) * n + torch.maximum(p, r)] if pool else None
                yield (row[:, None].expand_as(p).reshape(-1), (dd ^ _bit(p) ^ _bit(r)).reshape(-1), (f * sg).reshape(-1),
                       k.reshape(-1) if pool else None, torch.where(p > r, -sg, sg).reshape(-1) if pool else None)
            io, jo = torch.triu_indices(no, no, 1, device=dev)
            iv, jv = torch.triu_indices(nv, nv, 1, device=dev)
            for kind in ("aa", "bb", "ab"):
                if kind == "ab":
                    a = A[:, :no, None].expand(-1, no, no).reshape(len(d), -1)
                    b = B[:, None, :no].expand(-1, no, no).reshape(len(d), -1)
                    x = A[:, no:, None].expand(-1, nv, nv).reshape(len(d), -1)
                    y = B[:, None, no:].expand(-1, nv, nv).reshape(len(d), -1)
                else:
                    X = A if kind == "aa" else B
                    a, b, x, y = X[:, io], X[:, jo], X[:, no + iv], X[:, no + jv]
                if a.shape[1] == 0 or x.shape[1] == 0:
                    continue
                no2, nv2 = a.shape[1], x.shape[1]
                p, q = torch.minimum(a, b), torch.maximum(a, b)
                r, s = torch.minimum(x, y), torch.maximum(x, y)
                p, q = (v[:, :, None].expand(-1, no2, nv2).reshape(len(d), -1) for v in (p, q))
                r, s = (v[:, None, :].expand(-1, no2, nv2).reshape(len(d), -1) for v in (r, s))
                dd = d[:, None].expand_as(p)
                sg = 1.0 - 2.0 * _phase2(dd, p, q, r, s).to(torch.float64)
                v = self.g[((r * n + s) * n + p) * n + q] * sg
                k = sk = None
                if pool:
                    pa, pb = self._pair(p, q), self._pair(r, s)
                    k = self.two[torch.minimum(pa, pb) * self.np + torch.maximum(pa, pb)].reshape(-1)
                    sk = torch.where(pa > pb, -sg, sg).reshape(-1)
                yield (row[:, None].expand_as(p).reshape(-1), (dd ^ _bit(p) ^ _bit(q) ^ _bit(r) ^ _bit(s)).reshape(-1),
                       v.reshape(-1), k, sk)


def _hamiltonian_on(case, h, g, keys):
    """H restricted to the (ascending) keys, as (row, column, value)."""
    out = []
    for row, e, v, _, _ in _Pairs(case, h, g).blocks(keys, True, False):
        at = torch.searchsorted(keys, e).clamp(max=len(keys) - 1)
        hit = keys[at] == e
        out.append((row[hit], at[hit], v[hit]))
    return tuple(torch.cat(x) for x in zip(*out))


def _pool_step(case, h, g, keys, amps):
    pairs = _Pairs(case, h, g)
    es, vs = [], []
    for row, e, v, _, _ in pairs.blocks(keys, True, False):
        es.append(e)
        vs.append(v * amps[row])
    ext, inv = torch.unique(torch.cat(es), return_inverse=True)
    sigma = torch.zeros(len(ext), dtype=torch.float64, device=keys.device).index_add_(0, inv, torch.cat(vs))
    del es, vs, inv
    grad = torch.zeros(pairs.pool, dtype=torch.float64, device=keys.device)
    for row, e, _, k, sk in pairs.blocks(keys, False, True):
        grad.index_add_(0, k, sk * amps[row] * sigma[torch.searchsorted(ext, e)])
    n2 = (amps * amps).sum()
    energy = (amps * sigma[torch.searchsorted(ext, keys)]).sum() / n2
    return 2.0 * grad / n2, energy, n2


def _net_exact(case, seed):
    dev = _dev()
    x, t = _net_rows(case, seed)
    x, t = x.to(dev, torch.float64), t.to(dev, torch.float64)
    W1, b1, W2, b2, w3, b3 = (torch.from_numpy(v).to(dev) for v in _network(case, seed))
    W1, W2, w3 = (v.to(torch.bfloat16).to(torch.float64) for v in (W1, W2, w3))  # the network's weights are BF16
    par = [v.to(torch.float64).requires_grad_() for v in (W1, b1, W2, b2, w3, b3)]
    y = torch.relu(torch.relu(x @ par[0].T + par[1]) @ par[2].T + par[3]) @ par[4] + par[5]
    if case["kind"] == "net_predict":
        return y.detach()
    loss = ((y - t) ** 2).mean()
    loss.backward()
    return dict(grad=torch.cat([v.grad.reshape(-1) for v in par]), loss=loss.detach().reshape(1))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("net_predict", "net_grad"):
        return _net_exact(case, seed)
    if kind in ("batch", "screened"):
        return None
    dets, conn, _ = _shape(case)
    if dets * case["gates"] > GATE_WORK_EXACT or dets * (conn + 1) > PAIRS_EXACT[kind]:
        return None
    h, g, ops, theta = _system(case, seed)
    th = torch.tensor(theta, dtype=torch.float64, device=_dev(), requires_grad=kind == "vqe_grad")
    keys, amps = _gates(case, ops, th, kind == "vqe_grad")
    if kind == "pool_step":
        grad, energy, n2 = _pool_step(case, h, g, keys, amps)
        return dict(g=grad, e=float(energy), n2=float(n2), dets=None)
    i, j, v = _hamiltonian_on(case, h, g, keys)
    n2 = (amps * amps).sum()
    energy = (amps[i] * v * amps[j]).sum() / n2
    if kind == "state":
        return dict(e=float(energy), n2=float(n2), keys=None, amps=amps)
    energy.backward()
    return dict(e=float(energy.detach()), d=th.grad)
