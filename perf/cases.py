"""Performance cases: the calls a program makes of this framework, over the range of sizes it makes them in.

Four kinds of work, each through the public binding (paper_1810_07485_gb300.lcqmc):

  chain    one Markov chain: update(n), then its records; with "observe" the running averages too, with "export" the
           world-line configuration, as a program that writes a checkpoint reads it
  batch    many uneven chains updated together, then each chain's running averages
  served   simulation requests submitted to the continuous-batching server, polled until each is done
  ising    Swendsen-Wang updates of the 2D Ising lattice, their records and the spins

Chains are thermalized by a few updates from the Neel state before the first pass, and every pass goes on from the
state that the last one left, as a simulation does.  A record holds every count of its update and the exact 128-bit
sums over all loops; the next update's record depends on the whole configuration the last one wrote.
"""
import math
import time

import numpy as np
import torch

from paper_1810_07485_gb300 import lcqmc, workloads

KC = math.log(1.0 + math.sqrt(2.0)) / 2.0  # critical coupling of the 2D Ising model
MAX_VOLUME = float(1 << 30)                # largest Q^2 J beta L of one chain


def chain(L, beta, S=0.5, J=1.0, updates=1, thermal=8, temporal=False, observe=False, export=False):
    return dict(kind="chain", L=L, beta=beta, S=S, J=J, updates=updates, thermal=thermal, temporal=temporal,
                observe=observe, export=export)


def batch(chains, L_min, L_max, updates):
    return dict(kind="batch", chains=chains, L_min=L_min, L_max=L_max, updates=updates)


def served(requests, L_min, L_max, updates, slots):
    return dict(kind="served", requests=requests, L_min=L_min, L_max=L_max, updates=updates, slots=slots)


def ising(L, K, updates=1, spins=False):
    return dict(kind="ising", L=L, K=K, updates=updates, spins=spins)


def listed():
    return [
        # the accuracy configuration, driven one update and one record at a time
        dict(name="chain_L64_step", **chain(64, 16.0, thermal=40)),
        # the same chain in blocks of updates with its averages: how a program gathers statistics
        dict(name="chain_L64_block", **chain(64, 16.0, updates=100, thermal=40, observe=True, export=True)),
        # a mid-size chain checkpointed after a block of updates
        dict(name="chain_L1024_checkpoint", **chain(1024, 256.0, updates=16, thermal=24, export=True)),
        # a low-temperature chain, one record per update
        dict(name="chain_L16384_cold", **chain(16384, 4096.0, thermal=8)),
        # the largest single chain (7.4e8 vertices), one record per update
        dict(name="chain_L1048576", **chain(1 << 20, 1024.0, thermal=4)),
        # sizes no tile or window divides, the temporal moment (gap) on
        dict(name="chain_L4098_temporal", **chain(4098, 1000.7, J=0.7, updates=4, thermal=12, temporal=True)),
        # spin 1: four sub-bonds a bond, subspins joined at tau = 0
        dict(name="chain_S1_L4096", **chain(4096, 1024.0, S=1.0, thermal=8)),
        # spin 2, small: sixteen sub-bonds a bond; checkpointed after a block
        dict(name="chain_S2_L130", **chain(130, 60.5, S=2.0, updates=8, thermal=16, export=True)),
        # many uneven chains at once: a parameter scan
        dict(name="batch_192", **batch(192, 32, 4096, 10)),
        # requests of both spins arriving together, results polled
        dict(name="served_24", **served(24, 64, 1024, 50, 16)),
        # the paper's union-find benchmark: a block of updates at the critical point, the lattice read back
        dict(name="ising_L8192", **ising(8192, KC, updates=16, spins=True)),
        # a small odd lattice, spins read back
        dict(name="ising_L333", **ising(333, 0.5, updates=16, spins=True)),
    ]


def log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["chain"] * 6 + ["batch", "served", "ising", "ising"])
    if kind == "batch":
        L_max = 2 * int(log_uniform(rng, 32, 2048))
        return batch(int(log_uniform(rng, 4, 160)), 16, max(32, L_max), rng.randint(1, 10))
    if kind == "served":
        return served(rng.randint(2, 24), 8, 2 * int(log_uniform(rng, 32, 500)), rng.randint(5, 50), rng.randint(2, 24))
    if kind == "ising":
        L = int(log_uniform(rng, 16, 8192))
        K = KC if rng.random() < 0.5 else round(rng.uniform(0.1, 0.8), 3)
        return ising(L, K, updates=max(1, min(64, (1 << 23) // (L * L))), spins=L < 2048)
    while True:
        S = rng.choice([0.5, 0.5, 0.5, 1.0, 1.5, 2.0])
        J = rng.choice([1.0, 1.0, round(rng.uniform(0.3, 2.0), 2)])
        L = 2 * max(1, int(log_uniform(rng, 2, 1 << 20) / 2))
        beta = round(L * log_uniform(rng, 2.0 ** -10, 4.0) / J, 3)
        volume = 4 * S * S * J * beta * L
        if 64.0 <= volume <= MAX_VOLUME / 2:
            break
    return chain(L, beta, S, J, updates=max(1, min(100, int(2e6 / volume))), thermal=4 if volume > 1e8 else 12,
                 temporal=rng.random() < 0.25, observe=rng.random() < 0.3, export=volume < 3e5 and rng.random() < 0.5)


# ---- inputs -------------------------------------------------------------------------

def batch_specs(case, seed):
    return [dict(s, seed=seed * 100003 + s["seed"]) for s in
            workloads.batch_specs(case["chains"], case["L_min"], case["L_max"], seed=seed)]


def request_specs(case, seed):
    stream = workloads.request_stream(case["requests"], 1.0, case["L_min"], case["L_max"], n_updates=case["updates"],
                                      seed=seed)
    return [dict(s, seed=seed * 100003 + s["seed"]) for _, s in stream]


def ising_start(case, seed):
    return workloads.ising_spins(case["L"], seed)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "chain":
        ch = lcqmc.Chain(case["L"], case["beta"], S=case["S"], J=case["J"], seed=seed)
        if case["temporal"]:
            ch.set_temporal(True)
        ch.update(case["thermal"])
        ch.records()
        return dict(case=case, chain=ch)
    if kind == "batch":
        specs = batch_specs(case, seed)
        b = lcqmc.Batch(specs)
        b.update(4)
        b.sync()
        return dict(case=case, batch=b)
    if kind == "served":
        return dict(case=case, server=lcqmc.Server(hbm_budget=20 << 30, max_slots=case["slots"]),
                    requests=request_specs(case, seed))
    h = lcqmc.SWIsing(case["L"], case["K"], seed=seed)
    h.set_spins(ising_start(case, seed), 0)
    h.update(4)
    h.records()
    return dict(case=case, ising=h)


# ---- passes -------------------------------------------------------------------------

def fields(recs):
    """A record array as one array per field."""
    out = {}
    for name in recs.dtype.names:
        v = np.ascontiguousarray(recs[name])
        out[name] = v.view(np.int64) if v.dtype == np.uint64 else v
    return out


def padded(tau, case):
    """The operator times with zeros up to a length that the case alone gives: their number differs by seed."""
    volume = 4 * case["S"] ** 2 * case["J"] * case["beta"] * case["L"]
    out = np.zeros(int(0.45 * volume + 16.0 * math.sqrt(volume) + 64))
    out[:tau.size] = tau
    return out


def averages(o):
    out = dict(n_updates=int(o.n_updates), sum=np.array(o.sum), sumsq=np.array(o.sumsq))
    if hasattr(o, "xi"):
        out.update(xi=float(o.xi), xi_tau=float(o.xi_tau), gap=float(o.gap))
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "chain":
        ch = state["chain"]
        ch.update(case["updates"])
        out = dict(records=fields(ch.records()))
        if case["observe"]:
            out["averages"] = averages(ch.measure())
        if case["export"]:
            out["spins"], out["op_ptr"], tau = ch.export_config()
            out["op_tau"] = padded(tau, case)
        return out
    if case["kind"] == "batch":
        b = state["batch"]
        b.update(case["updates"])
        obs = [b.measure(i) for i in range(b.n)]
        return dict(sum=np.array([list(o.sum) for o in obs]), sumsq=np.array([list(o.sumsq) for o in obs]),
                    xi=np.array([o.xi for o in obs]))
    if case["kind"] == "served":
        srv, done = state["server"], {}
        tickets = [srv.submit(r["L"], r["beta"], r["n_updates"], S=r["S"], J=r["J"], seed=r["seed"])
                   for r in state["requests"]]
        while len(done) < len(tickets):
            for t in tickets:
                if t not in done:
                    r = srv.poll(t)
                    if r is not None:
                        done[t] = r
            if len(done) < len(tickets):
                time.sleep(0.0005)
        res = [done[t] for t in tickets]
        return dict(status=np.array([r.status for r in res]), sum=np.array([list(r.obs.sum) for r in res]),
                    sumsq=np.array([list(r.obs.sumsq) for r in res]), xi=np.array([r.obs.xi for r in res]))
    h = state["ising"]
    h.update(case["updates"])
    out = dict(records=fields(h.records()))
    if case["spins"]:
        out["spins"] = h.spins()
    return out


# ---- what a pass cannot do without ----------------------------------------------------

# Off-diagonal operators per Q^2 J beta L at low temperature: two thirds of the ground-state energy of the chain for
# S = 1/2 (ln 2 - 1/4), two thirds of -E / (4 S^2) for S = 1 (1.4015 / 4); larger S lie close above S = 1.
OPS = {0.5: 0.2954, 1.0: 0.2336, 1.5: 0.21, 2.0: 0.20}


def chain_work(L, beta, S, J, updates):
    """Per update: every operator time, cell offset and spin read once and written once, and one record; one fused
    multiply-add for each candidate vertex."""
    Q = int(round(2 * S))
    volume = Q * Q * J * beta * L
    cells = L * Q * Q * math.ceil(beta * J / 16.0)
    return dict(bytes=updates * (16.0 * OPS[S] * volume + 8.0 * (cells + 1) + 2.0 * L * Q + 136.0),
                flops=updates * volume)


def work(case):
    kind = case["kind"]
    if kind == "chain":
        return chain_work(case["L"], case["beta"], case["S"], case["J"], case["updates"])
    if kind == "ising":  # a byte a spin in and out
        return dict(bytes=case["updates"] * (2.0 * case["L"] ** 2 + 72.0), flops=0.0)
    specs = batch_specs(case, 0) if kind == "batch" else request_specs(case, 0)
    w = [chain_work(s["L"], s["beta"], s["S"], s["J"], case["updates"]) for s in specs]
    return dict(bytes=sum(x["bytes"] for x in w), flops=sum(x["flops"] for x in w))


# ---- the same in plain numpy, 64 bits ---------------------------------------------------

def philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 of arrays of counters: four arrays of 32-bit words."""
    m32 = np.uint64(0xFFFFFFFF)
    c0, c1, c2, c3 = (x.astype(np.uint64) for x in np.broadcast_arrays(*(np.asarray(v, dtype=np.int64)
                                                                          for v in (c0, c1, c2, c3))))
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c0, np.uint64(0xCD9E8D57) * c2
        c0, c1, c2, c3 = ((p1 >> np.uint64(32)) ^ c1 ^ np.uint64(k0), p1 & m32,
                          (p0 >> np.uint64(32)) ^ c3 ^ np.uint64(k1), p0 & m32)
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1, c2, c3


def coins(tag, ids, sweep, seed):
    """One fair coin per id: bit (id mod 128) of the block id / 128."""
    ids = np.asarray(ids, dtype=np.int64)
    w = np.stack(philox(tag << 24, ids >> 7, 0, sweep, seed))
    return ((w[(ids & 127) >> 5, np.arange(ids.size)] >> (ids & 31).astype(np.uint64)) & np.uint64(1)).astype(np.int64)


def components(n, a, b):
    """The smallest node of each node's component."""
    par = np.arange(n)
    while True:
        while True:
            g = par[par]
            if np.array_equal(g, par):
                break
            par = g
        ra, rb = par[a], par[b]
        open_ = ra != rb
        if not open_.any():
            return par
        a, b, ra, rb = a[open_], b[open_], ra[open_], rb[open_]
        np.minimum.at(par, np.maximum(ra, rb), np.minimum(ra, rb))


def thresholds(mu):
    p, cdf, out = math.exp(-mu), 0.0, []
    for k in range(47):
        p = p * mu / k if k else p
        cdf += p
        out.append(min(int(math.ldexp(cdf, 64)), 2 ** 64 - 1))
    return np.array(out, dtype=np.uint64)


class PlainChain:
    """The keyed loop update of one chain, vectorized over the whole lattice."""

    def __init__(self, L, beta, S, J, seed):
        self.L, self.Q, self.beta, self.J, self.seed = L, int(round(2 * S)), beta, J, seed
        self.w = 16.0 / J
        self.nwin = max(1, math.ceil(beta / self.w))
        self.nbond = L * self.Q ** 2
        self.spin = (np.arange(L * self.Q) // self.Q) & 1
        self.cell, self.tau = np.zeros(0, np.int64), np.zeros(0)
        self.sweep = 0
        b, j = np.meshgrid(np.arange(self.nbond), np.arange(self.nwin), indexing="ij")
        self.b, self.j = b.ravel(), j.ravel()  # of every cell, in no particular order
        blk = self.j // 4
        tw = np.minimum(4, self.nwin - 4 * blk)
        self.id = blk * self.nbond * 4 + self.b * tw + self.j % 4  # its place in the cell order
        self.bond_of = np.empty(self.b.size, np.int64)
        self.bond_of[self.id] = self.b

    def ends(self, bond):
        Q = self.Q
        i = bond // (Q * Q)
        return i * Q + bond // Q % Q, (i + 1) % self.L * Q + bond % Q

    def candidates(self):
        nw, w = self.nwin, self.w
        t0 = self.j * w
        d = np.where(self.j == nw - 1, self.beta, (self.j + 1) * w) - t0
        first = philox(1 << 24, self.b, self.j, self.sweep, self.seed)
        U = first[0] | (first[1] << np.uint64(32))
        last = self.j == nw - 1
        left = self.beta - (nw - 1) * w
        K = np.where(last, np.searchsorted(thresholds(self.J * left * 0.5), U, side="right"),
                     np.searchsorted(thresholds(8.0), U, side="right"))
        K = np.where(d > 0, K, 0)
        c = np.repeat(np.arange(K.size), K)
        k = np.arange(c.size) - np.repeat(np.cumsum(K) - K, K)
        o = philox((1 << 24) | ((k + 1) // 2), self.b[c], self.j[c], self.sweep, self.seed)
        odd = k & 1 == 1
        u53 = np.where(odd, o[0] | (o[1] << np.uint64(32)), o[2] | (o[3] << np.uint64(32))) >> np.uint64(11)
        tau = d[c] * np.ldexp(u53.astype(np.float64), -53) + t0[c]
        keep = tau < t0[c] + d[c]
        return self.id[c][keep], tau[keep], u53[keep], k[keep]

    def spins_at(self, u, tau, bond):
        """The spin of subsite u just before (tau, bond)."""
        ol, or_ = self.ends(self.bond_of[self.cell])
        n = u.size
        key_u = np.concatenate([u, ol, or_])
        key_t = np.concatenate([tau, self.tau, self.tau])
        ob = self.bond_of[self.cell]
        key_b = np.concatenate([bond, ob, ob])
        event = np.concatenate([np.zeros(n, np.int64), np.ones(2 * ob.size, np.int64)])
        order = np.lexsort((event, key_b, key_t, key_u))
        e, uu = event[order], key_u[order]
        run_ = np.cumsum(e) - e
        start = np.searchsorted(uu, uu, side="left")
        before = np.empty(order.size, np.int64)
        before[order] = run_ - run_[start]
        return self.spin[u] ^ (before[:n] & 1)

    def joins(self, site, top):
        """The bottom subspin that each top subspin of a site continues into."""
        Q, s0 = self.Q, self.spin[site * self.Q:(site + 1) * self.Q]
        if Q == 1:
            return [0]
        if Q == 2:
            same, swapped = list(top) == list(s0), list(top) == list(s0[::-1])
            swap = coins(4, [site], self.sweep, self.seed)[0] if same and swapped else int(swapped)
            return [1, 0] if swap else [0, 1]
        words = [int(x) for x in philox((4 << 24) | 1, site, 0, self.sweep, self.seed)]
        perm, d = [0] * Q, 0
        for spin in (1, 0):
            tops = [a for a in range(Q) if top[a] == spin]
            bots = [a for a in range(Q) if s0[a] == spin]
            for j in range(len(bots) - 1, 0, -1):
                r = (words[d & 3] * (j + 1)) >> 32
                d += 1
                bots[j], bots[r] = bots[r], bots[j]
            for a, b in zip(tops, bots):
                perm[a] = b
        return perm

    def update(self):
        L, Q, beta, sweep, seed = self.L, self.Q, self.beta, self.sweep, self.seed
        cc, ct, cu, ck = self.candidates()
        cb = self.bond_of[cc]
        cl, cr = self.ends(cb)
        keep = self.spins_at(cl, ct, cb) != self.spins_at(cr, ct, cb)
        cc, ct, cu, ck = cc[keep], ct[keep], cu[keep], ck[keep]
        old = np.concatenate([np.ones(self.cell.size, np.int64), np.zeros(cc.size, np.int64)])
        cell, tau = np.concatenate([self.cell, cc]), np.concatenate([self.tau, ct])
        place = np.concatenate([np.arange(self.cell.size), ck])
        u53 = np.concatenate([np.zeros(self.cell.size, np.uint64), cu])
        order = np.lexsort((place, u53, 1 - old, tau, cell))
        old, cell, tau = old[order], cell[order], tau[order]
        n = tau.size
        vl, vr = self.ends(self.bond_of[cell])
        # legs of each subsite in time order
        nsub = L * Q
        leg_u, leg_v = np.concatenate([vl, vr]), np.concatenate([np.arange(n), np.arange(n)])
        order = np.lexsort((leg_v, tau[leg_v], leg_u))
        su, sv = leg_u[order], leg_v[order]
        count = np.bincount(su, minlength=nsub)
        start = np.cumsum(count) - count
        last = np.where(count > 0, sv[np.maximum(start + count - 1, 0)] if n else -1, -1)
        # the tau = 0 cut
        ops_on = np.bincount(vl[old == 1], minlength=nsub) + np.bincount(vr[old == 1], minlength=nsub)
        top = self.spin ^ (ops_on & 1)
        feed, cross, free_min, free_len = (np.empty(nsub, np.int64) for _ in range(4))
        if Q == 1:
            feed[:], cross[:], free_min[:], free_len[:] = last, 1, np.arange(nsub), 1
        else:
            for site in range(L):
                perm = self.joins(site, top[site * Q:(site + 1) * Q])
                inv = [perm.index(a) for a in range(Q)]
                for a in range(Q):
                    x, steps, seen = a, 0, a
                    for _ in range(Q):
                        x = inv[x]
                        steps += 1
                        seen = min(seen, x)
                        if last[site * Q + x] >= 0 or x == a:
                            break
                    u = site * Q + a
                    feed[u], cross[u], free_min[u], free_len[u] = last[site * Q + x], steps, site * Q + seen, steps
        # predecessors of both legs of every vertex, fragment lengths
        first = np.zeros(2 * n, bool)
        first[start[count > 0]] = True
        pred = np.where(first, feed[su], np.roll(sv, 1))
        length = tau[sv] - tau[pred] + np.where(first, cross[su] * beta, 0.0)
        P, dl = np.empty(2 * n, np.int64), np.empty(2 * n)
        P[order], dl[order] = pred, length
        pl, pr = P[:n], P[n:]
        root = components(n, pl, pr)
        flip = np.zeros(n, np.int64)
        heads = np.flatnonzero(root == np.arange(n))
        flip[heads] = coins(2, heads, sweep, seed)
        flip = flip[root]
        loop = root[P]
        angle = 2.0 * math.pi * (np.concatenate([vl, vr]) // Q) / L
        W = np.bincount(loop, dl, n)
        C, D = np.bincount(loop, dl * np.cos(angle), n), np.bincount(loop, dl * np.sin(angle), n)
        w1 = 2.0 * math.pi / beta
        end = np.concatenate([tau, tau])
        zr = np.bincount(loop, np.cos(w1 * end) - np.cos(w1 * tau[P]), n)
        zi = np.bincount(loop, np.sin(w1 * end) - np.sin(w1 * tau[P]), n)
        # vertex-free loops
        free = (feed < 0) & (free_min == np.arange(nsub))
        free_w = free_len[free] * beta
        new = old ^ flip[pl] ^ flip if n else old
        bottom = feed >= 0
        turn = np.zeros(nsub, np.int64)
        turn[bottom] = flip[feed[bottom]]
        turn[~bottom] = coins(3, free_min[~bottom], sweep, seed)
        n_old, n_new, n_free = int(old.sum()), int(new.sum()), int(free.sum())
        self.spin = self.spin ^ turn
        self.cell, self.tau = cell[new == 1], tau[new == 1]
        self.sweep += 1
        scale = 1.0 / (4.0 * beta * L)
        rec = dict(energy=Q * Q * self.J / 4 - n / (beta * L),
                   chi_s=((W ** 2).sum() + (free_w ** 2).sum()) * scale,
                   chi_q=((C ** 2 + D ** 2).sum() + (free_w ** 2).sum()) * scale,
                   chi_w=(zr ** 2 + zi ** 2).sum() * beta / (16.0 * math.pi ** 2 * L))
        clusters = heads.size + n_free
        seg = 2 * n + n_free
        return rec, (rec["energy"], rec["chi_s"], rec["chi_q"], n, n_new, seg, clusters, seg + 2 * n, rec["chi_w"])


def plain_averages(rows, L, beta, temporal):
    """Running sums, sums of squares and correlation lengths of a chain's updates."""
    x = np.array(rows)
    if not temporal:
        x[:, 8] = 0.0
    s = x.sum(axis=0)
    ratio = s[1] / s[2] - 1.0 if s[2] > 0 else 0.0
    out = dict(sum=s, sumsq=(x ** 2).sum(axis=0), xi=L / (2 * math.pi) * math.sqrt(ratio) if ratio > 0 else 0.0)
    ratio = s[1] / s[8] - 1.0 if s[8] > 0 else 0.0
    out["xi_tau"] = beta / (2 * math.pi) * math.sqrt(ratio) if ratio > 0 else 0.0
    out["gap"] = 1.0 / out["xi_tau"] if out["xi_tau"] > 0 else 0.0
    return out


def plain_cost(L, beta, S, J, updates):
    """Rough seconds of `updates` plain updates."""
    Q = int(round(2 * S))
    return updates * (1e-3 + 6e-6 * Q * Q * J * beta * L + (0 if Q == 1 else 6e-5 * L * Q))


def exact(case, seed):
    kind = case["kind"]
    if kind == "chain":
        total = case["thermal"] + case["updates"]
        if plain_cost(case["L"], case["beta"], case["S"], case["J"], total) > 12.0:
            return None
        c = PlainChain(case["L"], case["beta"], case["S"], case["J"], seed)
        done = [c.update() for _ in range(total)]
        recs = [r for r, _ in done[case["thermal"]:]]
        out = dict(records={f: np.array([r[f] for r in recs]) for f in ("energy", "chi_s", "chi_q")})
        if case["temporal"]:
            out["records"]["chi_w"] = np.array([r["chi_w"] for r in recs])
        if case["observe"]:
            out["averages"] = plain_averages([x for _, x in done], case["L"], case["beta"], case["temporal"])
        if case["export"]:
            out["op_tau"] = padded(c.tau, case)
        return out
    if kind == "ising":
        L, N = case["L"], case["L"] ** 2
        total = 4 + case["updates"]
        if total * N > 4e6:
            return None
        T = min(max(int(math.floor(math.ldexp(-math.expm1(-2.0 * case["K"]), 32) + 0.5)), 0), 1 << 32)
        spin, ids = ising_start(case, seed).astype(np.int64), np.arange(N)
        right, down = ids // L * L + (ids + 1) % L, (ids + L) % N
        energy, chi = [], []
        for sweep in range(total):
            wr, wd, _, _ = philox(5 << 24, ids, 0, sweep, seed)
            er, ed = spin == spin[right], spin == spin[down]
            r, d = er & (wr < T), ed & (wd < T)
            root = components(N, np.concatenate([ids[r], ids[d]]), np.concatenate([right[r], down[d]]))
            energy.append((2.0 * N - 2.0 * (er.sum() + ed.sum())) / N)
            chi.append(float((np.bincount(root, minlength=N).astype(np.float64) ** 2).sum()) / N)
            spin = spin ^ coins(6, root, sweep, seed)
        return dict(records=dict(energy=np.array(energy[4:]), chi=np.array(chi[4:])))
    if kind == "batch":
        specs, total = batch_specs(case, seed), 4 + case["updates"]
    else:
        specs, total = request_specs(case, seed), case["updates"]
    if sum(plain_cost(s["L"], s["beta"], s["S"], s["J"], total) for s in specs) > 12.0:
        return None
    rows = []
    for s in specs:
        c = PlainChain(s["L"], s["beta"], s["S"], s["J"], s["seed"])
        rows.append(plain_averages([c.update()[1] for _ in range(total)], s["L"], s["beta"], False))
    return dict((f, np.array([r[f] for r in rows])) for f in ("sum", "sumsq", "xi"))
