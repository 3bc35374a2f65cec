"""The work that programs have this library do, as cases to be timed.

Three kinds of case, each through the public entry points that a solver calls:

  sweep    a run in progress: `ctaux_sweep` over a few submatrix blocks with a measurement after
           each (and, where `refresh` is set, the periodic from-scratch recomputation at that
           cadence), then the read-back of the accumulated Green's function and of the
           configuration that a program writes to its output or checkpoint;
  restart  a run that resumes: `ctaux_set_config` of a stored configuration (which rebuilds N
           from scratch) and the read-back of N of both spins;
  invert   `ctaux_invert_noalloc` on a matrix that another allocator owns.

The model systems are those of workloads/configs.py: the single-site impurity, the 4-, 8- and
16-site clusters and their uneven batches, the 6 x 6 cluster away from half filling and the
100-site cluster.  Every start is a seeded configuration of the stated order.
"""
import dataclasses
import functools
import math

import numpy as np
import torch

import paper_1010_3690_gb300 as pk
from paper_1010_3690_gb300 import ctaux as ct
from workloads import configs

BINS, ANCHORS = 32, 4


def listed():
    def sweep(name, **kw):
        base = dict(name=name, kind="sweep", precision="f64", gamma="inverse", p_flip=0.0, freqs=0,
                    chains=1)
        return {**base, **kw}

    return [
        # the smallest call: a few short blocks of the impurity, all launch and step latency
        sweep("impurity_f64", n_c=1, beta=10.0, U=4.0, order=30, k=8, blocks=8, refresh=8),
        # one 2x2x2 chain at its equilibrium order, the common production run on a small cluster
        sweep("cube8_f64", n_c=8, beta=5.0, U=8.0, order=415, k=64, blocks=16, refresh=16),
        # the same cluster in float32 with the options that direct frequency measurements use:
        # Gamma as L U, spin flips among the moves, 16 Matsubara frequencies
        sweep("cube8_mixed_lu_freqs", n_c=8, beta=5.0, U=8.0, order=401, k=32, blocks=8, refresh=8,
              precision="mixed", gamma="lu", p_flip=0.2, freqs=16),
        # 6 x 6 cluster off half filling, one refresh period
        sweep("square36_f64", n_c=36, beta=8.0, U=6.0, order=2085, k=128, blocks=8, refresh=8),
        sweep("square36_mixed_df64", n_c=36, beta=8.0, U=6.0, order=2085, k=128, blocks=16,
              refresh=16, precision="mixed_df64"),
        # uneven chains in one launch: many walkers of small clusters on one GPU
        sweep("batch_f64", n_c=0, beta=0.0, U=0.0, order=0, k=32, blocks=4, refresh=4, chains=40),
        sweep("batch_mixed", n_c=0, beta=0.0, U=0.0, order=0, k=64, blocks=8, refresh=8, chains=96,
              precision="mixed"),
        # 100 sites, float64: one block of two chains between refreshes
        sweep("cube100_f64", n_c=100, beta=4.0, U=8.0, order=6760, k=256, blocks=1, refresh=0,
              chains=2),
        # 100 sites, mixed form with the float64 refresh that it keeps, one refresh period
        sweep("cube100_mixed", n_c=100, beta=4.0, U=8.0, order=6760, k=256, blocks=16, refresh=16,
              precision="mixed"),
        # resuming from a checkpoint: small cluster, and the 6 x 6 cluster at an odd order
        dict(name="restart_cube8", kind="restart", n_c=8, beta=5.0, U=8.0, order=431),
        dict(name="restart_square36", kind="restart", n_c=36, beta=8.0, U=6.0, order=1999),
        # a caller-owned matrix of the size of a small cluster's N
        dict(name="invert", kind="invert", m=310),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    model = {1: (10.0, 4.0), 4: (6.0, 8.0), 8: (5.0, 8.0), 16: (5.0, 8.0), 36: (8.0, 6.0),
             100: (4.0, 8.0)}
    kind = rng.choice(["sweep", "sweep", "sweep", "batch", "restart", "invert"])
    if kind == "invert":
        return dict(kind="invert", m=log_int(8, 512))
    if kind == "restart":
        order = log_int(60, 4000)
        n_c = rng.choice([8, 16] if order < 1000 else [36, 100])
        return dict(kind="restart", n_c=n_c, beta=model[n_c][0], U=model[n_c][1], order=order)
    precision = rng.choice(["f64", "f64", "mixed", "mixed_df64"])
    if kind == "batch":
        blocks = rng.randint(2, 8)
        return dict(kind="sweep", n_c=0, beta=0.0, U=0.0, order=0, k=rng.choice([16, 32, 64]),
                    blocks=blocks, refresh=blocks, chains=log_int(6, 96), precision=precision,
                    gamma="inverse", p_flip=0.0, freqs=0)
    n_c = rng.choice([1, 4, 8, 16, 36, 100])
    order = log_int(*{1: (12, 60), 4: (80, 400), 8: (150, 800), 16: (200, 1100), 36: (900, 2600),
                      100: (3000, 6700)}[n_c])
    k = log_int(*{1: (4, 32), 4: (12, 64), 8: (16, 96), 16: (16, 128), 36: (32, 160),
                  100: (96, 256)}[n_c])
    blocks = 1 if n_c == 100 else rng.randint(2, 12)
    return dict(kind="sweep", n_c=n_c, beta=model[n_c][0], U=model[n_c][1], order=order, k=k,
                blocks=blocks, refresh=0 if n_c == 100 else blocks, chains=1, precision=precision,
                gamma=rng.choice(["inverse", "inverse", "lu"]) if n_c < 36 else "inverse",
                p_flip=rng.choice([0.0, 0.0, 0.2]), freqs=rng.choice([0, 0, 8]) if n_c < 36 else 0)


# ------------------------------------------------------------------ inputs
_GRID = {1: 64, 4: 8, 8: 8, 16: 6, 36: 12, 100: 4}   # patch points per direction of the G0 tables


@functools.lru_cache(maxsize=None)
def _chain(n_c, beta, U, K, k, capacity):
    if n_c == 1:
        return configs.aim1(K=K, k_max=k, capacity=capacity, beta=beta, U=U)
    return configs.cluster_chain("c%d" % n_c, n_c, beta, U, K, k, capacity,
                                 density=0.9 if n_c == 36 else 1.0, n_grid=_GRID[n_c],
                                 n_tau=4096 if n_c >= 8 else 1024)


def _capacity(order, k):
    return (int(1.3 * order) + k + 95) // 32 * 32


def _chains(case, seed):
    """(chain inputs, starting orders) of a case; the Philox key is the seed."""
    if case["n_c"]:
        n_c, beta, U, order = case["n_c"], case["beta"], case["U"], case["order"]
        # the expansion constant at which the chain stays near its starting order
        K = 1.0 if n_c == 1 else max(order - 0.37 * beta * U * n_c, 0.15 * order)
        ch = _chain(n_c, beta, U, K, case.get("k", 1), _capacity(order, case.get("k", 1)))
        out, orders = [ch] * case.get("chains", 1), [order] * case.get("chains", 1)
    else:   # an uneven batch: cluster size, temperature and interaction per chain
        rng = np.random.default_rng(12345)
        out, orders = [], []
        for _ in range(case["chains"]):
            n_c = int(rng.choice([4, 8, 16]))
            beta, U = float(rng.choice([2.0, 4.0, 6.0, 8.0, 10.0])), round(rng.uniform(4.0, 10.0), 3)
            K = round(0.3 * beta * U * n_c + 30.0, 3)
            orders.append(int(K + 0.37 * beta * U * n_c))
            out.append(_chain(n_c, beta, U, K, case["k"], _capacity(orders[-1], case["k"])))
    return [dataclasses.replace(c, seed=seed & 0xFFFFFFFF, chain_id=i) for i, c in enumerate(out)], orders


def _configuration(ch, order, seed):
    return configs.synthetic_configuration(ch, order, seed=[seed & 0xFFFFFFFF, ch.chain_id])


def _matrix(case, seed):
    """N^{-1} of a random configuration: unit-scale rows, columns scaled by e^V - 1."""
    g = torch.Generator().manual_seed(seed & 0x7FFFFFFF)
    m = case["m"]
    a = torch.randn(m, m, generator=g, dtype=torch.float64) * (0.5 / math.sqrt(m))
    s = torch.where(torch.rand(m, generator=g, dtype=torch.float64) < 0.5, 2.0, 0.5).to(torch.float64)
    return torch.diag(s) - a * (s - 1.0)[None, :]


def prepare(case, seed):
    if case["kind"] == "invert":
        m = case["m"]
        a = _matrix(case, seed).cuda()
        return dict(kind="invert", m=m, a=a.t().contiguous(), inv=torch.empty_like(a),
                    logdet=torch.empty(1, dtype=torch.float64, device=a.device))
    chains, orders = _chains(case, seed)
    starts = [_configuration(c, n, seed) for c, n in zip(chains, orders)]
    if case["kind"] == "restart":
        ctx = pk.Context(chains, refresh_every=32, use_graph=1)
        return dict(kind="restart", ctx=ctx, start=starts[0])
    mixed = case["precision"] != "f64"
    ctx = pk.Context(chains, precision=pk.CTAUX_MIXED if mixed else pk.CTAUX_FP64,
                     refresh_every=case["refresh"], p_insert=0.5 * (1.0 - case["p_flip"]),
                     p_flip=case["p_flip"], n_tau_bins=BINS, n_anchors=ANCHORS, use_graph=1,
                     refresh_df64=int(case["precision"] == "mixed_df64"),
                     gamma_form=ct.CTAUX_GAMMA_LU if case["gamma"] == "lu" else ct.CTAUX_GAMMA_INVERSE,
                     n_matsubara=case["freqs"])
    for i, cfg in enumerate(starts):
        ctx.set_config(i, **cfg)
    return dict(kind="sweep", ctx=ctx, blocks=case["blocks"], chains=len(chains), freqs=case["freqs"],
                capacity=[c.capacity for c in chains],
                # the float32 form's results carry float32 accuracy
                real=np.float32 if mixed else np.float64)


def run(state):
    if state["kind"] == "invert":
        m = state["m"]
        code = ct.ctaux_invert_noalloc(state["a"].data_ptr(), m, state["inv"].data_ptr(), m, m,
                                       state["logdet"].data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
        if code:
            raise RuntimeError("ctaux_invert_noalloc: %d" % code)
        return dict(inv=state["inv"].t(), logdet=state["logdet"])
    ctx = state["ctx"]
    if state["kind"] == "restart":
        ctx.set_config(0, **state["start"])
        return dict(n_up=ctx.get_N(0, 0), n_down=ctx.get_N(0, 1),
                    logdet=np.array(ctx.stats(0)["logdet"]))
    ctx.sweep(state["blocks"], measure=True)
    every = range(state["chains"])
    out = dict(G=[ctx.measure_G(c)[0].ravel() for c in every])
    cfg = [ctx.get_config(c) for c in every]
    if state["freqs"]:
        out["Gw"] = [ctx.measure_G_matsubara(c)[0].ravel() for c in every]
    out = {k: np.concatenate(v) for k, v in out.items()}
    out["G"] = out["G"].astype(state["real"])
    if "Gw" in out and state["real"] is np.float32:
        out["Gw"] = out["Gw"].astype(np.complex64)
    for key in ("tau", "site", "s", "birth"):
        out[key] = _padded([c[key] for c in cfg], state["capacity"])
    out["order"] = np.array([len(c["tau"]) for c in cfg])
    return out


def _padded(rows, capacity):
    """Checkpoint rows of fixed length: each chain's values, zeros up to its capacity."""
    out = np.zeros(sum(capacity), rows[0].dtype)
    at = 0
    for row, cap in zip(rows, capacity):
        out[at:at + len(row)] = row
        at += cap
    return out


def work(case):
    """Bytes and flops of one pass (both spins).  A block reads N once and writes it once; it
    forms R~ = C N and N B for the k/2 insertion candidates and the rank-k_acc flush
    (k_acc ~ 0.8 k); a refresh inverts N^{-1} (2 n^3) and writes N."""
    if case["kind"] == "invert":
        m = case["m"]
        return {"bytes": 16.0 * m * m, "flops": 2.0 * m ** 3}
    if case["kind"] == "restart":
        n = case["order"]
        return {"bytes": 2 * 8.0 * n * n, "flops": 2 * 2.0 * n ** 3}
    size = 8.0 if case["precision"] == "f64" else 4.0
    _, orders = _chains(case, 0)
    b = f = 0.0
    for n in orders:
        k = case["k"]
        b += case["blocks"] * 2 * (2 * size * n * n)
        f += case["blocks"] * 2 * (2 * 2.0 * (k / 2) * n * n + 2.0 * 0.8 * k * n * n
                                   + 2.0 * ANCHORS * n * n)
        if case["refresh"]:
            times = case["blocks"] / case["refresh"]
            b += times * 2 * size * n * n
            f += times * 2 * 2.0 * n ** 3
    return {"bytes": b, "flops": f}


# -------------------------------------------------- the same in plain numpy
class _Plain:
    """CT-AUX by rank-one updates of an explicit float64 N, one proposal at a time."""

    def __init__(self, ch, cfg, p_insert=0.5, p_flip=0.0, mixed=False):
        self.ch, self.t, self.mixed, self.forced = ch, int(cfg["t"]), mixed, False
        self.tau, self.site = np.array(cfg["tau"]), np.array(cfg["site"], np.int64)
        self.s, self.birth = np.array(cfg["s"], np.int64), np.array(cfg["birth"], np.int64)
        self.p_insert, self.p_flip = p_insert, p_flip
        self.gamma = math.acosh(1.0 + ch.beta * ch.U * ch.n_c / (2.0 * ch.K))
        self.dtau = ch.beta / (ch.table.shape[2] - 1)

    def g0(self, spin, ti, xi, tj, xj):
        row = self.ch.table[spin]
        dt = ti - tj
        cls = self.ch.dx_class[xi, xj]
        cls, dt = np.broadcast_arrays(cls, dt)
        pos = np.where(dt < 0.0, dt + self.ch.beta, dt) / self.dtau
        i = np.clip(np.floor(pos).astype(np.int64), 0, row.shape[1] - 2)
        v = row[cls, i] + (pos - i) * (row[cls, i + 1] - row[cls, i])
        return np.where(dt == 0.0, -row[cls, -1], np.where(dt < 0.0, -v, v))

    def ev(self, spin, s):
        return np.exp((self.gamma if spin == 0 else -self.gamma) * np.asarray(s, np.float64))

    def inverse_matrix(self, spin):
        e = self.ev(spin, self.s)
        g = self.g0(spin, self.tau[:, None], self.site[:, None], self.tau[None], self.site[None])
        return np.diag(e) - g * (e - 1.0)[None]

    def refresh(self):
        self.N = [np.linalg.inv(self.inverse_matrix(spin)) for spin in (0, 1)]

    @staticmethod
    def _uniforms(seed, chain, t, purpose):
        """Philox-4x32-10 of the counter (t, chain, purpose): two uniforms of 53 bits."""
        m32 = 0xFFFFFFFF
        c, k0, k1 = [t & m32, t >> 32, chain, purpose], seed & m32, seed >> 32
        for _ in range(10):
            p, q = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
            c = [(q >> 32) ^ c[1] ^ k0, q & m32, (p >> 32) ^ c[3] ^ k1, p & m32]
            k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
        return [((c[i] << 21) + (c[i + 1] >> 11)) * 2.0 ** -53 for i in (0, 2)]

    def near_tie(self, u, R):
        """The float32 form ends its block before a decision that its rounding could change, and
        starts the next block with that proposal."""
        if self.mixed and not self.forced and abs(u - abs(R)) < 1e-4 * max(u, abs(R)):
            self.forced = True
            return True
        self.forced = False
        return False

    def block(self, k):
        for _ in range(k):
            if not self.step():
                break
            self.t += 1

    def step(self):
        """Proposal t; false where the block ends before it."""
        ch, t, n = self.ch, self.t, len(self.tau)
        (u_move, u_acc), (u_tau, u_site), (u_spin, u_idx) = [
            self._uniforms(ch.seed, ch.chain_id, t, p) for p in range(3)]
        if u_move < self.p_insert:
            tau, site = u_tau * ch.beta, min(int(u_site * ch.n_c), ch.n_c - 1)
            s = 1 if u_spin < 0.5 else -1
            new, ratio = [], 1.0
            for spin in (0, 1):
                e, ep = self.ev(spin, self.s), float(self.ev(spin, s))
                u = -self.g0(spin, self.tau, self.site, tau, site) * (ep - 1.0)
                w = -self.g0(spin, tau, site, self.tau, self.site) * (e - 1.0)
                d = ep - float(self.g0(spin, np.float64(tau), site, np.float64(tau), site)) * (ep - 1.0)
                nu = self.N[spin] @ u
                new.append((nu, w, d - w @ nu))
                ratio *= new[-1][2]
            R = ch.K / (n + 1) * ratio
            if self.near_tie(u_acc, R):
                return False
            if u_acc < abs(R):
                for spin, (nu, w, r) in enumerate(new):
                    wn = w @ self.N[spin]
                    big = np.empty((n + 1, n + 1))
                    big[:n, :n] = self.N[spin] + np.outer(nu / r, wn)
                    big[:n, n], big[n, :n], big[n, n] = -nu / r, -wn / r, 1.0 / r
                    self.N[spin] = big
                self.tau, self.site = np.append(self.tau, tau), np.append(self.site, site)
                self.s, self.birth = np.append(self.s, s), np.append(self.birth, t)
            return True
        if n == 0:
            return True
        i = min(int(u_idx * n), n - 1)
        if u_move < self.p_insert + (1.0 - self.p_insert - self.p_flip):
            r = [self.N[spin][i, i] for spin in (0, 1)]
            R = n / ch.K * r[0] * r[1]
            if self.near_tie(u_acc, R):
                return False
            if u_acc < abs(R):
                keep = np.arange(n) != i
                for spin in (0, 1):
                    N = self.N[spin]
                    self.N[spin] = (N - np.outer(N[:, i] / N[i, i], N[i]))[keep][:, keep]
                self.tau, self.site = self.tau[keep], self.site[keep]
                self.s, self.birth = self.s[keep], self.birth[keep]
            return True
        new, ratio = [], 1.0
        for spin in (0, 1):
            step = float(self.ev(spin, -self.s[i]) - self.ev(spin, self.s[i]))
            d = -step * self.g0(spin, self.tau, self.site, self.tau[i], self.site[i])
            d[i] += step
            nd = self.N[spin] @ d
            new.append((nd, 1.0 + nd[i]))
            ratio *= new[-1][1]
        if self.near_tie(u_acc, ratio):
            return False
        if u_acc < abs(ratio):
            for spin, (nd, r) in enumerate(new):
                self.N[spin] = self.N[spin] - np.outer(nd / r, self.N[spin][i])
            self.s[i] = -self.s[i]
        return True

    def greens_function(self):
        """G_sigma(class, bin) of this configuration, averaged over anchors and sites."""
        ch = self.ch
        cls = ch.dx_class[:, 0]
        tau_c = (np.arange(BINS) + 0.5) * ch.beta / BINS
        out = np.zeros((2, ch.table.shape[1], BINS))
        sites = np.arange(ch.n_c)
        for spin in (0, 1):
            for a in range(ANCHORS):
                tb = a * ch.beta / ANCHORS
                ta = tb + tau_c
                sign = np.where(ta >= ch.beta, -1.0, 1.0)
                ta = np.where(ta >= ch.beta, ta - ch.beta, ta)
                val = self.g0(spin, ta[None], sites[:, None], np.float64(tb), 0)
                gb = self.g0(spin, self.tau, self.site, np.float64(tb), 0)
                v = (self.ev(spin, self.s) - 1.0) * (self.N[spin] @ gb)
                val = val + self.g0(spin, ta[None, :, None], sites[:, None, None],
                                    self.tau[None, None], self.site[None, None]) @ v
                np.add.at(out[spin], cls, sign * val / ANCHORS)
            out[spin] /= np.maximum(np.bincount(cls, minlength=out.shape[1]), 1)[:, None]
        return out

    def greens_function_matsubara(self, freqs):
        """G_xy(i w_n): the transform of the same estimator, G0 linear between table points."""
        ch = self.ch
        w = (2.0 * np.arange(freqs) + 1.0) * math.pi / ch.beta
        n_tau, h, T = ch.table.shape[2], self.dtau, ch.table
        t0 = np.arange(n_tau - 1) * h
        z = 1j * w[:, None] * h
        e1 = np.expm1(z)
        c0 = e1 / z                              # int_0^1 e^{z x} dx
        c1 = (np.exp(z) - c0) / z                # int_0^1 x e^{z x} dx
        ph = np.exp(1j * w[:, None] * t0[None]) * h
        g0w = (np.einsum("scj,fj->scf", T[..., :-1], ph * (c0 - c1))
               + np.einsum("scj,fj->scf", T[..., 1:], ph * c1))[:, ch.dx_class, :]
        sel = np.zeros((ch.n_c, len(self.tau)))
        sel[self.site, np.arange(len(self.tau))] = 1.0
        out = np.array(g0w)
        for spin in (0, 1):
            M = (self.ev(spin, self.s) - 1.0)[:, None] * self.N[spin]
            for f in range(freqs):
                p = sel * np.exp(1j * w[f] * self.tau)[None]
                S = p @ M @ p.conj().T
                out[spin, :, :, f] += g0w[spin, :, :, f] @ S @ g0w[spin, :, :, f] / ch.beta
        return out


def exact(case, seed):
    if case["kind"] == "invert":
        a = _matrix(case, seed).numpy()
        return dict(inv=np.linalg.inv(a), logdet=np.array([np.linalg.slogdet(a)[1]]))
    chains, orders = _chains(case, seed)
    if case["kind"] == "restart":
        p = _Plain(chains[0], _configuration(chains[0], orders[0], seed))
        m = [p.inverse_matrix(spin) for spin in (0, 1)]
        return dict(n_up=np.linalg.inv(m[0]), n_down=np.linalg.inv(m[1]),
                    logdet=np.array([np.linalg.slogdet(x)[1] for x in m]))
    # a proposal of the replay costs a few passes over N: leave out what takes minutes
    if sum(n * n for n in orders) * case["blocks"] * case["k"] > 1.5e9:
        return None
    G, Gw, cfg = [], [], []
    for ch, n in zip(chains, orders):
        p = _Plain(ch, _configuration(ch, n, seed), 0.5 * (1.0 - case["p_flip"]), case["p_flip"],
                   case["precision"] != "f64")
        p.refresh()
        g = gw = 0.0
        for _ in range(case["blocks"]):
            p.block(case["k"])
            p.refresh()
            g = g + p.greens_function() / case["blocks"]
            if case["freqs"]:
                gw = gw + p.greens_function_matsubara(case["freqs"]) / case["blocks"]
        G.append(g.ravel())
        Gw.append(np.ravel(gw))
        cfg.append(p)
    out = dict(G=np.concatenate(G), tau=_padded([p.tau for p in cfg], [c.capacity for c in chains]),
               site=None, s=None, birth=None, order=None)
    if case["freqs"]:
        out["Gw"] = np.concatenate(Gw)
    return out
