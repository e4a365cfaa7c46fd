"""Performance cases of the initiator-FCIQMC library: what they run and on what.

A case is a dict of plain numbers and texts.  `prepare` makes what a program
holds before the call (a run grown to its walker number, a checkpoint, a list
of requests), `run` is one pass through the public entry points, `work` the
bytes and binary64 operations a pass cannot do without, and `exact` the same
outputs from plain numpy where that is possible.

A pass of kind "steps" advances a run by a block of iterations and ends as
such a block ends in practice: the statistics rows of the block are read and
the walker list is written to the host (into pinned buffers that a program
keeps between checkpoints).
"""
import math

import numpy as np
import torch

import paper_2006_14956_gb300 as fq

# growth per iteration while a run fills up (S = GROWTH / tau); the shift then
# takes over with the full damping every two iterations
GROWTH = 0.05
ROW = ("iteration", "nw", "shift", "e_num", "e_den", "ndet", "attempts", "spawns", "rejected", "annihilated", "vary",
       "trial_num", "trial_den", "x_overlap", "x_var_num", "x_pt2")

HUBBARD = dict(system="hubbard", lx=4, ly=4, U=4.0, n_a=3.0, walkers=1e5, iters=40, settle=100)
ABINITIO = dict(system="abinitio", norb=24, na=6, nb=6, n_a=3.0, walkers=1e6, iters=20, settle=60, p_single=0.1,
                c_min=1.0, generator=0, semi=0, trial=0, adaptive=0, replicas=1)


def listed():
    return [
        # the smallest calls: twenty iterations of an 8-site ring (4900 determinants), where launches and latency count
        dict(HUBBARD, name="ring8", kind="steps", lx=8, ly=1, n_a=0.0, walkers=1e4, iters=20),
        # one lattice run of the batched set's kind, alone
        dict(HUBBARD, name="hubbard44", kind="steps"),
        # the trial-wave-function energy on a 4x5 lattice
        dict(HUBBARD, name="hubbard45-trial", kind="steps", lx=4, ly=5, U=8.0, walkers=3e5, trial=200),
        # the 24-orbital system (6 + 6 electrons, uniform generator, 1e6 walkers)
        dict(ABINITIO, name="orb24", kind="steps"),
        # its replica pair (variational energy and PT2)
        dict(ABINITIO, name="orb24-pair", kind="steps", walkers=2e5, replicas=2, iters=20),
        # heat-bath doubles: 40 orbitals, 10 + 10 electrons
        dict(ABINITIO, name="orb40-heatbath", kind="steps", norb=40, na=10, nb=10, walkers=2e6, generator=1),
        # odd electron numbers, another rounding threshold, adaptive shift
        dict(ABINITIO, name="orb31-adaptive", kind="steps", norb=31, na=9, nb=6, walkers=3e5, c_min=0.5, adaptive=1),
        # the 50-orbital system (10 + 10 electrons, deterministic space of 1e4) at 1e7 walkers ...
        dict(ABINITIO, name="orb50-1e7", kind="steps", norb=50, na=10, nb=10, walkers=1e7, semi=10000, iters=20),
        # ... and at 1e8, the headline size
        dict(ABINITIO, name="orb50-1e8", kind="steps", norb=50, na=10, nb=10, walkers=1e8, semi=10000, iters=20,
             settle=30),
        # 64 uneven lattice runs (1e4 .. 1e6 walkers) in one batch
        dict(name="batch64", kind="batch", runs=64, lo=4.0, hi=6.0, iters=40),
        # a stream of mixed small requests through the server, from admission to retirement
        dict(name="serving", kind="serving", requests=8, lo=4.0, hi=5.5, iters=800),
        # a checkpoint of 3e6 determinants loaded into a new run (H_ii of each computed) and written back sorted
        dict(name="restart", kind="restart", norb=50, na=10, nb=10, dets=3000000),
    ]


def draw(rng):
    def logu(lo, hi):
        return 10.0 ** rng.uniform(math.log10(lo), math.log10(hi))

    x = rng.random()
    if x < 0.3:
        ring = rng.random() < 0.4
        lx, ly = (rng.choice([8, 10, 12, 14, 16, 18]), 1) if ring else rng.choice([(3, 4), (4, 4), (4, 5), (3, 6), (4, 3)])
        # walkers beyond a few per determinant are no use: the smallest lattices stay small
        top = min(1e6, 4.0 * _fci(lx * ly, (lx * ly) // 2, (lx * ly) // 2))
        c = dict(HUBBARD, kind="steps", lx=lx, ly=ly, U=float(rng.randint(1, 8)), n_a=rng.choice([0.0, 3.0, 3.0]),
                 walkers=round(logu(5e3, top)), iters=rng.randint(10, 60))
        if rng.random() < 0.2:
            c["trial"] = rng.randint(20, 200)
        return c
    if x < 0.75:
        norb = rng.randint(16, 50)
        na = rng.randint(4, min(10, norb // 2))
        nb = max(2, na - rng.choice([0, 0, 0, 1, 2, 3]))
        c = dict(ABINITIO, kind="steps", norb=norb, na=na, nb=nb, n_a=rng.choice([0.0, 3.0, 3.0, 3.0]),
                 walkers=round(logu(1e4, min(3e7, 0.2 * _fci(norb, na, nb)))), iters=rng.randint(10, 30),
                 p_single=rng.choice([0.05, 0.1, 0.1, 0.3]))
        opt = rng.choice(["", "", "heatbath", "semi", "semi", "pair", "adaptive", "c_min"])
        if opt == "heatbath":
            c["generator"] = 1
        elif opt == "semi":
            c["semi"] = rng.randint(50, 10000)
        elif opt == "pair":
            c.update(replicas=2, walkers=min(c["walkers"], 1000003))
        elif opt == "adaptive":
            c.update(adaptive=1, walkers=min(c["walkers"], 1000003))
        elif opt == "c_min":
            c["c_min"] = rng.choice([0.3, 0.5, 2.0])
        return c
    if x < 0.85:
        lo = rng.uniform(3.7, 4.5)
        return dict(kind="batch", runs=rng.randint(2, 64), lo=lo, hi=lo + rng.uniform(0.2, 1.5), iters=rng.randint(10, 40))
    if x < 0.92:
        lo = rng.uniform(3.7, 4.5)
        return dict(kind="serving", requests=rng.randint(2, 10), lo=lo, hi=lo + rng.uniform(0.2, 1.0),
                    iters=rng.randint(300, 800))
    norb = rng.randint(16, 50)
    na = rng.randint(4, 10)
    return dict(kind="restart", norb=norb, na=min(na, norb // 2), nb=min(rng.randint(4, 10), norb // 2),
                dets=round(logu(3e3, 5e6)))


# ---------------------------------------------------------------- systems
def _fci(norb, na, nb):
    return float(math.comb(norb, na)) * math.comb(norb, nb)


def _pair(i, j):
    return max(i, j) * (max(i, j) + 1) // 2 + min(i, j)


def _integrals(norb, seed):
    """Synthetic integrals with 8-fold symmetry: h diagonal in [-2, 2] Eh, off-diagonal N(0, 0.05^2); (pq|rs) from
    4 norb Cholesky vectors N(0, 0.1^2) with 0.5 added on their diagonals."""
    rng = np.random.Generator(np.random.Philox(seed))
    h = np.zeros((norb, norb))
    iu = np.triu_indices(norb, 1)
    h[iu] = rng.normal(0.0, 0.05, size=iu[0].size)
    h = h + h.T
    h[np.diag_indices(norb)] = np.linspace(-2.0, 2.0, norb)
    p, q = np.tril_indices(norb)
    chol = rng.normal(0.0, 0.1, size=(4 * norb, p.size)) + 0.5 * (p == q)
    V = chol.T @ chol
    return h, np.ascontiguousarray(V[np.tril_indices(p.size)])


def _dense(norb, eri):
    """(pq|rs) as a four-index array."""
    pq = np.array([[_pair(p, q) for q in range(norb)] for p in range(norb)])
    a, b = pq.reshape(-1, 1), pq.reshape(1, -1)
    hi, lo = np.maximum(a, b), np.minimum(a, b)
    return eri[hi * (hi + 1) // 2 + lo].reshape(norb, norb, norb, norb)


def _couplings(h, g, na, nb):
    """sum_j |H_ref,j| over the singles and doubles of the determinant that fills the lowest orbitals."""
    n = h.shape[0]
    total = 0.0
    for o, other in ((na, nb), (nb, na)):
        k = np.arange(n)
        coul = g[:, :, k, k][:, :, :o].sum(-1) + g[:, :, k, k][:, :, :other].sum(-1)
        exch = np.einsum("akki->aik", g)[:, :, :o].sum(-1)
        total += np.abs(h + coul - exch)[o:, :o].sum()
        d = g[o:, :o, o:, :o]  # (ai|bj)
        total += np.abs(d - d.transpose(0, 3, 2, 1)).sum() / 4.0
    return total + np.abs(g[na:, :na, nb:, :nb]).sum()


def _system(case, seed):
    """(system, tau)"""
    if case["system"] == "hubbard":
        n = case["lx"] * case["ly"]
        square = case["ly"] > 1
        return dict(kind="hubbard", lx=case["lx"], ly=case["ly"], periodic_x=True, periodic_y=square, t=1.0,
                    U=case["U"], n_alpha=n // 2, n_beta=n // 2), 0.005 if square else 0.01
    h, eri = _integrals(case["norb"], seed)
    s = 0.5 / _couplings(h, _dense(case["norb"], eri), case["na"], case["nb"])
    e = math.floor(math.log10(s)) - 1
    return dict(kind="abinitio", norb=case["norb"], n_alpha=case["na"], n_beta=case["nb"], h1=h, eri=eri,
                ecore=0.0), math.floor(s / 10.0 ** e) * 10.0 ** e


def _params(case, tau, seed):
    # the shift takes hold a few iterations late: the walker number settles at about 1.3 times the target
    n0 = min(1e5, max(20.0, case["walkers"] / 1000.0))
    p = dict(tau=tau, target_walkers=case["walkers"] / 1.5, initial_walkers=float(round(n0)), initial_shift=GROWTH / tau,
             initiator_threshold=case["n_a"], shift_damping=1.0, shift_interval=2, seed=1 + seed,
             max_dets=int(1.3 * case["walkers"]) if case["walkers"] > 8e6 else 0)
    if case["system"] == "abinitio":
        p.update(p_single=case["p_single"], c_min=case["c_min"], generator=case["generator"], replicas=case["replicas"],
                 adaptive_shift=case["adaptive"], semistoch_size=case["semi"], semistoch_start=4)
    p.update(trial_size=case.get("trial", 0), trial_start=4)
    return p


def _grow(step, runs, settle):
    """Steps until the shift of every run varies, then `settle` iterations more."""
    for _ in range(400):
        step(4)
        if all(fq.fciqmc_export_shift(h)["vary"] for h in runs):
            break
    step(settle)


def _cap(case):
    """Room for the walker list of a run."""
    n, dim = case["walkers"] / min(1.0, case.get("c_min", 1.0)), \
        _fci(case["lx"] * case["ly"], *[case["lx"] * case["ly"] // 2] * 2) if case["system"] == "hubbard" else \
        _fci(case["norb"], case["na"], case["nb"])
    return int(min(1.3 * n + 5000, dim))


def _host_buffers(n):
    pinned = lambda t: torch.empty(n, dtype=t, pin_memory=True).zero_().numpy()  # noqa: E731
    return dict(alpha=pinned(torch.int64).view(np.uint64), beta=pinned(torch.int64).view(np.uint64),
                c=pinned(torch.float64), hdiag=pinned(torch.float64), flags=pinned(torch.int32))


def _random_dets(norb, na, nb, n, seed):
    """n (or all, if fewer) distinct determinants, low orbitals preferred, with amplitudes; key order shuffled."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    words = []
    for ne in (na, nb):
        w = torch.empty(n, dtype=torch.int64, device="cuda")
        for a in range(0, n, 1 << 20):
            m = min(n, a + (1 << 20)) - a
            score = torch.rand(m, norb, generator=g, device="cuda") + 0.5 / norb * torch.arange(norb, device="cuda")
            w[a:a + m] = (1 << score.topk(ne, largest=False).indices).sum(1)
        words.append(w)
    key = torch.unique(torch.stack(words, 1), dim=0)
    key = key[torch.randperm(key.shape[0], generator=g, device="cuda")].cpu().numpy().view(np.uint64)
    c = np.random.Generator(np.random.Philox(seed)).normal(0.0, 2.0, key.shape[0])
    return np.ascontiguousarray(key[:, 0]), np.ascontiguousarray(key[:, 1]), c


# ---------------------------------------------------------------- a pass
def prepare(case, seed):
    if case["kind"] == "steps":
        sysd, tau = _system(case, seed)
        h = fq.fciqmc_create(sysd, _params(case, tau, seed))
        runs = [h] + ([fq.fciqmc_replica(h, 1)] if case.get("replicas", 1) == 2 else [])
        _grow(lambda n: fq.fciqmc_step(h, n), runs, case["settle"])
        out = [_host_buffers(_cap(case)) for r in runs]
        return dict(kind="steps", h=h, runs=runs, iters=case["iters"], out=out)
    if case["kind"] == "batch":
        hs, out = [], []
        for k in range(case["runs"]):
            lx, ly = [(3, 4), (4, 4), (4, 5)][k % 3]
            w = round(10.0 ** (case["lo"] + (case["hi"] - case["lo"]) * k / max(1, case["runs"] - 1)))
            c = dict(HUBBARD, lx=lx, ly=ly, U=[2.0, 4.0, 8.0][(k // 3) % 3], walkers=w)
            sysd, tau = _system(c, seed)
            hs.append(fq.fciqmc_create(sysd, _params(c, tau, 1000 * seed + k)))
            out.append(_host_buffers(_cap(c)))
        _grow(lambda n: fq.fciqmc_step_batch(hs, n), hs, 60)
        return dict(kind="batch", hs=hs, iters=case["iters"], out=out)
    if case["kind"] == "serving":
        reqs = []
        for k in range(case["requests"]):
            w = round(10.0 ** (case["lo"] + (case["hi"] - case["lo"]) * k / max(1, case["requests"] - 1)))
            if k % 3 == 2:
                norb = 16 + (seed + 7 * k) % 25
                ne = 4 + (seed + k) % 5
                h, eri = _integrals(norb, 1000 * seed + k)
                sysd = dict(kind="abinitio", norb=norb, n_alpha=ne, n_beta=ne, h1=h, eri=eri, ecore=0.0)
                prm = dict(tau=0.0, initiator_threshold=3.0, p_single=0.1)
            else:
                c = dict(HUBBARD, lx=[8, 10, 12, 14, 16, 18][(seed + k) % 6] if k % 3 else [3, 4, 4][k // 3 % 3],
                         ly=1 if k % 3 else [4, 4, 5][k // 3 % 3], U=float(1 + (seed + k) % 8))
                sysd = _system(c, seed)[0]
                prm = dict(tau=0.0, initiator_threshold=3.0)
            prm.update(target_walkers=float(w), initial_walkers=1000.0, shift_damping=0.5, shift_interval=5,
                       seed=1000 * seed + k + 1)
            reqs.append((sysd, prm))
        return dict(kind="serving", reqs=reqs, iters=case["iters"])
    a, b, c = _random_dets(case["norb"], case["na"], case["nb"], case["dets"], seed)
    sysd, tau = _system(dict(case, system="abinitio"), seed)
    prm = dict(tau=tau, target_walkers=float(case["dets"]), initiator_threshold=3.0, seed=1 + seed)
    pin = lambda x: torch.from_numpy(x.view(np.int64)).pin_memory().numpy()  # noqa: E731
    return dict(kind="restart", sysd=sysd, prm=prm, a=pin(a).view(np.uint64), b=pin(b).view(np.uint64),
                c=pin(c).view(np.float64), out=_host_buffers(case["dets"] + 1))


def _rows(h, n):
    return fq.fciqmc_iter_stats_get(h, fq.fciqmc_iter_stats_count(h) - n, n)


def _list(h, out):
    """The walker list in the program's own buffers, which come back whole."""
    if fq.fciqmc_export_state(h, out)["c"].ctypes.data != out["c"].ctypes.data:
        raise RuntimeError("the walker list is larger than the buffers kept for it")
    return dict(out, alpha=out["alpha"].view(np.int64), beta=out["beta"].view(np.int64))


def run(state):
    if state["kind"] == "steps":
        fq.fciqmc_step(state["h"], state["iters"])
        return dict(rows=_rows(state["h"], state["iters"]), lists=[_list(h, o) for h, o in zip(state["runs"], state["out"])])
    if state["kind"] == "batch":
        hs, n = state["hs"], state["iters"]
        fq.fciqmc_step_batch(hs, n)
        rows = [_rows(h, n) for h in hs]
        lists = [_list(h, o) for h, o in zip(hs, state["out"])]
        return dict(rows={k: np.stack([r[k] for r in rows]) for k in ROW},
                    lists={k: np.concatenate([x[k] for x in lists]) for k in lists[0]})
    if state["kind"] == "serving":
        srv = fq.fciqmc_server_create(64 << 30, 64)
        ids = [fq.fciqmc_server_submit(srv, s, p, 1e-3, state["iters"]) for s, p in state["reqs"]]
        while fq.fciqmc_server_tick(srv, 50):
            pass
        got = [fq.fciqmc_server_poll(srv, i) for i in ids]
        fq.fciqmc_server_destroy(srv)
        return {k: np.array([g[k] for g in got]) for k in ("state", "error", "iterations", "energy", "sigma", "shift",
                                                          "attempts", "tau", "estimator")}
    h = fq.fciqmc_create(state["sysd"], state["prm"])
    fq.fciqmc_import_state(h, state["a"], state["b"], state["c"], 0, 0.0)
    out = dict(list=_list(h, state["out"]), couplings=fq.fciqmc_ref_offdiag_sum(h))
    fq.fciqmc_destroy(h)
    return out


# ---------------------------------------------------------------- what a pass needs
def work(case):
    """An iteration reads and writes the walker list once (key, C, H_ii, flag: 33 bytes each way; spawned walkers need not
    leave the chip) and spends three binary64 operations on a determinant's death and three on each attempt's weight;
    a restart moves the checkpoint (24 bytes in, 36 out) and adds up n (n + 1) / 2 integrals per determinant."""
    if case["kind"] == "restart":
        n = min(float(case["dets"]), _fci(case["norb"], case["na"], case["nb"]))
        e = case["na"] + case["nb"]
        return dict(bytes=60.0 * n, flops=n * e * (e + 1) / 2)
    if case["kind"] == "steps":
        dim = _fci(case["lx"] * case["ly"], *[case["lx"] * case["ly"] // 2] * 2) if case["system"] == "hubbard" else \
            _fci(case["norb"], case["na"], case["nb"])
        sizes = [(case["walkers"] / case.get("c_min", 1.0), dim)] * case.get("replicas", 1)
    elif case["kind"] == "batch":
        k = max(1, case["runs"] - 1)
        sizes = [(10.0 ** (case["lo"] + (case["hi"] - case["lo"]) * i / k), [853776.0, 165636900.0, 34134779536.0][i % 3])
                 for i in range(case["runs"])]
    else:
        k = max(1, case["requests"] - 1)
        sizes = [(10.0 ** (case["lo"] + (case["hi"] - case["lo"]) * i / k), 1e6) for i in range(case["requests"])]
    it = case["iters"]
    return dict(bytes=it * sum(66.0 * min(w, d) for w, d in sizes), flops=it * sum(3.0 * min(w, d) + 3.0 * w for w, d in sizes))


# ---------------------------------------------------------------- in plain numpy
U64 = np.uint64


def _mul128(a, m):
    """High and low words of a * m for 64-bit a (array) and m (int)."""
    m0, m1, lo32 = U64(m & 0xFFFFFFFF), U64(m >> 32), U64(0xFFFFFFFF)
    a0, a1, s = a & lo32, a >> U64(32), U64(32)
    mid = a1 * m0 + ((a0 * m0) >> s)
    mid2 = a0 * m1 + (mid & lo32)
    return a1 * m1 + (mid >> s) + (mid2 >> s), a * U64(m)


def _philox(a, b, it, tag, seed):
    """Philox4x64-10 words of the counters (a, b, it, tag) with key (seed, 0)."""
    c0, c1, c2, c3 = a.copy(), b.copy(), np.full(a.shape, it, U64), np.broadcast_to(np.asarray(tag, U64), a.shape).copy()
    k0, k1 = seed, 0
    for _ in range(10):
        h0, l0 = _mul128(c0, 0xD2E7470EE14C6C93)
        h1, l1 = _mul128(c2, 0xCA5A826395121157)
        c0, c1, c2, c3 = h1 ^ c1 ^ U64(k0), l1, h0 ^ c3 ^ U64(k1), l0
        k0 = (k0 + 0x9E3779B97F4A7C15) & (2 ** 64 - 1)
        k1 = (k1 + 0xBB67AE8584CAA73B) & (2 ** 64 - 1)
    return c0, c1, c2, c3


def _round(v, w):
    """Stochastic rounding at 1 of |v| < 1 with the word w."""
    u = (w >> U64(11)).astype(np.float64) * 2.0 ** -53
    return np.where((v == 0) | (np.abs(v) >= 1.0), v, np.where(u < np.abs(v), np.copysign(1.0, v), 0.0))


def _floor32(x):
    """floor(|x| 2^32) of each as Python can add them exactly."""
    return int(np.floor(np.abs(x) * 2.0 ** 32).astype(object).sum()) if x.size else 0


class _Lattice:
    """The same projection of a Hubbard lattice, written down in numpy: keys, amplitudes and rows."""

    def __init__(self, sysd, prm):
        lx, ly = sysd["lx"], sysd["ly"]
        self.n, self.z, self.p, self.U = lx * ly, 4 if ly > 1 else 2, prm, sysd["U"]
        self.sysd = sysd
        nb = [[y * lx + (x - 1) % lx, y * lx + (x + 1) % lx, ((y - 1) % ly) * lx + x, ((y + 1) % ly) * lx + x]
              for y in range(ly) for x in range(lx)]
        self.nbr = np.array(nb)[:, :self.z]
        self.ref = [sum(1 << (x + lx * y) for y in range(ly) for x in range(lx) if (x + y) % 2 == s) for s in (0, 1)]
        self.a, self.b = np.array([self.ref[0]], U64), np.array([self.ref[1]], U64)
        self.c = np.array([prm["initial_walkers"]])
        self.S, self.vary, self.cnt, self.last, self.it, self.rows = prm["initial_shift"], 0, 0, 0, 0, []

    def step(self):
        p, n = self.p, self.n
        one = U64(1)
        bits = lambda w: (w[:, None] >> np.arange(n, dtype=U64)) & one  # noqa: E731
        a, b, c = self.a, self.b, self.c
        # spawning
        nat = np.ceil(np.abs(c)).astype(np.int64)
        i = np.repeat(np.arange(c.size), nat)
        k = np.arange(i.size) - np.repeat(np.cumsum(nat) - nat, nat)
        pa, pb = a[i], b[i]
        _, w1, w2, w3 = _philox(pa, pb, self.it, (k.astype(U64) << U64(8)) | one, p["seed"])
        ne = self.sysd["n_alpha"] + self.sysd["n_beta"]
        e = _mul128(w1, ne)[0].astype(np.int64)
        sp = e >= self.sysd["n_alpha"]
        x = np.where(sp, pb, pa)
        occ = bits(x)
        rank = e - np.where(sp, self.sysd["n_alpha"], 0)
        o = (np.cumsum(occ, 1).astype(np.int64) == (rank + 1)[:, None]).argmax(1)
        q = self.nbr[o, _mul128(w2, self.z)[0].astype(np.int64)]
        ok = occ[np.arange(o.size), q] == 0
        lo, hi = np.minimum(o, q), np.maximum(o, q)
        site = np.arange(n)
        par = ((occ == 1) & (site > lo[:, None]) & (site < hi[:, None])).sum(1) & 1
        H = np.where(par == 1, self.sysd["t"], -self.sysd["t"])
        w = _round(-(H * ((p["tau"] / (1.0 / (float(ne) * self.z))) * (c[i] / nat[i]))), w3)
        ok &= w != 0
        y = x ^ (one << o.astype(U64)) ^ (one << q.astype(U64))
        init = (np.abs(c) > p["initiator_threshold"]) | ((a == U64(self.ref[0])) & (b == U64(self.ref[1])))
        ta, tb, w, si = np.where(sp, pa, y)[ok], np.where(sp, y, pb)[ok], w[ok], init[i][ok]
        # death
        d = self.U * np.bitwise_count(a & b).astype(np.float64)
        cp = _round(c * (1.0 - p["tau"] * (d - self.S)), _philox(a, b, self.it, 2, p["seed"])[0])
        # annihilation: all keys on one list, walkers first
        keys, own = np.unique(np.stack([np.concatenate([a, ta]), np.concatenate([b, tb])], 1), axis=0, return_inverse=True)
        own = own.reshape(-1)
        ka, kb = np.ascontiguousarray(keys[:, 0]), np.ascontiguousarray(keys[:, 1])
        base, occd = np.zeros(ka.size), np.zeros(ka.size, bool)
        base[own[:a.size]], occd[own[:a.size]] = cp, c != 0
        t = own[a.size:]
        acc = si | occd[t]
        s, hit = np.zeros(ka.size), np.zeros(ka.size, bool)
        np.add.at(s, t[acc], w[acc])
        hit[t[acc]] = True
        v = base + s
        ann = _floor32(w[acc]) + _floor32(base[hit]) - _floor32(v[hit])
        r = hit & (v != 0) & (np.abs(v) < 1.0)
        v[r] = _round(v[r], _philox(ka[r], kb[r], self.it, 3, p["seed"])[0])
        isref = (ka == U64(self.ref[0])) & (kb == U64(self.ref[1]))
        keep = (v != 0) | isref
        self.a, self.b, self.c = ka[keep], kb[keep], v[keep]
        # the projected energy: hops away from the reference
        num = 0.0
        for sgn, (x0, here, there) in enumerate(((self.ref[0], self.a, self.b == U64(self.ref[1])),
                                                 (self.ref[1], self.b, self.a == U64(self.ref[0])))):
            for o in range(n):
                if not (x0 >> o) & 1:
                    continue
                for q in sorted(set(self.nbr[o].tolist())):
                    if (x0 >> q) & 1:
                        continue
                    f = there & (here == U64(x0 ^ (1 << o) ^ (1 << q)))
                    m = bin(x0 >> (min(o, q) + 1) & ((1 << (abs(o - q) - 1)) - 1)).count("1") if abs(o - q) > 1 else 0
                    num += (self.sysd["t"] if m & 1 else -self.sysd["t"]) * self.c[f].sum()
        W = _floor32(self.c)
        nw = W * 2.0 ** -32
        if not self.vary:
            if nw >= p["target_walkers"]:
                self.vary, self.last, self.cnt = 1, W, 0
        else:
            self.cnt += 1
            if self.cnt == p["shift_interval"]:
                self.S -= p["shift_damping"] / (p["shift_interval"] * p["tau"]) * math.log(W / self.last)
                self.last, self.cnt = W, 0
        self.rows.append(dict(iteration=self.it, nw=nw, shift=self.S, e_num=num, e_den=float(v[isref][0]), ndet=self.c.size,
                              attempts=int(nat.sum()), spawns=int(w.size), rejected=int((~acc).sum()),
                              annihilated=ann * 2.0 ** -32, vary=self.vary))
        self.it += 1


def _padded(x, n):
    return np.concatenate([x, np.zeros(n - x.size, x.dtype)])


def exact(case, seed):
    if case["kind"] == "steps":
        # a lattice run of up to about 2e4 walkers without estimators can be followed draw by draw
        if case["system"] != "hubbard" or case.get("trial", 0) or case["walkers"] > 2e4:
            return None
        sysd, tau = _system(case, seed)
        r = _Lattice(sysd, _params(case, tau, seed))
        for _ in range(400):
            for _ in range(4):
                r.step()
            if r.vary:
                break
        for _ in range(case["settle"] + case["iters"]):
            r.step()
        rows = r.rows[-case["iters"]:]
        pad = lambda x: _padded(x, _cap(case))  # noqa: E731
        return dict(rows={k: np.array([x[k] for x in rows]) if k in rows[0] else None for k in ROW},
                    lists=[dict(alpha=pad(r.a.view(np.int64)), beta=pad(r.b.view(np.int64)), c=pad(r.c),
                                hdiag=pad(r.U * np.bitwise_count(r.a & r.b).astype(np.float64)), flags=None)])
    if case["kind"] != "restart":
        return None
    a, b, c = _random_dets(case["norb"], case["na"], case["nb"], case["dets"], seed)
    sysd, _ = _system(dict(case, system="abinitio"), seed)
    n, h, g = case["norb"], sysd["h1"], _dense(case["norb"], sysd["eri"])
    ra, rb = (1 << case["na"]) - 1, (1 << case["nb"]) - 1
    if not ((a == U64(ra)) & (b == U64(rb))).any():
        a, b, c = np.append(a, U64(ra)), np.append(b, U64(rb)), np.append(c, 0.0)
    order = np.lexsort((b, a))
    a, b, c = a[order], b[order], c[order]
    d = np.arange(n)
    J, K = torch.from_numpy(g[d[:, None], d[:, None], d, d]).cuda(), torch.from_numpy(g[d[:, None], d, d, d[:, None]]).cuda()
    hp = torch.from_numpy(np.diag(h).copy()).cuda()

    def energies(wa, wb):
        sh = torch.arange(n, device="cuda")
        na, nb = (((torch.from_numpy(w.view(np.int64)).cuda()[:, None] >> sh) & 1).double() for w in (wa, wb))
        both = na + nb
        return (both @ hp + 0.5 * ((both @ J) * both).sum(1) - 0.5 * ((na @ K) * na).sum(1) - 0.5 * ((nb @ K) * nb).sum(1))

    e0 = energies(np.array([ra], U64), np.array([rb], U64))
    hd = torch.cat([energies(a[k:k + (1 << 20)], b[k:k + (1 << 20)]) - e0 for k in range(0, a.size, 1 << 20)]).cpu().numpy()
    pad = lambda x: _padded(x, case["dets"] + 1)  # noqa: E731
    return dict(list=dict(alpha=pad(a.view(np.int64)), beta=pad(b.view(np.int64)), c=pad(c), hdiag=pad(hd), flags=None),
                couplings=float(_couplings(h, g, case["na"], case["nb"])))
