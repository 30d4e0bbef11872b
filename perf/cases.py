"""Timed workloads of the FCIQMC step: what a program that uses this package
has it do, through its public objects, from the smallest runs to the largest
that fit a card three times over.

A program equilibrates a run (or a batch of runs), then steps it in chunks and
reads the recorded time series and the amplitudes it follows.  `prepare` does
the first part and `run` one chunk of the second.  Every run here is
population-controlled at its target, so the work of a chunk stays what it is
however many chunks went before.

A case is a dict of plain values:
  form      "run" (one run), "batch" (independent runs stepped together),
            "replicas" (runs with overlaps after every step) or "spectral"
            (Gram-Schmidt states)
  kind      1 ring, 2 rectangular lattice, 3 ring in momentum space
  Lx, Ly    lattice; N bosons; u interaction (hopping 1)
  mode      "INT", "REAL64" or "REAL32" (fq.MODE_*)
  target    walkers; dt time step; equil untimed steps; steps of one pass
  threshold, t_rel, early, sort   options of the run, where they are not 1, 1,
            late compression and the default annihilation arm
  runs      number of runs of a batch, replicas or states
  g2        largest distance of the density correlator of replicas (-1: none)
"""
import math

import numpy as np

import paper_2601_19505_gb300 as fq

KIND_1D, KIND_2D, KIND_MOM = 1, 2, 3
EXPORT_MOST = 20000  # largest target whose whole vector a pass reads back
TRACKED = 16384      # amplitudes a pass reads from a larger vector


def _case(name, form, kind, Lx, Ly, N, u, mode, target, dt, equil, steps, **more):
    c = dict(name=name, form=form, kind=kind, Lx=Lx, Ly=Ly, N=N, u=u, mode=mode, target=target,
             dt=dt, equil=equil, steps=steps)
    c.update(more)
    return c


def listed():
    return [
        # a test or teaching calculation: integer walkers on six sites, where
        # each step is a few hundred configurations and latency is everything
        _case("ring6-int-1e3", "run", KIND_1D, 6, 1, 6, 6.0, "INT", 1e3, 1e-3, 1500, 400),
        # the common small calculation of the method's tutorials: 12 sites
        _case("ring12-fp64-1e4", "run", KIND_1D, 12, 1, 12, 6.0, "REAL64", 1e4, 1e-3, 500, 200),
        # a parameter scan's single run: half-full chip, 39-bit addresses
        _case("ring20-fp64-1e5", "run", KIND_1D, 20, 1, 20, 2.0, "REAL64", 1e5, 1e-3, 600, 100),
        # a production run on a ring: 1e7 walkers
        _case("ring20-fp64-1e7", "run", KIND_1D, 20, 1, 20, 2.0, "REAL64", 1e7, 1e-3, 600, 16),
        # one bit more than a machine word, single precision, restarted from a
        # double-precision run's vector
        _case("ring33-fp32-1e6", "run", KIND_1D, 33, 1, 33, 4.0, "REAL32", 1e6, 1e-3, 400, 16),
        # the 8 x 8 lattice (127-bit addresses) in both precisions; the large
        # one is the headline workload at the size that fits three times
        _case("square8-fp32-1e6", "run", KIND_2D, 8, 8, 64, 8.0, "REAL32", 1e6, 2e-4, 400, 16),
        _case("square8-fp64-1e8", "run", KIND_2D, 8, 8, 64, 8.0, "REAL64", 1e8, 2e-4, 260, 8),
        # momentum space: a strongly interacting small ring whose sign problem
        # annihilation overcomes, and a weakly interacting large one
        _case("momentum10-fp64-1e4", "run", KIND_MOM, 10, 1, 10, 6.0, "REAL64", 1e4, 1e-3, 1000,
              100),
        _case("momentum32-fp64-1e6", "run", KIND_MOM, 32, 1, 32, 0.5, "REAL64", 1e6, 5e-4, 1000,
              16),
        # 64 rings of uneven size and interaction stepped as one batch
        _case("batch64-fp64", "batch", KIND_1D, 0, 1, 0, 0.0, "REAL64", 1e6, 1e-3, 800, 32,
              runs=64),
        # replicas for unbiased expectation values, with density correlators
        _case("replicas3-g2-3e5", "replicas", KIND_1D, 20, 1, 20, 2.0, "REAL64", 3e5, 1e-3, 500,
              32, runs=3, g2=3),
        # ground and first excited state
        _case("spectral2-1e6", "spectral", KIND_1D, 20, 1, 20, 2.0, "REAL64", 1e6, 1e-3, 500, 16,
              runs=2),
    ]


def _log_uniform(rng, lo, hi):
    return float(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    x = rng.random()
    form = "run" if x < 0.76 else "batch" if x < 0.84 else "replicas" if x < 0.92 else "spectral"
    u = round(_log_uniform(rng, 1.0, 10.0), 3)
    if form == "batch":
        top = _log_uniform(rng, 2e4, 1e6)
        return dict(form=form, kind=KIND_1D, Lx=0, Ly=1, N=0, u=0.0, mode="REAL64", target=top,
                    dt=1e-3, equil=700, steps=rng.randint(8, 32), runs=rng.randint(2, 64),
                    points=rng.randint(2, 1 << 20))
    if form != "run":
        M = rng.randint(10, 24)
        c = dict(form=form, kind=KIND_1D, Lx=M, Ly=1, N=M, u=u, mode="REAL64",
                 target=_log_uniform(rng, 1e4, 1e6), dt=1e-3, equil=500, steps=rng.randint(8, 32))
        c["runs"] = rng.randint(2, 3)
        if form == "replicas":
            c["g2"] = rng.randint(-1, 4)
        return c
    kind = rng.choices((KIND_1D, KIND_2D, KIND_MOM), (5, 3, 2))[0]
    if kind == KIND_MOM:
        M = rng.randint(8, 32)
        small = M <= 11
        return dict(form=form, kind=kind, Lx=M, Ly=1, N=M,
                    u=round(rng.uniform(0.25, 4.0 if small else 0.6), 3), mode="REAL64",
                    target=_log_uniform(rng, 1e4, 1e5) if small else _log_uniform(rng, 2e5, 1.5e6),
                    dt=1e-3 if M <= 20 else 5e-4, equil=900, steps=rng.randint(8, 64))
    mode = rng.choices(("REAL64", "REAL32", "INT"), (6, 2, 2))[0]
    if kind == KIND_1D:
        M = rng.randint(6, 56)
        N, Lx, Ly, dt = max(4, round(M * rng.choice((0.5, 1.0, 1.0, 1.25)))), M, 1, 1e-3
    else:
        Lx, Ly = rng.randint(3, 8), rng.randint(3, 8)
        N, dt = max(4, round(Lx * Ly * rng.choice((0.5, 1.0, 1.0)))), 4e-4
    # a small system's spectrum allows a longer time step
    dt = round(max(dt, min(0.01, 1.0 / (0.5 * u * N * (N - 1)))), 5)
    top = 2e6 if mode == "INT" else 1e6 if mode == "REAL32" else 2e7
    top = max(2e3, min(top, 2.0 * math.comb(N + Lx * Ly - 1, N)))
    c = dict(form=form, kind=kind, Lx=Lx, Ly=Ly, N=N, u=u, mode=mode,
             target=_log_uniform(rng, 1e3, top), dt=dt, equil=600, steps=rng.randint(8, 32))
    option = rng.random()
    if mode == "REAL64" and option < 0.15:
        c["threshold"] = round(rng.uniform(0.75, 1.5), 3)
    elif mode == "REAL64" and option < 0.3:
        c["t_rel"] = round(rng.uniform(0.5, 3.0), 3)
    elif mode == "REAL64" and option < 0.4:
        c["early"] = True
    elif option > 0.92:
        c["sort"] = True
    return c


# ---------------------------------------------------------------------------
# inputs

_MODES = {"INT": fq.MODE_INT, "REAL64": fq.MODE_REAL64, "REAL32": fq.MODE_REAL32}


def _members(case):
    """(Lx, Ly, N, u, target) of every run of the case."""
    if case["form"] != "batch":
        return [(case["Lx"], case["Ly"], case["N"], case["u"], case["target"])] * case.get("runs", 1)
    n = case["runs"]
    rng = np.random.default_rng(case.get("points", 1))
    M = rng.integers(10, 31, size=n)
    U = rng.uniform(1.0, 10.0, size=n)
    Nt = 10.0 ** rng.uniform(4.0, math.log10(case["target"]), size=n)
    return [(int(M[i]), 1, int(M[i]), float(U[i]), float(Nt[i])) for i in range(n)]


def _params(case, target, seed, run_id, mode):
    return fq.default_params(
        dt=case["dt"], target=target, seed=seed + 1, run_id=run_id, mode=_MODES[mode],
        threshold=case.get("threshold", 1.0), t_rel=case.get("t_rel", 1.0),
        compression=1 if case.get("early") else 0, annihilation=1 if case.get("sort") else 0)


def _weight(target):
    return max(10.0, float(math.floor(target / 1000.0)))


def _encode(occ):
    """Addresses (lo, hi) of occupation vectors [n, M]: boson b, in ascending
    mode order, sits at bit b + its mode."""
    n, M = occ.shape
    N = int(occ[0].sum())
    modes = np.repeat(np.tile(np.arange(M), n), occ.ravel()).reshape(n, N)
    bits = (modes + np.arange(N)).astype(np.uint64)
    one = np.uint64(1)
    lo = np.bitwise_or.reduce(np.where(bits < 64, one << (bits & np.uint64(63)), 0), axis=1)
    hi = np.bitwise_or.reduce(np.where(bits >= 64, one << (bits & np.uint64(63)), 0), axis=1)
    return lo.astype(np.uint64), hi.astype(np.uint64)


def _start(kind, M, N):
    occ = np.full(M, N // M, dtype=np.int64)
    occ[: N % M] += 1
    if kind == KIND_MOM:
        occ[:] = 0
        occ[M // 2 - 1] = N
    return occ


def _neighbours(kind, Lx, Ly):
    s = np.arange(Lx * Ly)
    x, y = s % Lx, s // Lx
    ds = [(x + 1) % Lx + Lx * y, (x + Lx - 1) % Lx + Lx * y]
    if kind == KIND_2D:
        ds += [x + Lx * ((y + 1) % Ly), x + Lx * ((y + Ly - 1) % Ly)]
    return np.stack(ds)


def _tracked(kind, Lx, Ly, N, n, rng):
    """n addresses a few hops (or momentum-conserving pair moves) from the
    start: the configurations whose amplitudes a program follows."""
    M = Lx * Ly
    occ = np.tile(_start(kind, M, N), (n, 1))
    nbr, rows = _neighbours(kind, Lx, Ly), np.arange(n)
    moves = rng.integers(0, 4, size=n)

    def take():  # a random occupied mode of every row, one boson removed
        cum = np.cumsum(occ, axis=1)
        s = (cum > rng.integers(0, cum[:, -1])[:, None]).argmax(axis=1)
        occ[rows, s] -= 1
        return s

    for step in range(3):
        here = moves > step
        old = occ.copy()
        s = take()
        if kind == KIND_MOM:
            q = take()
            r = rng.integers(0, M, size=n)
            occ[rows, r] += 1
            occ[rows, (s + q - r) % M] += 1
        else:
            occ[rows, nbr[rng.integers(0, len(nbr), size=n), s]] += 1
        occ[~here] = old[~here]
    keys = np.zeros(n, dtype=fq.KEY_DTYPE)
    keys["lo"], keys["hi"] = _encode(occ)
    return keys


def prepare(case, seed):
    """Equilibrated runs, their batch, and the addresses the program follows."""
    st = {"case": case, "batch": None}
    kind, mode = case["kind"], case["mode"]
    evolve = "REAL64" if mode == "REAL32" else mode
    form = case["form"]
    runs = []
    for i, (Lx, Ly, N, u, target) in enumerate(_members(case)):
        ham = fq.Hamiltonian(kind, Lx, Ly, N, 1.0, u)
        run = fq.Run(ham, _params(case, target, seed, i, evolve))
        run.seed_default(_weight(target))
        if form == "spectral" and i:  # state i also starts on the i-th neighbour
            start = ham.starting_address()
            run.seed(fq.keys_from_ints([start, ham.column(start)[1][i]]),
                     [_weight(target), _weight(target)], run.stats()["shift"])
        runs.append(run)
    if form == "run":
        run = runs[0]
        run.advance(case["equil"], chunk=case["equil"])
        if mode == "REAL32":  # a single-precision run takes the vector over
            keys, amps = run.export()
            shift = run.stats()["shift"]
            run.close()
            run = fq.Run(ham, _params(case, target, seed, 0, mode))
            start = fq.keys_from_ints([ham.starting_address()])
            run.seed(keys, amps, shift)
            run.set_reference(start, [_weight(target)])
            run.step(2)
            runs = [run]
    else:
        st["batch"] = batch = fq.Batch(runs)
        if form == "spectral":
            batch.set_spectral(case["runs"])
        batch.step(case["equil"])
        batch.sync()
        if form == "replicas":
            batch.set_overlaps(tuple(range(case["g2"] + 1)))
            batch.step(1)
            batch.overlaps()
    for run in runs:
        run.history()
    st["runs"] = runs
    rng = np.random.default_rng(seed)
    st["keys"] = None
    if case["target"] > EXPORT_MOST or form != "run":
        n = TRACKED if form != "batch" else 256
        st["keys"] = [_tracked(kind, m[0], m[1], m[2], n, rng) for m in _members(case)]
    return st


# ---------------------------------------------------------------------------
# one pass: a chunk of steps, the time series, the amplitudes

def _rows(case, lo, hi, amps):
    """A vector in arrays of a fixed length, zeros after its last entry."""
    n = min(math.comb(case["N"] + case["Lx"] * case["Ly"] - 1, case["N"]),
            int(3 * case["target"]))
    out = {"lo": np.zeros(n, np.int64), "hi": np.zeros(n, np.int64), "amps": np.zeros(n)}
    for f, v in (("lo", lo.view(np.int64)), ("hi", hi.view(np.int64)), ("amps", amps)):
        out[f][:len(v)] = v
    return out


def run(st):
    case, runs = st["case"], st["runs"]
    out = {}
    if st["batch"] is None:
        runs[0].step(case["steps"])
    else:
        st["batch"].step(case["steps"])
        if case["form"] == "replicas":
            out["overlaps"] = st["batch"].overlaps(case["steps"])
    rows = np.stack([r.history(case["steps"]) for r in runs])
    for f in rows.dtype.names:
        out[f] = np.ascontiguousarray(rows[f])
    if st["keys"] is None:
        keys, amps = runs[0].export()
        out.update(_rows(case, np.ascontiguousarray(keys["lo"]),
                         np.ascontiguousarray(keys["hi"]), amps))
    else:
        out["amps"] = np.stack([r.lookup(k) for r, k in zip(runs, st["keys"])])
    return out


def work(case):
    """Each step reads every stored entry (address and amplitude) and writes
    the new vector once; a spawn is written and read once.  Overlaps and
    Gram-Schmidt read the vectors again.  About one spawn per walker; a vector
    holds no more entries than the space has addresses."""
    byts = flops = 0.0
    steps = case["steps"]
    amp = 4 if case["mode"] == "REAL32" else 8
    val = 8 if case["mode"] == "REAL64" else 4
    for Lx, Ly, N, u, target in _members(case):
        M = Lx * Ly
        key = 8 if N + M - 1 <= 64 else 16
        walkers = target / case.get("threshold", 1.0)
        entries = min(walkers, float(math.comb(N + M - 1, N)))
        byts += steps * (entries * 2 * (key + amp) + walkers * 2 * (key + val))
        flops += steps * (2 * entries + 3 * walkers)
        if case["form"] == "replicas":
            byts += steps * entries * (key + amp) * (case["runs"] - 1)
            flops += steps * 2 * entries
    if case["form"] == "spectral":
        K = case["runs"]
        pairs = K * (K - 1) // 2
        byts += steps * entries * (key + amp) * (4 * pairs + K - 1)
        flops += steps * 6 * pairs * entries
    if case["target"] > EXPORT_MOST or case["form"] != "run":
        byts += len(_members(case)) * 24.0 * (TRACKED if case["form"] != "batch" else 256)
    else:
        byts += 24.0 * entries
    return {"bytes": byts, "flops": flops}


# ---------------------------------------------------------------------------
# the same in plain numpy, in 64 bits, for small runs

def _splitmix64(z):
    z = z + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _philox(step, stream, h, k0, k1):
    """Philox4x32-10 of counter (step, stream, h_lo, h_hi), words 0..2."""
    mask, s32 = np.uint64(0xFFFFFFFF), np.uint64(32)
    c0 = np.full(h.shape, step, dtype=np.uint64)
    c1 = np.broadcast_to(np.asarray(stream, dtype=np.uint64), h.shape)
    c2, c3 = h & mask, h >> s32
    for r in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c0, np.uint64(0xCD9E8D57) * c2
        c0, c1, c2, c3 = ((p1 >> s32) ^ c1 ^ np.uint64(k0), p1 & mask,
                          (p0 >> s32) ^ c3 ^ np.uint64(k1), p0 & mask)
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1, c2


def _uniform(w0, w1):
    u = ((w0 >> np.uint64(5)) << np.uint64(26)) | (w1 >> np.uint64(6))
    return u.astype(np.float64) * 2.0 ** -53


class _Plain:
    """A run on a real-space lattice: occupations [n, M] and amplitudes [n]."""

    def __init__(self, case, seed):
        self.c = case
        self.M, self.N = case["Lx"] * case["Ly"], case["N"]
        self.nbr = _neighbours(case["kind"], case["Lx"], case["Ly"])
        w = _weight(case["target"])
        self.occ = _start(case["kind"], self.M, self.N)[None, :]
        self.start, self.w = self.occ[0].copy(), w
        self.a = np.array([w])
        self.S, self.norm, self.n = float(self.diag(self.occ)[0]), w, 0
        self.k = ((seed + 1) & 0xFFFFFFFF, (seed + 1) >> 32)
        # y^T H: the reference and its neighbours (a symmetric H)
        st = self.occ
        site = np.tile(np.flatnonzero(st[0]), len(self.nbr))
        to = self.nbr[np.repeat(np.arange(len(self.nbr)), len(site) // len(self.nbr)), site]
        dest = np.repeat(st, len(site), axis=0)
        h = -np.sqrt((dest[np.arange(len(site)), site]
                      * (dest[np.arange(len(site)), to] + 1)).astype(float))
        dest[np.arange(len(site)), site] -= 1
        dest[np.arange(len(site)), to] += 1
        self.ref_occ = np.concatenate([st, dest])
        self.ref_h = w * np.concatenate([self.diag(st), h])

    def diag(self, occ):
        return (self.c["u"] * 0.5) * (occ * (occ - 1)).sum(axis=1).astype(float)

    def rng_h(self, lo, hi):
        return lo if self.N + self.M - 1 <= 64 else lo ^ _splitmix64(hi)

    def step(self):
        c, dt, integer = self.c, self.c["dt"], self.c["mode"] == "INT"
        theta, occ, a, n = c.get("threshold", 1.0), self.occ, self.a, self.n + 1
        lo, hi = _encode(occ)
        h = self.rng_h(lo, hi)
        n_occ = (occ > 0).sum(axis=1)
        m = len(self.nbr) * n_occ
        exact = np.abs(a) * c.get("t_rel", 1.0) >= m
        if integer:
            exact[:] = False
        cnt = np.where(exact, m, np.ceil(np.abs(a)).astype(np.int64))
        coef = np.where(exact, -dt * a, (-dt * (m / np.maximum(cnt, 1))) * a)
        src = np.repeat(np.arange(len(a)), cnt)
        att = np.arange(len(src)) - np.repeat(np.cumsum(cnt) - cnt, cnt)
        w0, w1, w2 = _philox(n, att, h[src], *self.k)
        k = np.where(exact[src], att, ((w2 * m[src].astype(np.uint64)) >> np.uint64(32)).astype(int))
        d, r = k // n_occ[src], k % n_occ[src]
        site = (np.cumsum(occ > 0, axis=1)[src] == (r + 1)[:, None]).argmax(axis=1)
        to = self.nbr[d, site]
        dest, rows = occ[src], np.arange(len(src))
        hop = -np.sqrt((dest[rows, site] * (dest[rows, to] + 1)).astype(float))
        dest[rows, site] -= 1
        dest[rows, to] += 1
        w = a * (1.0 + dt * (self.S - self.diag(occ)))
        if integer:
            p = np.abs(hop) * (dt * m[src])
            val = np.sign(a[src]) * (np.floor(p) + (_uniform(w0, w1) < p - np.floor(p)))
            dest, val = dest[val != 0], val[val != 0]
            u = _uniform(*_philox(n, 0xFFFFFFFE, h, *self.k)[:2])
            w = np.floor(w) + (u < w - np.floor(w))
        else:
            val = hop * coef[src]
        spawns = len(val)
        occ, w = np.concatenate([occ, dest]), np.concatenate([w, val])
        lo, hi = _encode(occ)
        order = np.lexsort((lo, hi))
        lo, hi, occ = lo[order], hi[order], occ[order]
        first = np.r_[True, (lo[1:] != lo[:-1]) | (hi[1:] != hi[:-1])]
        w = np.bincount(np.cumsum(first) - 1, w[order])
        lo, hi, occ = lo[first], hi[first], occ[first]
        keep = w != 0
        if not integer:
            u = _uniform(*_philox(n, 0xFFFFFFFF, self.rng_h(lo, hi), *self.k)[:2])
            small = np.abs(w) < theta
            keep &= ~small | (u < np.abs(w) / theta)
            w = np.where(small, np.sign(w) * theta, w)
        self.occ, self.a, self.lo, self.hi = occ[keep], w[keep], lo[keep], hi[keep]
        norm = math.fsum(np.abs(self.a))
        zeta = 0.08
        self.S -= (zeta / dt) * math.log(norm / self.norm)
        self.S -= (zeta * zeta / 4.0 / dt) * math.log(norm / c["target"])
        at = {x.tobytes(): v for x, v in zip(self.occ, self.a)}
        cs = np.array([at.get(x.tobytes(), 0.0) for x in self.ref_occ])
        self.norm, self.n = norm, n
        return {"step": n, "len": len(self.a), "exact_steps": int(exact.sum()),
                "inexact_steps": int((~exact).sum()), "n_spawns": spawns, "shift": self.S,
                "norm": norm, "hproj": float(self.ref_h @ cs), "vproj": self.w * cs[0]}


def exact(case, seed):
    """One pass after `prepare`, in numpy: runs on real-space lattices whose
    whole vector is read back.  Larger runs, momentum space and batches would
    take minutes, single precision takes other random decisions in 64 bits."""
    if (case["form"] != "run" or case["kind"] == KIND_MOM or case["target"] > EXPORT_MOST
            or case["mode"] == "REAL32" or case.get("early")):
        return None
    cells = case["target"] * case["Lx"] * case["Ly"] * (case["equil"] + case["steps"])
    if cells > 9e7:
        return None
    p = _Plain(case, seed)
    for _ in range(case["equil"]):
        p.step()
    rows = [p.step() for _ in range(case["steps"])]
    out = {f: np.array([[r[f] for r in rows]]) for f in rows[0]}
    out.update(_rows(case, p.lo, p.hi, p.a))
    return out
