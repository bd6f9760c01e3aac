"""Workloads of the simulator, each through its public entry points.

What a user of this package does: advance a lattice by Monte Carlo steps (MCS)
between two measurement times, measure the roughness W^2 or the two-time
autocorrelations of a lattice, advance a batch of replicas and measure all of
them, serve a list of jobs.  `listed()` holds one workload for each; `draw(rng)`
gives others over the same ranges of size, rates, block layer, thread cell and
sub-tile.

Lattices are made here in plain torch from the seed: the flat start, roughened
by a few sublattice-parallel sweeps of the deposition / removal rule, so that
every one is a valid slope field like those a run goes through.
"""
import math
import random

import numpy as np
import torch

import paper_1705_01022_gb300 as oct_pkg
from paper_1705_01022_gb300 import _lib, autotune, serve

SWEEPS = 6  # roughening sweeps of a prepared lattice


def listed():
    return [
        # the smallest run: one L=256 KPZ lattice between two log-spaced measurement times,
        # then its W^2 (launch and latency bound)
        sim("run_256_kpz", 256, 1.0, 0.0, mcs=8, measure=True),
        # one Edwards-Wilkinson lattice of the ensemble size, L=4096, run alone with the default sub-tile
        sim("run_4096_ew", 4096, 0.5, 0.5, mcs=8, measure=True),
        # an L that no 64 x 64 sub-tile divides: the default falls to 32 x 16 sites
        sim("run_3136_ragged", 3136, 0.95, 0.05, mcs=8, measure=True),
        # the headline size, 2^17, both rates random, on its tuned sub-tile: one MCS
        sim("run_131072", 131072, 0.95, 0.05, Bx=1024, By=16, mcs=1),
        # the dead-border block layer (borders delayed: both rates are positive)
        sim("run_db_12288", 12288, 0.95, 0.05, scheme=1, Bx=256, By=64, mcs=2),
        # double tiling with a moving block origin, on the default sub-tile as the run command takes it
        sim("run_dtr_8192", 8192, 0.95, 0.05, scheme=2, mcs=2),
        # the paper's finest thread cell (8 x 8 sites) on a large lattice
        sim("run_cells8_16384", 16384, 0.95, 0.05, Bx=256, By=64, cx=8, cy=8, mcs=1),
        # the cell the tuner takes when W^2 may be 1 % off sequential updating (16 x 16 sites), default sub-tile
        sim("run_cells16_8192", 8192, 0.95, 0.05, cx=16, cy=16, mcs=1),
        # the exact roughness of the headline lattice
        {"name": "w2_131072", "kind": "w2", "L": 131072},
        # two-time autocorrelations of a large lattice against its snapshot
        {"name": "ac_65536", "kind": "ac", "L": 65536},
        # many replicas of uneven size and mixed rates between two measurement times, then every replica's W^2
        {"name": "batch_256_mixed", "kind": "batch", "n": 256, "L_min": 64, "L_max": 2048, "policy": "default",
         "mcs": 16, "fetch": False},
        # a list of jobs of mixed size and length through the serving engine, W^2 streamed at 8 times each;
        # the memory budget makes some of them wait for others to leave
        {"name": "serve_24", "kind": "serve", "n": 24, "L_min": 128, "L_max": 4096, "t_min": 10, "t_max": 120,
         "budget": 24 << 20},
    ]


def sim(name, L, p, q, scheme=0, Bx=0, By=0, cx=4, cy=4, mcs=1, measure=False):
    c = {"kind": "run", "L": L, "p": p, "q": q, "scheme": scheme, "Bx": Bx, "By": By, "cx": cx, "cy": cy, "mcs": mcs,
         "measure": measure}
    return {"name": name, **c} if name else c


def draw(rng: random.Random):
    kind = rng.choices(("run", "w2", "ac", "batch", "serve"), (10, 2, 2, 3, 1))[0]
    if kind == "run":
        return _draw_run(rng)
    if kind in ("w2", "ac"):
        return {"kind": kind, "L": 64 * round(_log(rng, 4, 1024 if kind == "w2" else 768))}
    if kind == "batch":
        fetch = rng.random() < 0.25  # a checkpoint of every replica: few replicas
        n = round(_log(rng, 4, 24 if fetch else 384))
        lo = 64 * rng.randint(1, 8)
        hi = lo + 64 * rng.randint(0, 28)
        if rng.random() < 0.3:  # an ensemble: realizations of one size
            lo = hi
        return {"kind": "batch", "n": n, "L_min": lo, "L_max": hi, "policy": rng.choice(("default", "default", "tall")),
                "mcs": rng.randint(3, 24), "fetch": fetch}
    return {"kind": "serve", "n": rng.randint(6, 24), "L_min": 128, "L_max": rng.choice((1024, 2048, 4096)), "t_min": 10,
            "t_max": rng.randint(40, 120), "budget": rng.choice((12 << 20, 24 << 20))}


def _draw_run(rng):
    p, q = rng.choice(((1.0, 0.0), (0.95, 0.05), (0.5, 0.5), (0.8, 0.2), (0.95, 0.0)))
    scheme = rng.choice((0, 0, 0, 1, 2))
    cx, cy = rng.choice((4, 8, 8, 16, 16, 32)), rng.choice((4, 8, 16))
    if scheme or rng.random() < 0.5:
        cx, cy = 4, 4
    # a coarse cell, DB or DTr costs several times a 4 x 4-cell DT attempt
    top = 512 if scheme == 0 and (cx, cy) == (4, 4) else 192
    L = 64 * round(_log(rng, 2, top))
    shapes = [(0, 0)] + [s for s in ((256, 64), (1024, 16), (128, 128), (64, 64), (32, 32))
                         if L % (2 * s[0]) == 0 and L % (2 * s[1]) == 0]
    Bx, By = rng.choice(shapes)
    mcs = max(1, min(rng.randint(1, 16), int(2e8 / (L * L)) + 1))
    return sim(None, L, p, q, scheme=scheme, Bx=Bx, By=By, cx=cx, cy=cy, mcs=mcs, measure=rng.random() < 0.5)


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# ------------------------------------------------------------------ inputs --

def flat(L):
    """The flat start h = (x + y) mod 2 as planar words [2, L, L/32]."""
    lat = torch.empty((2, L, L // 32), dtype=torch.int32, device="cuda")
    lat[:, 0::2] = -0x55555556  # odd x
    lat[:, 1::2] = 0x55555555   # even x
    return lat


def roughen(lat, gen, sweeps):
    """Sublattice-parallel sweeps on planar words, in place: every minimum of a
    sublattice rises with probability 1/2, every maximum falls with 1/4."""
    X, Y = lat[0], lat[1]
    L = X.shape[0]

    def words():
        return torch.randint(-2 ** 31, 2 ** 31, X.shape, dtype=torch.int32, device="cuda", generator=gen)

    row = torch.arange(L, device="cuda", dtype=torch.int64).reshape(-1, 1) & 1
    for _ in range(sweeps):
        for c in (0, 1):
            par = torch.where(row == c, 0x55555555, -0x55555556).to(torch.int32)
            xr = ((X >> 1) & 0x7FFFFFFF) | (torch.roll(X, -1, 1) << 31)
            yd = torch.roll(Y, -1, 0)
            up = words() & ~X & xr & ~Y & yd
            f = (up | (words() & words() & X & ~xr & Y & ~yd)) & par
            del xr, yd, up
            X ^= f ^ ((f << 1) | ((torch.roll(f, 1, 1) >> 31) & 1))
            Y ^= f ^ torch.roll(f, 1, 0)
    return lat


def generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def key(seed):
    return (seed * 0x9E3779B97F4A7C15 + 1) % 2 ** 64


def sizes(case):
    """The replicas' L: multiples of 64 spread over [L_min, L_max], the same for every seed."""
    m = (case["L_max"] - case["L_min"]) // 64 + 1
    return [case["L_min"] + 64 * ((i * 37 + i // m) % m) for i in range(case["n"])]


RATES = ((1.0, 0.0), (0.95, 0.05), (0.5, 0.5))


def jobs(case, seed):
    """Jobs that have all arrived; sizes and lengths log-uniform, the same for every seed."""
    rng = random.Random(case["n"])
    out = []
    for i in range(case["n"]):
        L = 128 * max(1, round(_log(rng, case["L_min"], case["L_max"]) / 128))
        t_max = round(_log(rng, case["t_min"], case["t_max"]))
        p, q = rng.choice(serve.PQ_SET)
        out.append(serve.Job(i, L, p, q, _lib.oct_replica_seed(key(seed), i), t_max, measure_at=serve.log_times(t_max)))
    return out


def prepare(case, seed):
    stream = torch.cuda.current_stream()
    st = {"case": case, "seed": seed}
    if case["kind"] == "batch":
        reps = []
        for i, L in enumerate(sizes(case)):
            shape = () if case["policy"] == "default" else autotune.batch_shape(L, case["policy"])
            reps.append((L, *RATES[i % 3], _lib.oct_replica_seed(key(seed), i), *shape))
        st["batch"] = oct_pkg.Batch(reps, stream=stream)
        return st
    if case["kind"] == "serve":
        st["engine"] = serve.ServingEngine(case["budget"], stream=stream)
        return st
    L, gen = case["L"], generator(seed)
    lat = roughen(flat(L), gen, SWEEPS)
    st["lattice"] = lat
    run_args = {k: case[k] for k in ("Bx", "By", "cx", "cy", "scheme")} if case["kind"] == "run" else {}
    st["sim"] = oct_pkg.Simulation(L, case.get("p", 1.0), case.get("q", 0.0), key(seed), stream=stream, lattice=lat,
                                   no_init=True, **run_args)
    if case["kind"] == "ac":
        st["sim"].snapshot()  # the state at the waiting time; the lattice then moves on
        st["snapshot"] = lat.clone()
        roughen(lat, gen, 2)
    return st


# --------------------------------------------------------------------- run --

def run(st):
    case = st["case"]
    if case["kind"] == "run":
        st["sim"].run(case["mcs"])
        out = {"lattice": st["lattice"]}
        if case["measure"]:
            out["w2"] = w2_out(st["sim"].measure())
        return out
    if case["kind"] == "w2":
        return w2_out(st["sim"].measure())
    if case["kind"] == "ac":
        m = st["sim"].measure_ac()
        return {"sum_ht": m.sum_ht, "sum_hs": m.sum_hs, "cross": signed(m.cross_lo), "occ_x": m.occ_x, "occ_y": m.occ_y,
                "m_t": m.m_t, "m_s": m.m_s, "c_h": np.float64(m.c_h), "c_s": np.float64(m.c_s)}
    if case["kind"] == "batch":
        b = st["batch"]
        b.run(case["mcs"])
        ms = [w2_out(m) for m in b.measure()]
        out = {k: np.array([m[k] for m in ms]) for k in ms[0]}
        if case["fetch"]:
            out["planes"] = [b.planes(r) for r in range(len(b))]
        return out
    todo = jobs(case, st["seed"])
    st["engine"].run(todo)
    # every streamed record of every job: t, S1, S2, net flips, W^2
    recs = [r for j in todo for r in j.results]
    return {"counts": np.array([(r[0], r[1], r[2], r[4]) for r in recs], dtype=np.int64),
            "w2": np.array([r[3] for r in recs], dtype=np.float64)}


def w2_out(m):
    return {"t": m.t, "s1": m.s1, "s2": signed(m.s2_lo), "s2_hi": int(m.s2_hi), "net_flips": m.net_flips, "hmax": m.hmax,
            "w2": np.float64(m.w2)}


def signed(lo):
    """The low 64 bits of a sum as a signed integer."""
    return lo - 2 ** 64 if lo >= 2 ** 63 else lo


# ------------------------------------------------------------------- exact --

def height_chunks(lat):
    """Heights relative to h(0, 0) = 0 of planar words, as int64 blocks of rows."""
    X, Y = lat[0], lat[1]
    L = X.shape[0]
    steps = 2 * (Y[:, 0].to(torch.int64) & 1) - 1
    steps[0] = 0
    h0 = torch.cumsum(steps, 0)
    bit = torch.arange(32, device="cuda", dtype=torch.int32)
    rows = max(1, (1 << 26) // L)
    for y in range(0, L, rows):
        s = 2 * ((X[y:y + rows].unsqueeze(-1) >> bit) & 1).reshape(-1, L).to(torch.int64) - 1
        s[:, 0] = h0[y:y + rows]
        yield torch.cumsum(s, 1)


def popcount(words):
    return sum(int(((words >> i) & 1).sum(dtype=torch.int64)) for i in range(32))


def exact(case, seed):
    """The measurements in 64-bit integers by plain torch; a run has no value
    but its own random streams'."""
    if case["kind"] not in ("w2", "ac"):
        return None
    L, gen = case["L"], generator(seed)
    lat = roughen(flat(L), gen, SWEEPS)
    N = L * L
    if case["kind"] == "w2":
        s1 = s2 = hmax = 0
        for h in height_chunks(lat):
            s1 += int(h.sum())
            s2 += int((h * h).sum())
            hmax = max(hmax, int(h.abs().max()))
        return {"t": 0, "s1": s1, "s2": s2, "s2_hi": 0, "net_flips": 0, "hmax": hmax,
                "w2": np.float64((N * s2 - s1 * s1) / (N * N))}
    snap = lat.clone()
    roughen(lat, gen, 2)
    st = ss = cross = 0
    for a, b in zip(height_chunks(lat), height_chunks(snap)):
        st += int(a.sum())
        ss += int(b.sum())
        cross += int((a * b).sum())
    ox, oy = popcount(lat[0] & snap[0]), popcount(lat[1] & snap[1])
    mt, ms = popcount(lat), popcount(snap)
    return {"sum_ht": st, "sum_hs": ss, "cross": cross, "occ_x": ox, "occ_y": oy, "m_t": mt, "m_s": ms,
            "c_h": np.float64((N * cross - st * ss) / (N * N)),
            "c_s": np.float64((2 * N * (ox + oy) - mt * ms) / (4 * N * N))}


# -------------------------------------------------------------------- work --

def work(case):
    """One pass: every lattice read once and, where it is advanced, written
    once; `flops` counts integer operations (8 per update attempt with
    acceptance draws, 6 without; 2 per site measured, 4 for two lattices)."""
    if case["kind"] == "run":
        n = case["L"] ** 2
        ops = 8 if 0 < case["p"] < 1 or 0 < case["q"] < 1 else 6
        return {"bytes": n // 2, "flops": n * case["mcs"] * ops + (2 * n if case["measure"] else 0)}
    if case["kind"] == "w2":  # the X plane and one word of Y a row
        return {"bytes": case["L"] ** 2 // 8 + 4 * case["L"], "flops": 2 * case["L"] ** 2}
    if case["kind"] == "ac":  # both planes of both lattices
        return {"bytes": case["L"] ** 2 // 2, "flops": 4 * case["L"] ** 2}
    if case["kind"] == "batch":
        n = sum(L * L for L in sizes(case))
        return {"bytes": n // 2, "flops": n * (7 * case["mcs"] + 2)}
    todo = jobs(case, 1)
    return {"bytes": sum(j.L * j.L for j in todo) // 2, "flops": sum(7 * j.attempts + 2 * j.L * j.L * len(j.measure_at) for j in todo)}
