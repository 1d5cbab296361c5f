"""The work that programs have this library do, as cases to measure.

Every case is one call sequence of a user's program through the public entry
points: a whole solve (``Solver.run`` and the reads after it), a burst of
requests through the serving loop, a dense instance, or sweeps on the caller's
own device buffers.  All results are whole numbers (cuts, configurations,
energies, controller state), the same bit for bit for any correct
implementation, so every tolerance is "exact".
"""
import math

import numpy as np
import torch

import paper_2606_25203_gb300 as pg
import workloads as W
from paper_2606_25203_gb300.serving import Server

DEVICE = 0
# a program that samples reads the whole population back; a solver of a large
# one reads the best configuration only
READ_POPULATION = 1 << 23


def listed():
    return [
        # the smallest calls: a toy instance solved from a loop, all latency and launches
        dict(name="solve_tiny", do="solve", graph="torus", n=256, R=32, sweeps=2, steps=20,
             beta0=0.1, beta1=3.0),
        # G1-G10 class, a short anneal with a small population: narrow levels of dense rows
        dict(name="solve_er800", do="solve", graph="er", n=800, degree=48.0, R=128, sweeps=5, steps=50,
             beta0=0.1, beta1=3.0),
        # toroidal G-set class with the augmented method (cluster moves, reheating), a large population
        dict(name="solve_torus141", do="solve", graph="torus", n=19881, R=4096, sweeps=10, steps=60,
             beta0=0.1, beta1=4.0, stagnation=True, z_rst=400),
        # sparse +-1 graph (G55-G64 class), the same method and population
        dict(name="solve_sparse7000", do="solve", graph="gnm", n=7000, degree=5.7, signed=True, R=4096,
             sweeps=10, steps=60, beta0=0.1, beta1=4.0, stagnation=True, z_rst=400),
        # one request of a serving stream solved alone: degree 20, ragged sizes, Metropolis
        dict(name="solve_er20_ragged", do="solve", graph="er", n=10007, degree=20.0, R=509, sweeps=10,
             steps=20, beta0=0.1, beta1=3.0, rule=1),
        # Max-3-Cut with the cascaded sampler
        dict(name="maxcut3_cascaded", do="solve", graph="gnm", n=2000, degree=12.0, kind=1, R=2048,
             sweeps=10, steps=30, beta0=0.1, beta1=3.0),
        # Max-3-Cut with the softmax noisy argmax
        dict(name="maxcut3_softmax", do="solve", graph="gnm", n=2000, degree=12.0, kind=1, rule=2, K=3,
             R=2048, sweeps=10, steps=30, beta0=0.1, beta1=3.0),
        # integer weights up to 100: field ranges beyond a byte
        dict(name="solve_weighted", do="solve", graph="weighted", n=2500, degree=12.0, wmax=100, R=250,
             sweeps=5, steps=20, beta0=0.01, beta1=0.3),
        # a burst of uneven requests through the continuous-batching server
        dict(name="serve_burst", do="serve", requests=10, mix=1, n_lo=800, n_hi=20000, max3=0.25, R=512,
             sweeps=10, steps=40, beta0=0.1, beta1=3.0),
        # the fully connected instance, annealed from the random start to the cold end
        dict(name="dense_100k", do="dense", n=100000, R=64, sweeps=2, steps=20, beta0=0.01, beta1=1.0),
        # a fully connected instance of odd size
        dict(name="dense_odd", do="dense", n=5001, R=24, sweeps=2, steps=30, beta0=0.045, beta1=4.5),
        # sweeps at one temperature on the caller's own device buffers
        dict(name="sweeps_fixed_beta", do="sweeps", graph="gnm", n=7000, degree=5.7, signed=True, R=1024,
             sweeps=4, beta=0.7, rule=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["solve"] * 6 + ["dense"] * 2 + ["serve", "sweeps"])
    if do == "dense":
        n = _log_int(rng, 256, 40000)
        return dict(do=do, n=n, R=_log_int(rng, 4, 64), sweeps=rng.randint(1, 2), steps=rng.randint(5, 20),
                    rule=rng.randint(0, 1), beta0=round(3.2 / math.sqrt(n), 4),
                    beta1=round(rng.uniform(100.0, 320.0) / math.sqrt(n), 3))
    if do == "serve":
        return dict(do=do, requests=rng.randint(2, 8), mix=rng.randint(2, 10**6), n_lo=800, n_hi=_log_int(rng, 1500, 20000),
                    max3=round(rng.uniform(0.0, 0.5), 2), R=_log_int(rng, 64, 512),
                    sweeps=rng.randint(2, 10), steps=rng.randint(10, 40), beta0=0.1,
                    beta1=round(rng.uniform(2.0, 4.0), 2))
    if do == "sweeps":
        return dict(do=do, graph="gnm", n=_log_int(rng, 64, 20000), degree=round(rng.uniform(3.0, 8.0), 2),
                    signed=rng.random() < 0.5, R=_log_int(rng, 4, 2048), sweeps=rng.randint(1, 8),
                    beta=round(rng.uniform(0.1, 2.0), 3), rule=rng.randint(0, 1))
    graph = rng.choice(["torus", "gnm", "er", "weighted"])
    n = _log_int(rng, 64, 20000)
    R = _log_int(rng, 4, 4096)
    sweeps = rng.randint(1, 10)
    # bounded attempts, so that no drawn solve costs more than the largest listed case
    steps = max(2, min(rng.randint(10, 60), int(3e9 / (n * R * sweeps))))
    case = dict(do=do, graph=graph, n=n, R=R, sweeps=sweeps, steps=steps, beta0=0.1,
                beta1=round(rng.uniform(2.0, 4.0), 2), rule=rng.randint(0, 1))
    if graph == "torus":
        case["n"] = max(3, int(round(math.sqrt(n)))) ** 2
    elif graph == "gnm":
        case.update(degree=round(rng.uniform(3.0, 12.0), 2), signed=rng.random() < 0.5)
    elif graph == "er":
        case.update(degree=round(min(rng.uniform(10.0, 48.0), n / 4), 2), signed=rng.random() < 0.5)
    else:
        case.update(degree=round(rng.uniform(4.0, 16.0), 2), wmax=rng.choice([3, 10, 100]), beta0=0.01,
                    beta1=0.3)
    if graph in ("torus", "gnm") and rng.random() < 0.4:   # Max-K-Cut, either sampler
        case.update(kind=1, rule=rng.choice([0, 2]), K=3)
        if case["rule"] == 2:
            case["K"] = rng.randint(2, 5)
    elif rng.random() < 0.4:   # the augmented method, with restarts
        case.update(stagnation=True, z_rst=rng.choice([15, 400]))
    return case


# ---------------------------------------------------------------- inputs
def _graph(case, seed):
    g, n = case["graph"], case["n"]
    if g == "torus":
        side = int(round(math.sqrt(n)))
        return W.torus(side, side, signed=True, seed=seed)
    if g == "er":
        return W.er_avg_degree(n, case["degree"], signed=case.get("signed", False), seed=seed)
    if g == "gnm":
        return W.gnm(n, int(round(n * case["degree"] / 2)), signed=case.get("signed", False), seed=seed)
    base = W.er_avg_degree(n, case["degree"], signed=False, seed=seed)
    src = np.repeat(np.arange(n, dtype=np.int64), np.diff(base.row_ptr))
    up = src < base.col
    w = np.random.default_rng([seed, n]).integers(1, case["wmax"] + 1, size=int(up.sum()))
    w = np.where(np.random.default_rng([seed, n, 1]).random(w.shape[0]) < 0.5, w, -w)
    return W.csr_from_edges(n, src[up], base.col[up], w, "weighted")


def _params(case, seed):
    p = dict(kind=case.get("kind", 0), rule=case.get("rule", 0), R=case["R"], sweeps=case["sweeps"],
             steps=case["steps"], beta0=case["beta0"], beta1=case["beta1"], seed=seed, K=case.get("K", 3))
    if case.get("stagnation"):
        p.update(stagnation=1, z_rst=case["z_rst"])
    return p


class _DenseState:
    """A dense handle with its owner's lifetime."""

    def __init__(self, case, seed):
        n = case["n"]
        dev = torch.device("cuda", DEVICE)
        w = torch.empty((n, n), dtype=torch.int8, device=dev)
        rows = max(1, (1 << 27) // n)
        for r0 in range(0, n, rows):
            r1 = min(n, r0 + rows)
            w[r0:r1] = -W.dense_rows_torch(n, r0, r1, seed, dev)
        self.n, self.params = n, _params(case, seed)
        self.h = pg.pamc_create_dense(n, w, DEVICE)

    def __del__(self):
        pg.pamc_destroy(self.h)


class _ServeState:
    def __init__(self, case, seed):
        # sizes, graph types and problems of the mix belong to the case, the graphs to the seed
        rng = np.random.default_rng([case["mix"], case["requests"]])
        self.requests = []
        for i in range(case["requests"]):
            n, s = int(rng.integers(case["n_lo"], case["n_hi"] + 1)), seed * 1009 + i
            g = int(rng.integers(0, 3))
            side = int(round(math.sqrt(n)))
            inst = W.torus(side, side, signed=True, seed=s) if g == 2 else \
                W.er_avg_degree(n, 20.0, signed=g == 1, seed=s)
            self.requests.append(W.Request(i, inst, 0.0, int(rng.random() < case["max3"])))
        self.params = dict(R=case["R"], sweeps=case["sweeps"], steps=case["steps"], beta0=case["beta0"],
                           beta1=case["beta1"], seed=seed)
        self.server = Server(DEVICE, keep_spins=True)


class _SweepsState:
    def __init__(self, case, seed):
        inst = _graph(case, seed)
        dev = torch.device("cuda", DEVICE)
        self.n, self.nnz = inst.n, inst.nnz
        self.H = int(max(np.add.reduceat(np.abs(np.append(inst.w, 0)), inst.row_ptr[:-1]).max(), 1))
        self.rp, self.col, self.w = (torch.from_numpy(a).to(dev) for a in (inst.row_ptr, inst.col, inst.w))
        self.spins = torch.from_numpy(_spins(case, seed)).to(dev)
        self.case, self.seed = case, seed


def _spins(case, seed):
    bits = np.random.default_rng([seed, 7]).integers(0, 2, size=(case["R"], case["n"]), dtype=np.int8)
    return (2 * bits - 1).astype(np.int8)


def prepare(case, seed):
    if case["do"] == "dense":
        return _DenseState(case, seed)
    if case["do"] == "serve":
        return _ServeState(case, seed)
    if case["do"] == "sweeps":
        return _SweepsState(case, seed)
    inst = _graph(case, seed)
    return pg.Solver(inst.row_ptr, inst.col, inst.w, DEVICE), _params(case, seed)


# ---------------------------------------------------------------- one pass
def _read(h, n, R):
    cut, best = pg.pamc_best(h, n)
    ctl = pg.pamc_control_state(h)
    out = {"cut": cut, "best": best, "t": ctl["t"], "cycle": ctl["cycle"], "ncm_flipped": ctl["ncm_flipped"],
           "beta": ctl["beta"], "family": pg.pamc_lineage(h, R)[0]}
    if R * n <= READ_POPULATION:
        out["spins"], out["E"], out["parents"], out["counts"] = pg.pamc_state(h, R, n)
    return out


def run(state):
    if isinstance(state, _DenseState):
        pg.pamc_run(state.h, **state.params)
        return _read(state.h, state.n, state.params["R"])
    if isinstance(state, _ServeState):
        stats = state.server.serve(state.requests, state.params)
        res = sorted(stats.results, key=lambda r: r.rid)
        return {"cuts": np.array([r.cut for r in res], dtype=np.int64),
                "spins": np.concatenate([r.spins for r in res])}
    if isinstance(state, _SweepsState):
        c = state.case
        out = torch.empty_like(state.spins)
        E = torch.empty(c["R"], dtype=torch.int64, device=out.device)
        pg.pamc_sweeps_noalloc(state.n, state.nnz, state.rp, state.col, state.w, state.H, c["rule"], c["R"],
                               c["sweeps"], c["beta"], state.seed, 3, state.spins, out, E)
        return {"spins": out, "E": E}
    solver, params = state
    solver.run(**params)
    return _read(solver.h, solver.n, params["R"])


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: the instance and the results once; for a dense instance one bit
    per coupling for each step's recompute (it fits no on-chip memory).
    Operations: 18 integer operations per spin-flip attempt (a quarter of a
    Philox4x32-10 call and the threshold compare), and the 2 n^2 R of a dense
    instance's recompute."""
    R, sweeps, steps = case["R"], case["sweeps"], case.get("steps", 1)
    if case["do"] == "dense":
        n = case["n"]
        return {"bytes": n * n / 8 * steps + n + 4 * R,
                "flops": (2.0 * n * n * R + 18.0 * n * R * sweeps) * steps}
    if case["do"] == "serve":
        n = case["requests"] * (case["n_lo"] + case["n_hi"]) / 2
        return {"bytes": 2 * n + 8 * 15 * n, "flops": 18.0 * n * R * sweeps * steps}
    n = case["n"]
    deg = 4.0 if case["graph"] == "torus" else case["degree"]
    b = 8 * deg * n + 4 * n + n + 4 * R
    if case["do"] == "sweeps":
        b += 2.0 * n * R + 8 * R
    elif n * R <= READ_POPULATION:
        b += n * R + 16 * R
    return {"bytes": b, "flops": 18.0 * n * R * sweeps * steps}


def tolerance(case):
    return "exact"


# ---------------------------------------------------------------- 64-bit restatement of the fixed-temperature sweeps
def _philox(c0, c1, c2, c3, seed):
    m = np.uint64(0xFFFFFFFF)
    c0, c1, c2, c3 = (np.asarray(c, dtype=np.uint64) for c in (c0, c1, c2, c3))
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, b = c0 * np.uint64(0xD2511F53), c2 * np.uint64(0xCD9E8D57)
        c0, c1, c2, c3 = ((b >> np.uint64(32)) ^ c1 ^ np.uint64(k0), b & m,
                          (a >> np.uint64(32)) ^ c3 ^ np.uint64(k1), a & m)
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1, c2, c3


def exact(case, seed):
    """Sweeps at one temperature, position by position, every replica at once.
    The solves are chains of such sweeps and integer resampling whose results
    are whole numbers; they have no 64-bit value other than themselves."""
    if case["do"] != "sweeps":
        return None
    inst = _graph(case, seed)
    n, R, t = inst.n, case["R"], 3
    s = np.ascontiguousarray(_spins(case, seed).T.astype(np.int64))   # [n][R]
    J = -inst.w.astype(np.int64)
    rp, col = inst.row_ptr, inst.col
    H = max(int(np.abs(J[rp[k]:rp[k + 1]]).sum()) for k in range(n))
    h = np.arange(-H, H + 1, dtype=np.float64)
    if case["rule"] == 0:
        T = np.floor(2.0 ** 32 / (1.0 + np.exp(-2.0 * case["beta"] * h)) + 0.5)
    else:
        T = np.floor(2.0 ** 32 * np.exp(-case["beta"] * np.maximum(2.0 * h, 0.0)) + 0.5)
    groups = (R + 3) // 4
    for sw in range(case["sweeps"]):
        keys = _philox(np.arange(n), sw, t, 2 << 24, seed)[0]
        u = _philox(np.arange(n)[:, None], sw, t, ((3 << 24) + np.arange(groups))[None, :], seed)
        u = np.stack(np.broadcast_arrays(*u), axis=2).astype(np.float64).reshape(n, 4 * groups)[:, :R]
        for k in np.argsort(keys, kind="stable"):
            e0, e1 = rp[k], rp[k + 1]
            f = J[e0:e1] @ s[col[e0:e1]] if e1 > e0 else np.zeros(R, dtype=np.int64)
            if case["rule"] == 0:
                s[k] = np.where(u[k] < T[f + H], 1, -1)
            else:
                s[k] = np.where(u[k] < T[s[k] * f + H], -s[k], s[k])
    E = np.zeros(R, dtype=np.int64)
    for k in range(n):
        E -= s[k] * (J[rp[k]:rp[k + 1]] @ s[col[rp[k]:rp[k + 1]]])
    return {"spins": s.T.astype(np.int8), "E": E // 2}
