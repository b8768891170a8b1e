"""Performance cases: what users of this framework have it do, through its public entry points.

A case names a path ("series": transient distributions, "loglik": snapshot log-likelihoods of a batch of
parameter vectors, "batch": uneven birth-death instances, "csr": general rate matrices, "train": the
surrogate's training, "sampler": delayed-acceptance iterations) and its sizes.  `listed` holds the
configurations of the benchmark and the tests beside small and odd ones, `draw` spreads over the same ranges,
`prepare` makes what a program holds before the call, `run` is one call, `work` counts what the call cannot do
without and `exact` computes the result in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

import paper_2312_05647_gb300 as mjp
from paper_2312_05647_gb300 import surrogate

KINDS = {"bd": mjp.BD1D, "twostate": mjp.TWOSTATE, "mrna": mjp.MRNA_PROT2D, "autoreg": mjp.AUTOREG}
PREC = {"f32": mjp.FP32, "f64": mjp.FP64}
# Nominal rates: immigration-death, two-state promoter, mRNA/protein box, autoregulatory network.
RATES = {"bd": [10.0, 1.0], "twostate": [100.0, 1.0, 2.0, 1.0], "mrna": [20.0, 1.0, 5.0, 0.1],
         "autoreg": [10.0, 0.5, 1.0, 0.1, 0.1, 0.05]}


def listed():
    return [
        # The smallest solve: immigration-death on 64 states at five times, FP64; latency and launches count.
        dict(name="series_bd64_f64", path="series", kind="bd", d0=64, d1=1, prec="f64", nt=5, t0=0.1, t1=5.0),
        # One transient solve of the mRNA/protein box at 20 log-spaced times: 69,089 jumps of 40,000 states.
        dict(name="series_mrna200_f32", path="series", kind="mrna", d0=200, d1=200, prec="f32", nt=20, t0=0.1, t1=50.0),
        # The headline workload: log-likelihoods of 152 thetas on the same box.
        dict(name="loglik_mrna200_152_f32", path="loglik", kind="mrna", d0=200, d1=200, prec="f32", nt=20, t0=0.1,
             t1=50.0, cells=100, B=152, host=False),
        # The samplers' exact evaluation: 256 thetas of the two-state promoter, 50 times x 100 cells.
        dict(name="loglik_promoter300_256_f32", path="loglik", kind="twostate", d0=300, d1=1, prec="f32", nt=50, t0=0.5,
             t1=10.0, cells=100, B=256, host=False),
        # One theta from host memory on an odd promoter in FP64: what an optimiser or a check calls.
        dict(name="loglik_promoter131_1_f64", path="loglik", kind="twostate", d0=131, d1=1, prec="f64", nt=13, t0=0.5,
             t1=6.0, cells=30, B=1, host=True),
        # A parameter scan of the small immigration-death model in FP64.
        dict(name="loglik_bd64_10000_f64", path="loglik", kind="bd", d0=64, d1=1, prec="f64", nt=5, t0=0.1, t1=5.0,
             cells=100, B=10000, host=False),
        # The autoregulatory network, 6,000 observations with the gene state summed out.
        dict(name="loglik_autoreg40x120_152_f32", path="loglik", kind="autoreg", d0=40, d1=120, prec="f32", nt=50,
             t0=0.5, t1=10.0, cells=120, B=152, host=False),
        # 4,096 uneven birth-death instances in one call (N 100 .. 20,000, K 10 .. several 100,000).
        dict(name="batch_4096_f32", path="batch", n=4096, nlo=100, nhi=20000, tlo=0.01, thi=10.0, prec="f32",
             graph=False),
        # A general random rate matrix on 2^20 states, eight transitions a row.
        dict(name="csr_1048576_f32", path="csr", n=1048576, dlo=8, dhi=8, near=0.0, x=220.0, nt=1, prec="f32"),
        # An odd rate matrix in FP64 with ragged rows, half of the transitions between nearby states, three times.
        dict(name="csr_100003_f64", path="csr", n=100003, dlo=0, dhi=13, near=0.5, x=150.0, nt=3, prec="f64"),
        # Training the surrogate on recorded evaluations: Adam steps on minibatches of 1,024 of 65,536 rows.
        dict(name="train_65536_1024", path="train", rows=65536, batch=1024, steps=100),
        # Delayed-acceptance iterations of 256 chains on the promoter data: the whole inference loop.
        dict(name="sampler_da_256", path="sampler", d0=300, nt=50, t0=0.5, t1=10.0, cells=100, chains=256, iters=20),
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _kind_dims(rng):
    kind = rng.choice(["bd", "twostate", "mrna", "autoreg"])
    if kind == "bd":
        return kind, _logint(rng, 16, 8000), 1
    if kind == "twostate":
        return kind, _logint(rng, 16, 900), 1
    if kind == "mrna":
        return kind, _logint(rng, 10, 200), _logint(rng, 10, 200)
    return kind, _logint(rng, 8, 40), _logint(rng, 8, 120)


def _scaled_rates(kind, d0, d1):
    """Rates whose stationary distribution lies inside the box (means near 40% of each side)."""
    r = list(RATES[kind])
    if kind == "bd":
        r[0] = 0.4 * d0 * r[1]
    elif kind == "twostate":
        r[0] = 0.5 * d0 * r[1]
    elif kind == "mrna":
        r[0] = 0.3 * d0 * r[1]
        r[2] = 0.4 * d1 * r[3] / (0.3 * d0)
    else:
        r[0] = 0.4 * d0 * r[2]
        r[1] = 0.4 * d1 * r[3] / (0.4 * d0)
    return r


def draw(rng):
    path = rng.choice(["series", "series", "loglik", "loglik", "loglik", "batch", "csr", "csr", "train", "sampler"])
    prec = rng.choice(["f32", "f64"])
    if path in ("series", "loglik"):
        kind, d0, d1 = _kind_dims(rng)
        n = math.prod(_shape(kind, d0, d1))
        B = 1 if path == "series" else _logint(rng, 1, 2048)
        # x = Omega t1, the number of jumps, within what the largest listed cases cost.
        most = (2e8 if prec == "f64" else 1e9) if B == 1 else (1.5e9 if prec == "f64" else 1.5e10)
        x = math.exp(rng.uniform(math.log(20.0), math.log(max(40.0, min(5000.0, most / (B * n))))))
        t1 = x / (1.1 * _max_exit(kind, d0, d1, _scaled_rates(kind, d0, d1)))
        c = dict(path=path, kind=kind, d0=d0, d1=d1, prec=prec, nt=_logint(rng, 1, 50), t0=t1 * rng.uniform(0.02, 0.9),
                 t1=t1)
        if path == "loglik":
            c.update(cells=_logint(rng, 10, 120), B=B, host=rng.random() < 0.3)
        return c
    if path == "batch":
        nhi = _logint(rng, 200, 6000)
        return dict(path=path, n=_logint(rng, 1, 400), nlo=max(2, nhi // 20), nhi=nhi, tlo=0.01,
                    thi=rng.uniform(0.1, 2.0), prec=prec, graph=rng.random() < 0.5)
    if path == "csr":
        dlo = rng.randint(0, 8)
        return dict(path=path, n=_logint(rng, 1000, 1 << 19), dlo=dlo, dhi=dlo + rng.randint(0, 8) + (dlo == 0),
                    near=rng.choice([0.0, 0.5, 1.0]), x=rng.uniform(20.0, 250.0), nt=rng.randint(1, 4), prec=prec)
    if path == "train":
        rows = _logint(rng, 1000, 65536)
        return dict(path=path, rows=rows, batch=_logint(rng, 32, 2048), steps=rng.randint(10, 100))
    return dict(path=path, d0=_logint(rng, 60, 320), nt=rng.randint(5, 50), t0=0.5, t1=rng.uniform(2.0, 10.0),
                cells=rng.randint(20, 100), chains=_logint(rng, 16, 512), iters=rng.randint(4, 20))


# ---- models as transitions on a grid ---------------------------------------

def _shape(kind, d0, d1):
    """Grid of a model in index order (the last axis runs fastest)."""
    return {"bd": (d0,), "twostate": (2, d0), "mrna": (d1, d0), "autoreg": (2, d1, d0)}[kind]


def _transitions(kind, th, c):
    """(step, rate) of each reaction: th the parameters, c the grid coordinates (both broadcast)."""
    if kind == "bd":
        return [((1,), th[0] + 0 * c[0]), ((-1,), th[1] * c[0])]
    if kind == "twostate":
        s, n = c
        return [((0, 1), th[0] * (s == 0)), ((0, -1), th[1] * n), ((1, 0), th[3] * (s == 0)), ((-1, 0), th[2] * (s == 1))]
    if kind == "mrna":
        p, m = c
        return [((0, 1), th[0] + 0 * m), ((0, -1), th[1] * m), ((1, 0), th[2] * m), ((-1, 0), th[3] * p)]
    s, p, r = c
    return [((0, 0, 1), th[0] * (s == 0)), ((0, 1, 0), th[1] * r), ((0, 0, -1), th[2] * r), ((0, -1, 0), th[3] * p),
            ((1, -1, 0), th[5] * p * (s == 0)), ((-1, 1, 0), th[4] * (s == 1))]


def _sides(step):
    """Source and target slices of a step inside the box."""
    src = tuple(slice(0, -1) if d > 0 else slice(1, None) if d < 0 else slice(None) for d in step)
    dst = tuple(slice(1, None) if d > 0 else slice(0, -1) if d < 0 else slice(None) for d in step)
    return src, dst


def _max_exit(kind, d0, d1, theta):
    shape = _shape(kind, d0, d1)
    c = np.meshgrid(*[np.arange(n, dtype=np.float64) for n in shape], indexing="ij")
    e = np.zeros(shape)
    for step, rate in _transitions(kind, theta, c):
        src, _ = _sides(step)
        e[src] += np.broadcast_to(rate, shape)[src]
    return float(e.max())


def _jumps(x):
    return math.floor(x + 6.0 * math.sqrt(x)) + 1


def _theta(case):
    """The listed configurations' own rates; drawn boxes get rates that fit them."""
    if "name" in case:
        return list(RATES[case["kind"]])
    return _scaled_rates(case["kind"], case["d0"], case["d1"])


def _times(case):
    space = np.geomspace if case["kind"] == "mrna" else np.linspace
    return space(case["t0"], case["t1"], case["nt"]) if case["nt"] > 1 else np.array([case["t1"]])


def _thetas(theta, B, g):
    """B parameter vectors within 20% of the nominal one."""
    return np.asarray(theta)[None, :] * g.uniform(0.8, 1.2, size=(B, len(theta)))


def _snapshots(kind, d0, d1, theta, times, cells, g):
    """Observed cells per time, each its own system from the empty state, by 192 tau-leaps inside the box; grouped by
    the observed value, the gene state summed out: [(members, counts)] per time."""
    shape = _shape(kind, d0, d1)
    T = np.repeat(times, cells)
    st = np.zeros((len(shape), len(T)), dtype=np.int64)
    top = np.array(shape)[:, None] - 1
    dt = T / 192
    for _ in range(192):
        move = np.zeros_like(st)
        for step, rate in _transitions(kind, theta, st):
            hits = g.poisson(np.broadcast_to(rate, T.shape) * dt)
            for a, d in enumerate(step):
                if d:
                    move[a] += d * hits
        st = np.clip(st + move, 0, top)
    flat = np.ravel_multi_index(st[1:] if kind in ("twostate", "autoreg") else st,
                                shape[1:] if kind in ("twostate", "autoreg") else shape)
    half = math.prod(shape[1:])
    out = []
    for i in range(len(times)):
        v, n = np.unique(flat[i * cells:(i + 1) * cells], return_counts=True)
        out.append(([np.array([s, s + half]) if kind in ("twostate", "autoreg") else np.array([s]) for s in v],
                    n.astype(np.float64)))
    return out


def _rng(seed):
    return np.random.default_rng(seed)


def _rho0(n, g):
    """The empty state, with a tenth of the mass spread over the next few (a start that is not quite known)."""
    r = np.zeros(n)
    k = min(n, 8)
    r[:k] = 0.1 * g.dirichlet(np.ones(k))
    r[0] += 0.9
    return r / r.sum()


def _data(case, seed):
    """Host inputs of a series, log-likelihood or sampler case."""
    g = _rng(seed)
    kind, d0, d1 = case.get("kind", "twostate"), case["d0"], case.get("d1", 1)
    theta = _theta(case) if "kind" in case else RATES["twostate"] if "name" in case else _scaled_rates(kind, d0, d1)
    n = math.prod(_shape(kind, d0, d1))
    d = dict(kind=kind, n=n, theta=theta, times=_times({**case, "kind": kind}))
    if case["path"] == "series":
        d["theta"] = list(_thetas(theta, 1, g)[0])
        d["rho0"] = _rho0(n, g)
    else:
        d["rho0"] = np.zeros(n)
        d["rho0"][0] = 1.0
        d["obs"] = _snapshots(kind, d0, d1, theta, d["times"], case["cells"], g)
        d["thetas"] = _thetas(theta, case.get("B", case.get("chains")), g)
    return d


def _csr_data(case, seed):
    g = _rng(seed)
    n = case["n"]
    deg = g.integers(case["dlo"], case["dhi"] + 1, n)
    ptr = np.zeros(n + 1, np.int64)
    np.cumsum(deg, out=ptr[1:])
    nnz = int(ptr[-1])
    row = np.repeat(np.arange(n, dtype=np.int64), deg)
    hop = g.integers(1, n, nnz)
    if case["near"] > 0.0:
        w = min(n - 1, 400)
        close = g.integers(1, w + 1, nnz) * g.choice(np.array([-1, 1]), nnz)
        hop = np.where(g.random(nnz) < case["near"], close, hop)
    col = (row + hop) % n
    rate = g.lognormal(0.0, 1.0, nnz)
    rate *= 200.0 / np.add.reduceat(np.concatenate([rate, [0.0]]), np.minimum(ptr[:-1], nnz))[deg > 0].max()
    rho0 = np.zeros(n)
    some = g.choice(n, size=min(n, 1024), replace=False)
    rho0[some] = 1.0 / len(some)
    times = np.linspace(0.25, 1.0, case["nt"]) * case["x"] / 220.0 if case["nt"] > 1 else np.array([case["x"] / 220.0])
    return ptr, col.astype(np.int32), rate, rho0, times


def _batch_data(case, seed):
    g = _rng(seed)
    n = case["n"]
    sizes = _rng([n, case["nlo"], case["nhi"]])  # the sizes belong to the case, rates and times to the seed
    N = np.floor(np.exp(sizes.uniform(math.log(case["nlo"]), math.log(case["nhi"]), n))).astype(np.int64)
    beta = g.uniform(1.0, np.maximum(N / 4.0, 1.5))
    gamma = g.uniform(0.5, 2.0, n)
    t = np.exp(g.uniform(math.log(case["tlo"]), math.log(case["thi"]), n))
    return N, np.stack([beta, gamma], axis=1), t


def _train_data(case, seed):
    """Rows (Psi, log-likelihood) as the samplers record them: a peaked surface around the promoter's log-rates."""
    g = _rng(seed)
    psi = np.log(RATES["twostate"]) + 0.15 * g.standard_normal((case["rows"], 4))
    d = (psi - np.log(RATES["twostate"])) @ np.array([[1.0, -0.8, 0.2, -0.2], [0, 0.7, 0.1, 0], [0, 0, 0.5, -0.4],
                                                       [0, 0, 0, 0.4]])
    return psi, -20000.0 - 2500.0 * (d ** 2).sum(axis=1) * (1.0 + 0.2 * np.tanh(d[:, 0]))


# ---- the four entry points of a case ----------------------------------------

def prepare(case, seed):
    path = case["path"]
    if path == "series":
        d = _data(case, seed)
        dims = [case["d0"]] if d["kind"] in ("bd", "twostate") else [case["d0"], case["d1"]]
        m = mjp.Model(KINDS[d["kind"]], dims, d["theta"], PREC[case["prec"]])
        return dict(path=path, m=m, rho0=torch.tensor(d["rho0"], dtype=m.torch_dtype, device="cuda"), times=d["times"])
    if path == "loglik":
        d = _data(case, seed)
        dims = [case["d0"]] if d["kind"] in ("bd", "twostate") else [case["d0"], case["d1"]]
        m = mjp.Model(KINDS[d["kind"]], dims, d["theta"], PREC[case["prec"]])
        th = d["thetas"] if case["host"] else torch.tensor(d["thetas"], dtype=torch.float64, device="cuda")
        return dict(path=path, m=m, obs=mjp.Obs(d["n"], d["times"], d["obs"], d["rho0"]), theta=th)
    if path == "batch":
        N, theta, t = _batch_data(case, seed)
        b = mjp.Batch(N, theta, t, precision=PREC[case["prec"]])
        return dict(path=path, b=b, out=b.empty_out(), graph=case["graph"])
    if path == "csr":
        ptr, col, rate, rho0, times = _csr_data(case, seed)
        m = mjp.Model.from_csr(case["n"], ptr, col, rate, PREC[case["prec"]])
        return dict(path=path, m=m, rho0=torch.tensor(rho0, dtype=m.torch_dtype, device="cuda"), times=times)
    if path == "train":
        psi, y = _train_data(case, seed)
        net = surrogate.MLP(seed=seed)
        return dict(path=path, net=net, p0=net.get_params()[0], psi=torch.tensor(psi, device="cuda"),
                    y=torch.tensor(y, device="cuda"), steps=case["steps"], batch=case["batch"], seed=seed)
    d = _data(case, seed)
    m = mjp.Model(mjp.TWOSTATE, [case["d0"]], d["theta"], mjp.FP32)
    obs = mjp.Obs(d["n"], d["times"], d["obs"], d["rho0"])
    C = case["chains"]
    s = surrogate.Sampler(m, obs, C, capacity=case["iters"], eval_capacity=0, seed=seed)
    g = _rng(seed + 1)
    psi = np.log(d["theta"]) + 0.02 * g.standard_normal((C, 4))
    s.set_cov(np.diag([4e-5, 4e-5, 4e-4, 4e-4]))
    net = surrogate.MLP(seed=seed)
    ll = mjp.loglik(m, obs, np.exp(psi))
    fine = np.isfinite(ll)
    net.train(psi[fine], ll[fine], steps=200, batch=256, lr=2e-3, seed=seed)
    return dict(path=path, s=s, net=net, psi=psi, iters=case["iters"])


def run(state):
    path = state["path"]
    if path in ("series", "csr"):
        return state["m"].expv(state["rho0"], state["times"])
    if path == "loglik":
        return mjp.loglik(state["m"], state["obs"], state["theta"])
    if path == "batch":
        return state["b"].run(state["out"], use_graph=state["graph"])
    if path == "train":
        # The surrogate is trained again on new evaluations from its first weights.
        state["net"].set_params(state["p0"])
        losses = state["net"].train(state["psi"], state["y"], steps=state["steps"], batch=state["batch"], lr=2e-3,
                                    seed=state["seed"], device_data=True)
        params, norm = state["net"].get_params()
        return dict(losses=losses, params=params, norm=norm)
    s = state["s"]
    s.set_state(state["psi"])
    s.run_da(state["net"], state["iters"], max_inner=32)
    psi, ll = s.get_state()
    return dict(psi=psi, loglik=ll, trace=s.trace())


def work(case):
    path = case["path"]
    elt = 8 if case.get("prec") == "f64" else 4
    if path in ("series", "loglik"):
        kind, d0, d1 = case["kind"], case["d0"], case["d1"]
        n = math.prod(_shape(kind, d0, d1))
        nth = len(RATES[kind])
        K = _jumps(1.1 * _max_exit(kind, d0, d1, _theta(case)) * case["t1"])
        terms = {"bd": 3, "twostate": 4, "mrna": 5, "autoreg": 6}[kind]
        if path == "series":
            return {"bytes": n * elt * (1 + case["nt"]), "flops": 2.0 * terms * n * K}
        B = case["B"]
        return {"bytes": 8.0 * B * (nth + 1) + n * elt + 16.0 * case["nt"] * case["cells"], "flops": 2.0 * terms * n * K * B}
    if path == "batch":
        N, theta, t = _batch_data(case, 1)
        x = 1.1 * (theta[:, 0] + theta[:, 1] * (N - 2)) * t
        K = np.floor(x + 6.0 * np.sqrt(x)) + 1
        return {"bytes": float(N.sum()) * elt + 32.0 * case["n"], "flops": 6.0 * float((K * N).sum())}
    if path == "csr":
        nnz = case["n"] * 0.5 * (case["dlo"] + case["dhi"])
        # The matrix once (index and rate of each transition, the diagonal), the start and the results.
        return {"bytes": nnz * (4 + elt) + case["n"] * elt * (2.0 + case["nt"]),
                "flops": 2.0 * _jumps(case["x"]) * (nnz + case["n"])}
    if path == "train":
        rows = case["steps"] * min(case["batch"], case["rows"])
        return {"bytes": 40.0 * case["rows"] + 4.0 * 17281 * 2, "flops": 6.0 * 17024 * rows}
    # One delayed-acceptance iteration per chain: the surrogate, then an exact log-likelihood of about half of them.
    theta = RATES["twostate"] if "name" in case else _scaled_rates("twostate", case["d0"], 1)
    K = _jumps(1.1 * _max_exit("twostate", case["d0"], 1, theta) * case["t1"])
    its = case["chains"] * case["iters"]
    return {"bytes": 40.0 * its, "flops": its * (0.5 * 2.0 * 4 * 2 * case["d0"] * K + 2.0 * 17024)}


# ---- the results in 64 bits --------------------------------------------------

def _schedule(omega, times):
    """Weight of every jump 0 .. kmax for each (row, time): Poisson up to K = floor(x + 6 sqrt x) + 1, the tail added
    at K.  Returns the largest K and a function that gives the weights [row, time, jump] of a range of jumps."""
    x = omega[:, None] * times[None, :]
    K = torch.floor(x + 6.0 * torch.sqrt(x)) + 1
    # Ratios to the mode by cumulative sums of logarithms, on the CPU once per (row, time).
    tables = []
    xs, Ks = x.cpu().numpy().ravel(), K.cpu().numpy().ravel().astype(np.int64)
    for xv, kv in zip(xs, Ks):
        m = int(math.floor(xv))
        lo = max(0, int(xv - 10.0 * math.sqrt(xv)))
        hi = int(xv + 10.0 * math.sqrt(xv)) + 60
        up = np.cumsum(np.log(xv / np.arange(m + 1, hi + 1)))
        dn = np.cumsum(np.log(np.arange(m, lo, -1) / xv))[::-1] if m > lo else np.zeros(0)
        w = np.exp(np.concatenate([dn, [0.0], up]))
        w /= w.sum()
        tail = w[kv - lo + 1:].sum()
        w = w[:kv - lo + 1].copy()
        w[-1] += tail
        tables.append((lo, w))
    start = np.array([t[0] for t in tables])
    end = np.array([t[0] + len(t[1]) for t in tables])

    def chunk(k0, k1):
        w = np.zeros((len(tables), k1 - k0))
        for j in np.nonzero((start < k1) & (end > k0))[0]:
            a, b = max(k0, start[j]), min(k1, end[j])
            w[j, a - k0:b - k0] = tables[j][1][a - start[j]:b - start[j]]
        return torch.from_numpy(w).to(x.device).reshape(x.shape[0], x.shape[1], k1 - k0)

    return int(Ks.max()), chunk


def _series64(kind, d0, d1, thetas, times, rho0, states):
    """sum_k w_k (rho0 B^k)[states] for every theta and time, FP64: [B, times, len(states)] (None: all states)."""
    dev = torch.device("cuda")
    shape = _shape(kind, d0, d1)
    B = len(thetas)
    th = torch.tensor(np.asarray(thetas), dtype=torch.float64, device=dev).T.reshape(-1, B, *[1] * len(shape))
    c = [v[None] for v in torch.meshgrid(*[torch.arange(n, dtype=torch.float64, device=dev) for n in shape],
                                         indexing="ij")]
    moves, e = [], torch.zeros((B,) + shape, dtype=torch.float64, device=dev)
    for step, rate in _transitions(kind, th, c):
        src, dst = _sides(step)
        r = rate.expand((B,) + shape)[(slice(None),) + src]
        e[(slice(None),) + src] += r
        moves.append(((slice(None),) + src, (slice(None),) + dst, r))
    omega = 1.1 * e.reshape(B, -1).amax(dim=1)
    om = omega.reshape(-1, *[1] * len(shape))
    moves = [(s, d, (r / om).contiguous()) for s, d, r in moves]
    stay = 1.0 - e / om
    kmax, chunk = _schedule(omega, torch.tensor(times, dtype=torch.float64, device=dev))
    rho = torch.tensor(rho0, dtype=torch.float64, device=dev).reshape((1,) + shape).expand((B,) + shape).contiguous()
    nxt = torch.empty_like(rho)
    idx = None if states is None else torch.tensor(states, dtype=torch.int64, device=dev)
    S = math.prod(shape) if states is None else len(states)
    acc = torch.zeros((B, len(times), S), dtype=torch.float64, device=dev)
    L = int(max(1, min(64, 2e9 // (8 * B * S))))
    hist = torch.empty((B, L, S), dtype=torch.float64, device=dev)
    k = 0
    while k <= kmax:
        w = chunk(k, k + L)
        used = torch.nonzero(w.abs().amax(dim=(0, 2)) > 0).reshape(-1)
        for j in range(L):
            if len(used):
                flat = rho.reshape(B, -1)
                hist[:, j] = flat if idx is None else flat.index_select(1, idx)
            torch.mul(rho, stay, out=nxt)
            for s, d, r in moves:
                nxt[d].addcmul_(rho[s], r)
            rho, nxt = nxt, rho
        if len(used):
            acc[:, used] += torch.bmm(w[:, used], hist)
        k += L
    return acc


def _philox(c0, c1, c2, key):
    """Word 0 of Philox4x32-10 blocks (c0, c1, c2, 0)."""
    u = np.uint64
    lo32 = u(0xFFFFFFFF)
    x = [np.asarray(v, dtype=u) for v in np.broadcast_arrays(c0, c1, c2, 0)]
    k0, k1 = u(key & 0xFFFFFFFF), u(key >> 32)
    for _ in range(10):
        p0, p1 = u(0xD2511F53) * x[0], u(0xCD9E8D57) * x[2]
        x = [(p1 >> u(32)) ^ x[1] ^ k0, p1 & lo32, (p0 >> u(32)) ^ x[3] ^ k1, p0 & lo32]
        k0, k1 = (k0 + u(0x9E3779B9)) & lo32, (k1 + u(0xBB67AE85)) & lo32
    return x[0]


def _train64(case, seed):
    psi, y = _train_data(case, seed)
    net = surrogate.MLP(seed=seed)  # the network's first weights are an input
    p = torch.tensor(net.get_params()[0].astype(np.float64), device="cuda")
    norm = np.concatenate([psi.mean(0), psi.std(0), [y.mean()], [y.std()]])
    X = torch.tensor((psi - psi.mean(0)) / psi.std(0), device="cuda")
    t = torch.tensor((y - y.mean()) / y.std(), device="cuda")
    n, b = case["rows"], case["batch"]
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    losses = []
    for s in range(case["steps"]):
        if b >= n:
            xb, tb = X, t
        else:
            w = _philox(np.arange(b), s, 0x4D4C5001, seed)
            rows = torch.from_numpy(((w * np.uint64(n)) >> np.uint64(32)).astype(np.int64)).cuda()
            xb, tb = X[rows], t[rows]
        q = p.clone().requires_grad_(True)
        h = torch.tanh(xb @ q[:512].reshape(4, 128) + q[512:640])
        h = torch.tanh(h @ q[640:17024].reshape(128, 128) + q[17024:17152])
        loss = ((h @ q[17152:17280] + q[17280] - tb) ** 2).mean()
        loss.backward()
        g = q.grad
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        p = p - 2e-3 * (m / (1 - 0.9 ** (s + 1))) / (torch.sqrt(v / (1 - 0.999 ** (s + 1))) + 1e-8)
        losses.append(loss.detach())
    return dict(losses=torch.stack(losses), params=p, norm=norm)


def exact(case, seed):
    path = case["path"]
    if path in ("series", "loglik"):
        d = _data(case, seed)
        if path == "series":
            return _series64(d["kind"], case["d0"], case["d1"], [d["theta"]], d["times"], d["rho0"], None)[0]
        mem = [np.stack(groups) for groups, _ in d["obs"]]
        states, where = np.unique(np.concatenate([m.ravel() for m in mem]), return_inverse=True)
        acc = _series64(d["kind"], case["d0"], case["d1"], d["thetas"], d["times"], d["rho0"], states)
        ll = torch.zeros(len(d["thetas"]), dtype=torch.float64, device="cuda")
        at = 0
        for i, (_, counts) in enumerate(d["obs"]):
            cols = torch.from_numpy(where[at:at + mem[i].size].reshape(mem[i].shape)).cuda()
            at += mem[i].size
            ll += torch.log(acc[:, i][:, cols].sum(dim=2)) @ torch.tensor(counts, device="cuda")
        return ll.cpu().numpy() if case["host"] else ll
    if path == "batch":
        N, theta, t = _batch_data(case, seed)
        x = 1.1 * (theta[:, 0] + theta[:, 1] * (N - 2)) * t
        # Jump by jump on the padded batch: small batches only.
        if (x.max() + 6 * math.sqrt(x.max())) * (5e-5 + 5e-11 * case["n"] * N.max()) > 15.0:
            return None
        dev = torch.device("cuda")
        Nt, W = torch.tensor(N, device=dev)[:, None], int(N.max())
        s = torch.arange(W, dtype=torch.float64, device=dev)[None, :]
        beta, gamma = (torch.tensor(theta[:, i], device=dev)[:, None] for i in (0, 1))
        up = beta * (s < Nt - 1)
        dn = gamma * s * (s < Nt)
        omega = 1.1 * (up + dn).amax(dim=1)
        stay, up, dn = 1.0 - (up + dn) / omega[:, None], up / omega[:, None], dn / omega[:, None]
        rows = []
        kmax = 0
        for j in range(len(N)):
            k, ch = _schedule(omega[j:j + 1], torch.tensor([t[j]], device=dev))
            rows.append(ch)
            kmax = max(kmax, k)
        rho = torch.zeros((len(N), W), dtype=torch.float64, device=dev)
        rho[:, 0] = 1.0
        acc = torch.zeros_like(rho)
        for k0 in range(0, kmax + 1, 64):
            w = torch.cat([ch(k0, k0 + 64)[0] for ch in rows])
            some = bool((w.amax() > 0).item())
            for j in range(64):
                if some:
                    acc.addcmul_(rho, w[:, j:j + 1])
                y = rho * stay
                y[:, 1:].addcmul_(rho[:, :-1], up[:, :-1])
                y[:, :-1].addcmul_(rho[:, 1:], dn[:, 1:])
                rho = y
        return acc[s.expand_as(acc) < Nt]
    if path == "csr":
        ptr, col, rate, rho0, times = _csr_data(case, seed)
        n, dev = case["n"], torch.device("cuda")
        row = torch.from_numpy(np.repeat(np.arange(n), np.diff(ptr))).to(dev)
        c, r = torch.from_numpy(col.astype(np.int64)).to(dev), torch.from_numpy(rate).to(dev)
        e = torch.zeros(n, dtype=torch.float64, device=dev).index_add_(0, row, r)
        omega = 1.1 * e.max()
        order = torch.argsort(c, stable=True)
        bptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
        bptr[1:] = torch.cumsum(torch.bincount(c, minlength=n), 0)
        Bt = torch.sparse_csr_tensor(bptr, row[order], (r / omega)[order], size=(n, n))
        stay = 1.0 - e / omega
        kmax, chunk = _schedule(omega.reshape(1), torch.tensor(times, device=dev))
        w = chunk(0, kmax + 1)[0]
        rho = torch.from_numpy(rho0).to(dev)
        acc = torch.zeros((len(times), n), dtype=torch.float64, device=dev)
        for k in range(kmax + 1):
            acc += w[:, k:k + 1] * rho
            rho = rho * stay + Bt @ rho
        return acc
    if path == "train":
        return _train64(case, seed)
    return None  # a chain's accept decisions have no 64-bit value of their own
