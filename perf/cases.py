"""The calls that users of this library make, as timed cases.

Every case is one call of a public entry point on data shaped like the paper's
(coupled logistic maps and vector autoregressive processes on a random
directed graph): target process 0, its present as Y, its own past and some
sources' past as Z, candidate sources' past as X.  `kind` names the entry
point; the sizes are plain numbers.
"""
import math

import numpy as np
import torch

import paper_1902_06828_gb300 as te


def listed():
    return [
        # one estimate on a short series, no surrogates: the smallest call, all latency
        dict(name="call_T203", kind="call", proc="var", n=3, T=203, max_lag=2, dx=1, dz=2, cands=1,
             S=0, k=4, theiler=0),
        # one estimate and its 200 surrogates on a 3-node VAR, T = 1000
        dict(name="call_T1000_S200", kind="call", proc="var", n=3, T=1000, max_lag=2, dx=1, dz=2,
             cands=1, S=200, k=4, theiler=0),
        # the same test at the paper's largest sample size: one request of a target's loop
        dict(name="call_T10000_S200", kind="call", proc="var", n=10, T=10000, max_lag=5, dx=1,
             dz=1, cands=1, S=200, k=4, theiler=0),
        # a batch of one source test: every candidate of a 10-node VAR with its surrogates
        dict(name="batch_var_T10000", kind="batch", proc="var", n=10, T=10000, max_lag=5, dx=1,
             dz=2, cands=45, S=200, k=4, theiler=0),
        # a late source test on coupled logistic maps: eight variables selected already
        dict(name="batch_clm_T10000_dz8", kind="batch", proc="clm", n=20, T=10000, max_lag=5,
             dx=1, dz=8, cands=89, S=200, k=4, theiler=0),
        # the omnibus test: all selected sources' rows as one block X
        dict(name="omnibus_T10000", kind="call", proc="clm", n=10, T=10000, max_lag=5, dx=3, dz=2,
             cands=1, S=200, k=4, theiler=0),
        # a source test with a Theiler window (autocorrelated recordings), odd length, k = 4
        dict(name="theiler_T2999", kind="batch", proc="var", n=10, T=2999, max_lag=5, dx=1, dz=3,
             cands=9, S=200, k=4, theiler=12),
        # the allocation-free entry point, as a latency-bound loop calls it
        dict(name="static_T1000_S200", kind="static", proc="var", n=5, T=1000, max_lag=5, dx=1,
             dz=2, cands=1, S=200, k=4, theiler=0),
        # linear-Gaussian estimate with 1000 surrogates, few conditioning variables
        dict(name="gauss_T10000_dz4", kind="gauss", proc="var", n=100, T=10000, max_lag=5, dx=1,
             dz=4, cands=1, S=1000, k=4, theiler=0),
        # the same at the widest conditioning set (40 joint dimensions)
        dict(name="gauss_T10000_dz38", kind="gauss", proc="var", n=100, T=10000, max_lag=5, dx=1,
             dz=38, cands=1, S=1000, k=4, theiler=0),
        # a whole Gaussian network, every target
        dict(name="gauss_network_T10000", kind="gauss_network", proc="var", n=10, T=10000,
             max_lag=5, dx=1, dz=0, cands=0, S=200, k=4, theiler=0),
        # a whole KSG network, every target: all four steps of the greedy loop
        dict(name="ksg_network_T3000", kind="ksg_network", proc="clm", n=10, T=3000, max_lag=5,
             dx=1, dz=0, cands=0, S=200, k=4, theiler=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["call", "call", "call", "batch", "batch", "batch", "static", "gauss",
                       "gauss", "gauss_network", "ksg_network"])
    c = dict(kind=kind, proc=rng.choice(["var", "clm"]), n=_log(rng, 3, 20), T=_log(rng, 200, 10000),
             max_lag=rng.randint(2, 5), dx=1, dz=0, cands=1, S=0, k=4, theiler=0)
    if kind in ("call", "batch", "static"):
        c["k"] = rng.choice([4, 4, 4, 4, rng.randint(1, 12)])
        c["theiler"] = rng.choice([0, 0, 0, 0, rng.randint(1, 25)])
        c["dz"] = rng.randint(0, min(10, (c["n"] - 1) * c["max_lag"] - 2))
    if kind == "call":
        c["S"] = rng.choice([0, _log(rng, 20, 1000)])
        if rng.random() < 0.3 and c["n"] > 3:
            c["dx"], c["S"] = rng.randint(2, 4), min(c["S"], 200)
            c["dz"] = min(c["dz"], 5)
            c["n"] = max(c["n"], 6)
    elif kind == "batch":
        c["S"] = _log(rng, 20, 500)
        pool = (c["n"] - 1) * c["max_lag"] - c["dz"]
        # members x points^2 at most half the largest listed batch's
        most = int(89 * 201 * 9995 ** 2 / 2 / (c["S"] + 1) / c["T"] ** 2)
        if c["theiler"]:
            most //= 16
        c["cands"] = max(1, min(pool, most, _log(rng, 2, 95)))
    elif kind == "static":
        c["T"] = _log(rng, 200, 5000)
        c["S"] = _log(rng, 20, 400)
        c["dz"] = min(c["dz"], 6)
    elif kind == "gauss":
        c["proc"], c["n"], c["T"] = "var", rng.randint(20, 100), _log(rng, 500, 10000)
        c["S"], c["dz"] = _log(rng, 100, 1000), rng.randint(0, 38)
        c["dx"] = rng.choice([1, 1, 1, 2])
        c["dz"] = min(c["dz"], 39 - c["dx"])
    else:
        c["proc"] = "var" if kind == "gauss_network" else c["proc"]
        c["S"] = rng.randint(100, 200)
        c["n"] = rng.randint(3, 10)
        c["T"] = _log(rng, 300, 2500 if kind == "ksg_network" else 10000)
    return c


def _series(case, seed):
    """float32 [n][T]: the paper's validation processes (self-coupling 0.5, one
    random lag 1..5 per source, three sources per target on average), the
    graph fixed by the size and the noise by the seed, standardised."""
    n, T, L, burn = case["n"], case["T"], 5, 300
    g = np.random.default_rng(1000 + n)
    adj = g.random((n, n)) < min(0.5, 3.0 / n)
    np.fill_diagonal(adj, False)
    src, tgt = np.nonzero(adj)
    lag = g.integers(1, L + 1, src.size)
    indeg = np.maximum(np.bincount(tgt, minlength=n), 1)
    clm = case["proc"] == "clm"
    rng = np.random.default_rng(seed)
    buf = np.zeros((T + burn + L, n))
    buf[:L] = rng.random((L, n)) if clm else rng.normal(size=(L, n))
    eta = rng.normal(0.0, 0.1 if clm else 1.0, size=buf.shape)
    wts = (0.5 if clm else 0.4) / indeg[tgt]
    flat = buf.reshape(-1)
    off = src - lag * n
    for t in range(L, buf.shape[0]):
        a = 0.5 * buf[t - 1]
        if src.size:
            a = a + np.bincount(tgt, weights=wts * flat[off + t * n], minlength=n)
        if clm:
            a = 4.0 * a * (1.0 - a) + eta[t]
            buf[t] = a - np.floor(a)
        else:
            buf[t] = a + eta[t]
    x = buf[-T:].T
    x = (x - x.mean(1, keepdims=True)) / x.std(1, keepdims=True)
    x = x + rng.normal(0.0, 1e-8, size=x.shape)
    return np.ascontiguousarray(x, dtype=np.float32)


def _variables(case):
    """Target 0's present as Y; Z = its own lags 1 and 2, then sources'
    past; the X candidates are the next variables of the sources."""
    n, L = case["n"], case["max_lag"]
    own = [(0, 1), (0, 2)][:min(2, L)]
    pool = [(q, 1 + (q + r) % L) for r in range(L) for q in range(1, n)]
    z = (own + pool)[:case["dz"]]
    rest = [v for v in pool if v not in z]
    xs = [rest[a * case["dx"]:(a + 1) * case["dx"]] for a in range(max(case["cands"], 1))]
    return xs, [(0, 0)], z


def prepare(case, seed):
    series = _series(case, seed)
    xs, y, z = _variables(case)
    st = dict(case=case, xs=xs, y=y, z=z, seed=seed)
    if case["kind"] == "static":
        st["series"] = torch.from_numpy(series).cuda()
        return st
    st["ctx"] = te.Context(0)
    st["data"] = te.te_data_create(st["ctx"], series)
    if case["kind"] == "batch":
        st["jobs"] = [te.Job(st["data"], x, y, z, k=case["k"], theiler=case["theiler"],
                             max_lag=case["max_lag"], n_surr=case["S"], seed=seed, stream_tag=3)
                      for x in xs]
    return st


def run(st):
    c = st["case"]
    kind = c["kind"]
    common = dict(max_lag=c["max_lag"], n_surr=c["S"], seed=st["seed"], stream_tag=3)
    if kind == "call":
        return te.cmi_ksg(st["ctx"], st["data"], st["xs"][0], st["y"], st["z"], k=c["k"],
                          theiler=c["theiler"], **common)
    if kind == "static":
        return te.cmi_ksg_static(st["series"], st["xs"][0], st["y"], st["z"], k=c["k"],
                                 theiler=c["theiler"], **common)
    if kind == "batch":
        return np.stack(te.cmi_ksg_batch(st["ctx"], st["jobs"]))
    if kind == "gauss":
        return te.cmi_gauss(st["ctx"], st["data"], st["xs"][0], st["y"], st["z"], **common)
    net = te.te_network_infer(st["ctx"], st["data"], k=c["k"], max_lag_target=c["max_lag"],
                              max_lag_sources=c["max_lag"], n_surr=c["S"], seed=st["seed"],
                              estimator="gauss" if kind == "gauss_network" else "ksg")
    tg = net["targets"]
    chosen = np.zeros((2, c["n"], c["n"], c["max_lag"] + 1), np.int32)   # [past | sources][target]
    for t in tg:
        for a, sel in enumerate((t["sel_target"], t["sel_sources"])):
            for q, l in sel:
                chosen[a, t["target"], q, l] = 1
    return dict(adjacency=net["adjacency"], min_lag=net["min_lag"],
                omnibus_cmi=np.array([t["omnibus_cmi"] for t in tg]),
                omnibus_p=np.array([t["omnibus_p"] for t in tg]),
                selected=chosen,
                n_estimates=np.array([t["n_estimates"] for t in tg]))


def work(case):
    """Bytes: the series columns that the call reads and its results.  Flops:
    for KSG the comparisons of one neighbour search and three range counts
    per estimate and point by an ordered structure, log2 N each; for the
    Gaussian estimator the covariances.  A network counts one test of each of
    the first two steps per target (what it does beyond that depends on the data)."""
    N = case["T"] - case["max_lag"]
    dims = case["dx"] * case["cands"] + 1 + case["dz"]
    members = case["cands"] * (case["S"] + 1)
    dw = 1 + case["dz"]
    if case["kind"].endswith("network"):
        members = case["n"] * case["n"] * case["max_lag"] * (case["S"] + 1)
        dims, dw = case["n"], 2
    if case["kind"].startswith("gauss"):
        flops = 2.0 * N * dw * (members * case["dx"] + dw)
    else:
        flops = 4.0 * members * N * math.log2(N)
    return {"bytes": 4.0 * dims * N + 8.0 * members, "flops": flops}


def _permutations(seed, tag, S, N):
    """[S][N] Fisher-Yates permutations, SplitMix64 keyed by (seed, tag, 0, 0, s)."""
    m64 = (1 << 64) - 1
    gamma = 0x9E3779B97F4A7C15

    def mix(v):
        v = (v ^ (v >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        v = (v ^ (v >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return v ^ (v >> np.uint64(31))

    def once(v):
        return int(mix(np.array([(v + gamma) & m64], np.uint64))[0])

    h = once(once(once(seed ^ tag)))
    state = np.array([once(h ^ s) for s in range(1, S + 1)], np.uint64)
    p = np.tile(np.arange(N)[:, None], (1, S))
    cols = np.arange(S)
    lo32 = np.uint64(0xFFFFFFFF)
    for i in range(N - 1, 0, -1):
        r = mix(state + np.uint64(((N - i) * gamma) & m64))
        w = np.uint64(i + 1)
        j = (((r >> np.uint64(32)) * w + ((r & lo32) * w >> np.uint64(32))) >> np.uint64(32))
        j = j.astype(np.int64)
        a = p[i].copy()
        p[i] = p[j, cols]
        p[j, cols] = a
    return p.T


def exact(case, seed):
    kind, S = case["kind"], case["S"]
    N = case["T"] - case["max_lag"]
    if kind.endswith("network"):
        return None
    if kind != "gauss" and (S + 1) * case["cands"] * N * N > 2.5e8:
        return None
    series = _series(case, seed).astype(np.float64)
    xs, y, z = _variables(case)
    L, k = case["max_lag"], case["k"]
    col = lambda v: series[v[0], L - v[1]:case["T"] - v[1]]
    Y, Z = np.array([col(v) for v in y]), np.array([col(v) for v in z]).reshape(len(z), N)
    perms = _permutations(seed, 3, S, N) if S else np.zeros((0, N), np.int64)
    order = [np.arange(N)] + list(perms)
    if kind == "gauss":
        X = np.array([col(v) for v in xs[0]])
        X = X - X.mean(1, keepdims=True)
        W = np.concatenate([Y, Z])
        W = W - W.mean(1, keepdims=True)
        sxx, sww = X @ X.T / (N - 1), W @ W.T / (N - 1)
        dy, out = len(y), np.zeros(S + 1)
        inv_w = np.linalg.inv(sww)
        inv_z = np.linalg.inv(sww[dy:, dy:]) if len(z) else np.zeros((0, 0))
        for s, p in enumerate(order):
            cw = X[:, p] @ W.T / (N - 1)
            cz = cw[:, dy:]
            out[s] = 0.5 * (np.linalg.slogdet(sxx - cz @ inv_z @ cz.T)[1]
                            - np.linalg.slogdet(sxx - cw @ inv_w @ cw.T)[1])
        return out, None
    psi = np.concatenate([[0.0], -np.euler_gamma + np.concatenate([[0.0], np.cumsum(1.0 / np.arange(1, N + 1))])])
    gap = np.abs(np.arange(N)[:, None] - np.arange(N)[None, :])
    masked = gap <= case["theiler"]

    def dist(rows):
        d = np.full((N, N), -np.inf)
        for r in rows:
            d = np.maximum(d, np.abs(r[:, None] - r[None, :]))
        d[masked] = np.inf
        return d

    dz_ = dist(Z)
    dyz = np.maximum(dz_, dist(Y))
    res = []
    for x in xs:
        X = np.array([col(v) for v in x])
        out = np.zeros(S + 1)
        for s, p in enumerate(order):
            dx = dist(X[:, p])
            eps = np.partition(np.maximum(dx, dyz), k - 1, axis=1)[:, k - 1:k]
            nz, nyz, nxz = ((d < eps).sum(1) for d in (dz_, dyz, np.maximum(dx, dz_)))
            out[s] = psi[k] + np.mean(psi[nz + 1] - psi[nxz + 1] - psi[nyz + 1])
        res.append(out)
    return np.stack(res) if kind == "batch" else res[0]
