"""Measured cases: the calls a user of this package makes, over the sizes they are made at.

Each case is one call of a public entry point (:mod:`paper_2408_05459_gb300.ancka`) on inputs that are
already on the GPU, as a program that holds its network in device memory makes it.  The inputs are drawn
on the GPU with torch, in the shapes of the package's own workloads (``synth.py``): Gaussian-mixture and
TF-IDF-like attributes, stochastic-block-model graphs, multiplex graphs, hypergraphs with power-law
hyperedge sizes and degree-corrected graphs with power-law degrees.

``call`` names the entry point: ``knn`` and ``knn_ivf`` (the attribute neighbours alone), ``cluster``
(Algorithm 4 from attributes and topology to labels), ``discretize`` (labels from a given block),
``warm_gradients`` (one forward and backward pass of the learned start) and ``warm_predict`` (its forward
pass alone).
"""
import math

import numpy as np
import torch

from paper_2408_05459_gb300 import ancka

DEV = "cuda"


def listed():
    return [
        # a small attributed network (the parity size): every launch and copy of the KNN call shows
        dict(name="knn-small", call="knn", n=2000, d=128, K=10, prec="bf16", attrs="mixture", k=5, sigma=1.5),
        # K = 50, the neighbourhood the method uses on small networks, on sparse text attributes
        dict(name="knn-small-k50", call="knn", n=3001, d=500, K=50, prec="bf16", attrs="tfidf", k=7),
        # the attributes of the 100k-node hypergraph: sparse, with many equal cosines
        dict(name="knn-tfidf", call="knn", n=100_000, d=500, K=10, prec="bf16", attrs="tfidf", k=10),
        # the FP8 contraction (the other tensor-core precision), an odd number of rows
        dict(name="knn-fp8", call="knn", n=100_003, d=256, K=10, prec="fp8", attrs="mixture", k=20, sigma=2.0),
        # large and narrow: the contraction of the large graph at half its rows
        dict(name="knn-large", call="knn", n=1_200_000, d=100, K=10, prec="bf16", attrs="mixture", k=47, sigma=1.5),
        # approximate neighbours by inverted lists, the choice for large graphs
        dict(name="knn-ivf", call="knn_ivf", n=600_000, d=100, K=10, nlist=500, nprobe=8, attrs="mixture", k=47,
             sigma=1.5),
        # the whole method on a small graph: latency
        dict(name="cluster-small", call="cluster", topo="graph", n=2000, d=128, k=5, deg=5.6, inside=0.71, K=10, T=10,
             T_i=25, beta=0.5, attrs="mixture", sigma=1.5),
        # the whole method on the hypergraph (keyword / co-authorship type)
        dict(name="cluster-hypergraph", call="cluster", topo="hypergraph", n=100_000, m=200_000, d=500, k=10, K=10,
             T=10, T_i=25, beta=0.5, attrs="tfidf"),
        # the whole method on a three-layer multiplex graph
        dict(name="cluster-multiplex", call="cluster", topo="multiplex", n=500_000, d=256, k=20, deg=20.0, K=10, T=8,
             T_i=25, beta=0.5, attrs="mixture", sigma=2.0),
        # the whole method at the largest size: a co-purchase-scale graph with power-law degrees
        dict(name="cluster-large", call="cluster", topo="powerlaw", n=2_400_000, d=100, k=47, deg=50.0, inside=0.8,
             K=10, T=10, T_i=1, beta=0.4, attrs="mixture", sigma=1.5),
        # labels from a block a caller already holds, at the large graph's size
        dict(name="discretize-large", call="discretize", n=2_400_000, k=47, noise=0.05),
        # a training step of the learned start at its training size (gradients: Adam's first updates follow
        # the sign of a gradient alone, so updated weights say nothing about how close two gradients are)
        dict(name="warm-gradients", call="warm_gradients", topo="multiplex", n=200_000, d=256, k=20, deg=20.0,
             attrs="mixture", sigma=2.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    call = rng.choice(["knn", "knn", "knn", "knn_ivf", "cluster", "cluster", "discretize", "warm_gradients",
                       "warm_predict"])
    if call == "knn":
        attrs = rng.choice(["mixture", "mixture", "tfidf"])
        prec = rng.choice(["bf16", "bf16", "bf16", "fp8", "fp32"])
        K = rng.choice([1, 5, 8, 10, 10, 10, 12, 15, 25, 50])
        d = rng.randint(60, 512) if attrs == "tfidf" else rng.randint(16, 512)
        if K > 12:
            n = _log(rng, 500, 4000)
        elif prec == "fp32":
            n = _log(rng, 500, 20_000)
        else:
            n = _log(rng, 500, min(1_000_000, int(math.sqrt(1.0e14 / d))))
        c = dict(call=call, n=n, d=d, K=K, prec=prec, attrs=attrs, k=rng.randint(2, 50))
        if attrs == "mixture":
            c["sigma"] = rng.choice([1.0, 1.5, 2.0])
        return c
    if call == "knn_ivf":
        n = _log(rng, 20_000, 800_000)
        nlist = max(8, n // rng.choice([600, 1200, 2400]))
        return dict(call=call, n=n, d=rng.randint(32, 256), K=rng.choice([5, 10, 16]), nlist=min(1000, nlist),
                    nprobe=rng.choice([4, 8, 16]) if nlist >= 16 else 4, attrs="mixture", k=rng.randint(5, 50),
                    sigma=rng.choice([1.0, 1.5]))
    if call == "cluster":
        topo = rng.choice(["graph", "hypergraph", "multiplex", "powerlaw"])
        n = _log(rng, 1000, 200_000)
        c = dict(call=call, topo=topo, n=n, k=rng.randint(3, 24), K=10, T=rng.randint(5, 12),
                 T_i=rng.choice([1, 10, 25]), beta=rng.choice([0.4, 0.5]))
        if topo == "hypergraph":
            c.update(m=2 * n + rng.randint(0, 99), d=rng.randint(200, 512), attrs="tfidf")
        else:
            c.update(d=rng.randint(32, 300), attrs="mixture", sigma=1.5, deg=float(rng.randint(8, 40)))
            if topo != "multiplex":
                c["inside"] = rng.choice([0.7, 0.8, 0.9])
        return c
    if call == "discretize":
        return dict(call=call, n=_log(rng, 2000, 2_400_000), k=rng.randint(2, 64), noise=rng.choice([0.03, 0.05]))
    return dict(call=call, topo="multiplex", n=_log(rng, 2000, 300_000), d=rng.randint(16, 300), k=rng.randint(2, 40),
                deg=float(rng.randint(5, 20)), attrs="mixture", sigma=2.0)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _rand(g, *shape, dtype=torch.float32):
    return torch.rand(*shape, generator=g, device=DEV, dtype=dtype)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _labels(g, n, sizes):
    """Planted cluster of every node (ids carry no order) and the nodes of each cluster in turn."""
    order = torch.randperm(n, generator=g, device=DEV)
    lab = torch.empty(n, dtype=torch.int64, device=DEV)
    lab[order] = torch.repeat_interleave(torch.arange(len(sizes), device=DEV), torch.as_tensor(sizes, device=DEV))
    return lab, order


def _sizes(n, k, zipf):
    if zipf:
        w = 1.0 / np.arange(1, k + 1)
        s = np.maximum(1, np.floor(n * w / w.sum())).astype(np.int64)
        s[0] += n - s.sum()
    else:
        s = np.full(k, n // k, np.int64)
        s[: n - s.sum()] += 1
    return s


def _attributes(case, g, lab):
    n, d, k = case["n"], case["d"], case["k"]
    if case["attrs"] == "mixture":
        mu = _randn(g, k, d)
        X = _randn(g, n, d) * case["sigma"]
        for s in range(0, n, 1 << 18):
            X[s:s + (1 << 18)] += mu[lab[s:s + (1 << 18)]]
        return X
    # TF-IDF-like: 2% distinct words a row, 0.7 cluster Zipf(1.1) + 0.3 background Zipf(1.1), tf * log(n / df)
    words = max(3, d // 50)
    base = 1.0 / torch.arange(1, d + 1, device=DEV, dtype=torch.float32) ** 1.1
    base = base / base.sum()
    logp = torch.empty(k, d, device=DEV)
    background = base[torch.randperm(d, generator=g, device=DEV)]
    for c in range(k):
        logp[c] = torch.log(0.7 * base[torch.randperm(d, generator=g, device=DEV)] + 0.3 * background)
    cols = torch.empty(n, words, dtype=torch.int64, device=DEV)
    for s in range(0, n, 1 << 16):
        lb = lab[s:s + (1 << 16)]
        gumbel = -torch.log(-torch.log(_rand(g, lb.numel(), d).clamp_(1e-20, 1 - 1e-7)))
        cols[s:s + lb.numel()] = torch.topk(logp[lb] + gumbel, words, dim=1).indices
    tf = 1.0 + torch.poisson(torch.full((n, words), 0.5, device=DEV), generator=g)
    df = torch.bincount(cols.reshape(-1), minlength=d).clamp_(min=1).float()
    X = torch.zeros(n, d, device=DEV)
    X.scatter_(1, cols, tf * torch.log(n / df + 1e-3)[cols])
    return X


def _csr(n, src, dst):
    """Symmetric, duplicate-free, loop-free adjacency, columns sorted in each row."""
    keep = src != dst
    src, dst = src[keep], dst[keep]
    key = torch.unique(torch.cat([src * n + dst, dst * n + src]))
    row = torch.div(key, n, rounding_mode="floor")
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return ptr, (key - row * n).to(torch.int32)


def _sbm(g, n, lab, order, sizes, deg, inside):
    """Edges of mean degree deg, a share `inside` of them within a cluster."""
    e = int(n * deg / 2)
    off = torch.as_tensor(np.concatenate([[0], np.cumsum(sizes)]), device=DEV)
    u = torch.randint(0, n, (e,), generator=g, device=DEV)
    c = lab[u]
    size = (off[1:] - off[:-1])[c]
    mate = order[off[c] + torch.minimum((_rand(g, e, dtype=torch.float64) * size).long(), size - 1)]
    other = torch.randint(0, n, (e,), generator=g, device=DEV)
    return _csr(n, u, torch.where(_rand(g, e) < inside, mate, other))


def _powerlaw(g, n, order, sizes, deg, inside):
    """Degree-corrected edges: power-law propensities (exponent 2.5), clusters by squared mass."""
    e = int(n * deg / 2)
    theta = (1.0 - _rand(g, n, dtype=torch.float64)).pow(-1.0 / 1.5).clamp_(max=math.sqrt(2.0 * e))
    cdf = torch.cumsum(theta, 0)  # in the order of `order`: cluster by cluster
    ends = cdf[torch.as_tensor(np.cumsum(sizes) - 1, device=DEV)]
    begins = torch.cat([torch.zeros(1, dtype=torch.float64, device=DEV), ends[:-1]])
    mass = ends - begins
    e_in = int(round(inside * e))
    pc = torch.cumsum(mass ** 2, 0)
    c = torch.searchsorted(pc, _rand(g, e_in, dtype=torch.float64) * pc[-1]).clamp_(max=len(sizes) - 1)

    def pick(lo, span, count):
        at = torch.searchsorted(cdf, lo + _rand(g, count, dtype=torch.float64) * span)
        return order[at.clamp_(max=n - 1)]

    src = torch.cat([pick(begins[c], mass[c], e_in), pick(0.0, cdf[-1], e - e_in)])
    dst = torch.cat([pick(begins[c], mass[c], e_in), pick(0.0, cdf[-1], e - e_in)])
    return _csr(n, src, dst)


def _topology(case, g, lab, order, sizes):
    """The device topology dict, laid out as ancka.topology_to_device returns it."""
    n, k = case["n"], case["k"]
    if case["topo"] == "hypergraph":
        m = case["m"]
        p = torch.arange(2, 21, device=DEV, dtype=torch.float32) ** -2.5
        esz = 2 + torch.multinomial(p, m, replacement=True, generator=g)
        home = torch.randint(0, k, (m,), generator=g, device=DEV)
        eid = torch.repeat_interleave(torch.arange(m, device=DEV), esz)
        t = eid.numel()
        away = torch.randint(0, max(1, k - 1), (t,), generator=g, device=DEV)
        h = home[eid]
        c = torch.where(_rand(g, t) < 0.85, h, (away + (away >= h)).clamp_(max=k - 1))
        off = torch.as_tensor(np.concatenate([[0], np.cumsum(sizes)]), device=DEV)
        size = (off[1:] - off[:-1])[c]
        node = order[off[c] + torch.minimum((_rand(g, t, dtype=torch.float64) * size).long(), size - 1)]
        key = torch.unique(eid * n + node)
        e = torch.div(key, n, rounding_mode="floor")
        ptr = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
        ptr[1:] = torch.cumsum(torch.bincount(e, minlength=m), 0)
        return dict(kind="hypergraph", n=n, directed=0, he_ptr=ptr, he_nodes=(key - e * n).to(torch.int32), m=m)
    if case["topo"] == "multiplex":  # in/out probability ratios 8, 4, 2
        layers = [_sbm(g, n, lab, order, sizes, case["deg"], (r - 1.0) / (r + k - 1.0)) for r in (8.0, 4.0, 2.0)]
    elif case["topo"] == "graph":
        layers = [_sbm(g, n, lab, order, sizes, case["deg"], case["inside"])]
    else:
        layers = [_powerlaw(g, n, order, sizes, case["deg"], case["inside"])]
    ptrs, base = [], 0
    for ptr, col in layers:
        ptrs.append(ptr + base)
        base += col.numel()
    return dict(kind="multiplex" if case["topo"] == "multiplex" else "graph", n=n, directed=0,
                row_ptr=torch.cat(ptrs), col_idx=torch.cat([c for _, c in layers]), L=len(layers), nnz=base)


def _block(case, g):
    """A block like the iteration's: cluster indicators plus noise, turned a little, rows of a wider block."""
    n, k = case["n"], case["k"]
    lab, _ = _labels(g, n, _sizes(n, k, True))
    turn = torch.linalg.qr(torch.eye(k, device=DEV) + 0.3 / math.sqrt(k) * _randn(g, k, k)).Q
    Q = torch.empty(n, k + 1, device=DEV)
    Q[:, 0] = 1.0 / math.sqrt(n)
    for s in range(0, n, 1 << 19):
        B = case["noise"] * _randn(g, min(n - s, 1 << 19), k)
        B.scatter_add_(1, lab[s:s + B.shape[0], None], torch.full((B.shape[0], 1), 0.3, device=DEV))
        Q[s:s + B.shape[0], 1:] = B @ turn
    return Q


def prepare(case, seed):
    g = _gen(seed)
    if case["call"] == "discretize":
        return dict(case=case, Q=_block(case, g))
    n, k = case["n"], case["k"]
    sizes = _sizes(n, k, case.get("topo") == "powerlaw")
    lab, order = _labels(g, n, sizes)
    st = dict(case=case, X=_attributes(case, g, lab))
    if "topo" in case:
        st["topo"] = _topology(case, g, lab, order, sizes)
    if case["call"] == "cluster":
        st["params"] = ancka.default_params(k=k, K=case["K"], T=case["T"], T_i=case["T_i"], beta=case["beta"],
                                            knn_prec="bf16")
    if case["call"].startswith("warm"):
        d_in = 2 * case["d"]
        st["weights"] = dict(W1=_randn(g, d_in, 256) * math.sqrt(2.0 / d_in), b1=torch.zeros(256, device=DEV),
                             W2=_randn(g, 256, k) / 16.0, b2=torch.zeros(k, device=DEV))
        # the target: an orthonormal block near the planted clusters, as a clustering call returns
        B = torch.nn.functional.one_hot(lab, k).float() + 0.2 * _randn(g, n, k)
        st["Qt"] = torch.linalg.qr(B).Q.contiguous()
    return st


def run(state):
    c = state["case"]
    if c["call"] == "knn":
        idx, sim, _ = ancka.knn(state["X"], c["K"], c["prec"], with_info=False)
        return dict(idx=idx, sim=sim)
    if c["call"] == "knn_ivf":
        idx, sim, _ = ancka.knn_ivf(state["X"], c["K"], c["nlist"], c["nprobe"], with_info=False)
        return dict(idx=idx, sim=sim)
    if c["call"] == "cluster":
        labels, extras, _ = ancka.cluster(state["topo"], state["X"], state["params"], want_Q=True, with_info=False)
        return dict(labels=labels, Q=extras["Q"])
    if c["call"] == "discretize":
        labels, iters = ancka.discretize(state["Q"][:, 1:])
        return dict(labels=labels, iters=iters)
    if c["call"] == "warm_predict":
        return dict(W=ancka.warm_predict(state["topo"], state["X"], state["weights"]))
    grads, loss = ancka.warm_gradients(state["topo"], state["X"], state["Qt"], state["weights"])
    return dict(grads, loss=loss)


def work(case):
    n, k = case["n"], case["k"]
    if case["call"] == "discretize":
        return dict(bytes=4.0 * n * (k + 1), flops=4.0 * n * k * k)  # two alternations at least
    d = case["d"]
    b = 4.0 * n * d
    f = 0.0
    if case["call"] in ("knn", "cluster"):
        f += 2.0 * n * n * d
    if case["call"] == "knn_ivf":  # rows of the probed cells, and the assignment to cells
        f += 2.0 * n * d * (n * case["nprobe"] / case["nlist"] + case["nlist"])
    if case["call"].startswith("knn"):
        return dict(bytes=b + 8.0 * n * case["K"], flops=f)
    nnz = 2.0 * 3.5 * case["m"] if case["topo"] == "hypergraph" else n * case["deg"] * (3 if case["topo"] == "multiplex" else 1)
    b += 4.0 * nnz + 8.0 * n
    if case["call"] == "cluster":
        w = k + 1.0
        f += case["T"] * (2.0 * (nnz + 1.5 * n * case["K"]) * w + 4.0 * n * w * w)
        return dict(bytes=b + 4.0 * n * (w + 1), flops=f)
    d_in = 2.0 * d
    f += 2.0 * nnz * d + 2.0 * n * 256 * (d_in + k)
    if case["call"] == "warm_predict":
        return dict(bytes=b + 4.0 * n * k, flops=f)
    return dict(bytes=b + 4.0 * n * k, flops=f + 2.0 * n * 256 * (d_in + 2 * k) + 8.0 * n * k * k)


# ----------------------------------------------------------------------------
# the same in 64 bits, with torch alone
# ----------------------------------------------------------------------------
def _unit(X):
    X = X.double()
    nrm = X.norm(dim=1, keepdim=True)
    return torch.where(nrm > 0, X / nrm.clamp(min=1e-300), torch.zeros_like(X))


def _exact_knn(X, K):
    U = _unit(X)
    n = U.shape[0]
    idx = torch.empty(n, K, dtype=torch.int64, device=DEV)
    sim = torch.empty(n, K, dtype=torch.float64, device=DEV)
    step = max(1, min(n, (1 << 28) // n))
    for s in range(0, n, step):
        S = U[s:s + step] @ U.T
        r = torch.arange(S.shape[0], device=DEV)
        S[r, s + r] = -math.inf
        sim[s:s + step], idx[s:s + step] = torch.topk(S, K, dim=1)
    return idx, sim


def _coo(row, col, val, shape):
    return torch.sparse_coo_tensor(torch.stack([row, col]), val, shape, check_invariants=False).coalesce().to_sparse_csr()


def _inv(v):
    return torch.where(v > 0, 1.0 / v.clamp(min=1e-300), torch.zeros_like(v))


def _walks(t):
    """P_N as factors to apply in turn (last first), its transpose likewise, and the degrees."""
    n = t["n"]
    if t["kind"] == "hypergraph":
        m = t["m"]
        e = torch.repeat_interleave(torch.arange(m, device=DEV), t["he_ptr"][1:] - t["he_ptr"][:-1])
        v = t["he_nodes"].long()
        dv = torch.bincount(v, minlength=n).double()
        de = torch.bincount(e, minlength=m).double()
        PV, PE = (v, e, _inv(dv)[v], (n, m)), (e, v, _inv(de)[e], (m, n))
        fwd = [_coo(*PV), _coo(*PE)]
        back = [_coo(PE[1], PE[0], PE[2], (n, m)), _coo(PV[1], PV[0], PV[2], (m, n))]
        return fwd, back, dv
    rows, cols, vals, deg = [], [], [], torch.zeros(n, dtype=torch.float64, device=DEV)
    for l in range(t["L"]):
        ptr = t["row_ptr"][l * (n + 1):(l + 1) * (n + 1)]
        cnt = ptr[1:] - ptr[:-1]
        r = torch.repeat_interleave(torch.arange(n, device=DEV), cnt)
        deg += cnt
        rows.append(r)
        cols.append(t["col_idx"][int(ptr[0]):int(ptr[-1])].long())
        vals.append(_inv(cnt.double())[r] / t["L"])
    r, c, v = torch.cat(rows), torch.cat(cols), torch.cat(vals)
    return [_coo(r, c, v, (n, n))], [_coo(c, r, v, (n, n))], deg


def _apply(factors, Q):
    for M in reversed(factors):
        Q = M @ Q
    return Q


def _splitmix_sign(n, c):
    with np.errstate(over="ignore"):
        z = np.arange(n, dtype=np.uint64) * np.uint64(64) + np.uint64(c) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.as_tensor(np.where(z >> np.uint64(63) == 1, -1.0, 1.0), device=DEV)


def _exact_block(case, st):
    """The block Q of the last orthogonal iteration."""
    X, t, n, k, K = st["X"], st["topo"], case["n"], case["k"], case["K"]
    idx, _ = _exact_knn(X, K)
    U = _unit(X)
    src = torch.arange(n, device=DEV).repeat_interleave(K)
    dst = idx.reshape(-1)
    f = torch.cat([(U[src[s:s + (1 << 18)]] * U[dst[s:s + (1 << 18)]]).sum(1) for s in range(0, n * K, 1 << 18)])
    A = _coo(torch.cat([src, dst]), torch.cat([dst, src]), torch.cat([f, f]), (n, n))
    D = (A @ torch.ones(n, 1, dtype=torch.float64, device=DEV))
    fwd, back, deg = _walks(t)
    beta = torch.full((n, 1), float(np.float32(case["beta"])), dtype=torch.float64, device=DEV)
    beta[deg == 0] = 1.0
    beta[~(X != 0).any(dim=1)] = 0.0
    beta[D[:, 0] <= 0] = 0.0
    # initial labels: truncated walks from the k nodes of largest degree (ties to the smaller id)
    alpha = float(np.float32(0.2))
    centre = torch.sort(torch.sort(-deg, stable=True).indices[:k]).values
    Z0 = torch.zeros(n, k, dtype=torch.float64, device=DEV)
    Z0[centre, torch.arange(k, device=DEV)] = alpha
    Pi = Z0.clone()
    for _ in range(case["T_i"]):
        Pi = (1.0 - alpha) * _apply(back, Pi) + Z0
    best = Pi.max(dim=1, keepdim=True).values
    y = torch.where(Pi == best, torch.arange(k, device=DEV)[None, :], k).min(dim=1).values
    count = torch.bincount(y, minlength=k).double()
    Q = torch.zeros(n, k + 1, dtype=torch.float64, device=DEV)
    Q[:, 0] = 1.0 / math.sqrt(n)
    Q[torch.arange(n, device=DEV), 1 + y] = (1.0 / count.clamp(min=1).sqrt())[y]
    full = set(torch.nonzero(count > 0)[:, 0].tolist())
    for c in [c for c in range(k) if c not in full] + [max(full)]:
        Q[:, 1 + c] = _splitmix_sign(n, c) / math.sqrt(n)
    for _ in range(case["T"]):
        Z = (1.0 - beta) * _apply(fwd, Q) + beta * _inv(D) * (A @ Q)
        Q, R = torch.linalg.qr(Z)
        Q = Q * torch.where(torch.diagonal(R) < 0, -1.0, 1.0)
    return Q


def _exact_warm(case, st):
    t, n, k, lam = st["topo"], case["n"], case["k"], float(np.float32(1e-3))
    U = _unit(st["X"])
    A = torch.cat([U, _apply(_walks(t)[0], U)], dim=1)
    W1, b1, W2, b2 = (st["weights"][q].double() for q in ("W1", "b1", "W2", "b2"))
    Z1 = A @ W1 + b1
    cdf = 0.5 * (1.0 + torch.erf(Z1 / math.sqrt(2.0)))
    H = Z1 * cdf
    W = H @ W2 + b2
    if case["call"] == "warm_predict":
        return dict(W=W)
    Qt = st["Qt"].double()
    G, M = W.T @ W, Qt.T @ W
    Gi = torch.linalg.inv(G)
    eye = torch.eye(k, dtype=torch.float64, device=DEV)
    loss = k - torch.trace(Gi @ M.T @ M) + lam * ((G / n - eye) ** 2).sum()
    dW = -2.0 * (Qt @ (M @ Gi) - W @ (Gi @ M.T @ M @ Gi)) + (4.0 * lam / n) * W @ (G / n - eye)
    dZ = (dW @ W2.T) * (cdf + Z1 * torch.exp(-0.5 * Z1 * Z1) / math.sqrt(2.0 * math.pi))
    return dict(W1=A.T @ dZ, b1=dZ.sum(0), W2=H.T @ dW, b2=dW.sum(0), loss=float(loss))


def exact(case, seed):
    if case["call"] in ("discretize", "knn_ivf"):
        return None  # whole numbers; lists that depend on the cells
    if case["call"].startswith("warm"):
        return _exact_warm(case, prepare(case, seed))
    if float(case["n"]) ** 2 * case["d"] > 5.5e12:
        return None  # the pairs alone take over 20 seconds in 64 bits
    st = prepare(case, seed)
    if case["call"] == "knn":
        return dict(idx=None, sim=_exact_knn(st["X"], case["K"])[1])
    return dict(labels=None, Q=_exact_block(case, st))
