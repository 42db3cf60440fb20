"""The work that users of the DPMM sweep library have it do, as cases that can be timed.

Every case is a pass through the public entry points of the package: a chain that is
advanced some sweeps and read, a fitted model that labels a new batch, a batch of chains,
a chain fed by a stream, or the statistics of given labels.  Data are seeded mixtures of
the kinds that the repository's benchmark and tests use, made on the GPU.
"""
import math

import numpy as np
import torch

import paper_2204_08988_gb300 as P

PREC = {"fp64": P.PREC_FP64_PLAIN, "tf32": P.PREC_TF32, "bf16": P.PREC_BF16, "fp32": P.PREC_FP32,
        "x3": P.PREC_BF16X3}
ESZ = {"fp64": 8, "tf32": 4, "bf16": 2, "fp32": 4, "x3": 4}
SEED = 7  # Philox key of every chain


def listed():
    return [
        # the paper's smallest synthetic setting: launches and latency count, not the points
        dict(name="chain_d2", kind="gauss", prec="fp64", d=2, N=10_000, K=10, K_max=64, iters=10),
        # low-dimensional data in FP32 on the CUDA cores, a ragged N
        dict(name="chain_d8_fp32", kind="gauss", prec="fp32", d=8, N=100_003, K=12, K_max=64, iters=10),
        # the parity path: everything in FP64
        dict(name="chain_d32_fp64", kind="gauss", prec="fp64", d=32, N=30_001, K=20, K_max=64, iters=3),
        # the headline workload: a settled chain of a million points on the tensor cores
        dict(name="chain_d32", kind="gauss", prec="tf32", d=32, N=1_000_000, K=20, K_max=64, iters=10),
        # features of an image or text encoder after PCA: the largest data and many clusters
        dict(name="chain_d128", kind="gauss", prec="x3", d=128, N=4_000_000, K=64, K_max=128, iters=1),
        # count vectors of 100 draws over 200 categories, 50 topics
        dict(name="chain_topics", kind="counts", prec="bf16", d=200, N=1_000_000, K=50, K_max=128, words=100, iters=5),
        # a small, odd-sized set of count vectors
        dict(name="chain_topics_small", kind="counts", prec="bf16", d=77, N=20_011, K=9, K_max=64, words=60, iters=10),
        # documents over a vocabulary of 20,000 words, compressed rows (the 20newsgroups shape)
        dict(name="chain_documents", kind="documents", prec="fp32", d=20_000, N=11_314, K=20, K_max=64, iters=5),
        # many independent data sets at once, one stream each, mixed dimensions
        dict(name="batch", kind="batch", problems=64, N_min=1_000, N_max=200_000, sizes=5, iters=1),
        # streaming: each sweep takes a new set of values from page-locked host memory
        dict(name="stream_d32", kind="stream", prec="tf32", d=32, N=250_000, K=20, K_max=64),
        # a fitted model labels a new batch of points that is on the GPU; many clusters
        dict(name="assign_d32", kind="assign", prec="tf32", d=32, N=200_003, K=60, K_max=64),
        # statistics of given labels for a host program that allocates nothing
        dict(name="statistics", kind="statistics", d=32, N=1_000_000, K=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gauss_fp64", "gauss_fp32", "gauss_tf32", "gauss_tf32", "gauss_x3", "counts", "documents", "batch",
                       "stream", "assign", "statistics"])
    if kind == "gauss_fp64":
        d = rng.randint(2, 32)
        return dict(kind="gauss", prec="fp64", d=d, N=_log(rng, 1_000, 40_000), K=rng.randint(2, 20), K_max=64,
                    iters=rng.randint(1, 6))
    if kind == "gauss_fp32":
        return dict(kind="gauss", prec="fp32", d=rng.randint(2, 16), N=_log(rng, 1_000, 300_000), K=rng.randint(2, 24),
                    K_max=64, iters=rng.randint(1, 10))
    if kind == "gauss_tf32":
        return dict(kind="gauss", prec="tf32", d=rng.choice([32, rng.randint(9, 32)]), N=_log(rng, 2_000, 1_500_000),
                    K=rng.randint(2, 40), K_max=64, iters=rng.randint(1, 10))
    if kind == "gauss_x3":
        return dict(kind="gauss", prec="x3", d=rng.choice([64, 128, rng.randint(33, 128)]), N=_log(rng, 5_000, 2_000_000),
                    K=rng.randint(4, 64), K_max=128, iters=1)
    if kind == "counts":
        return dict(kind="counts", prec="bf16", d=rng.randint(16, 256), N=_log(rng, 5_000, 1_000_000), K=rng.randint(3, 60),
                    K_max=128, words=rng.randint(30, 150), iters=rng.randint(1, 8))
    if kind == "documents":
        return dict(kind="documents", prec="fp32", d=_log(rng, 1_000, 30_000), N=_log(rng, 2_000, 40_000), K=rng.randint(4, 40),
                    K_max=64, iters=rng.randint(1, 5))
    if kind == "batch":
        return dict(kind="batch", problems=rng.randint(8, 64), N_min=1_000, N_max=_log(rng, 10_000, 200_000),
                    sizes=rng.randint(1, 10_000), iters=rng.randint(1, 2))
    if kind == "stream":
        return dict(kind="stream", prec="tf32", d=rng.randint(8, 32), N=_log(rng, 10_000, 500_000), K=rng.randint(2, 26),
                    K_max=64)
    if kind == "assign":
        return dict(kind="assign", prec="tf32", d=rng.randint(8, 32), N=_log(rng, 5_000, 400_000), K=rng.randint(4, 64),
                    K_max=64)
    return dict(kind="statistics", d=rng.randint(1, 32), N=_log(rng, 10_000, 1_000_000), K=rng.randint(1, 16))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _model(g, d, K, spread, even=False):
    """A mixture: weights, means N(0, spread^2 I), covariance factors of Wishart(I, d + 2)
    draws (the identity at d = 2, as in the paper's two-dimensional setting)."""
    e = torch.empty(K, device="cuda", dtype=torch.float64).exponential_(generator=g)
    w = torch.full_like(e, 1.0) + e if even else e
    w = w / w.sum()
    mu = torch.randn(K, d, generator=g, device="cuda", dtype=torch.float64) * spread
    G = torch.randn(K, d, d + 2, generator=g, device="cuda", dtype=torch.float64)
    S = G @ G.transpose(1, 2)
    L = torch.eye(d, device="cuda", dtype=torch.float64).repeat(K, 1, 1) if d == 2 else torch.linalg.cholesky(S)
    return w, mu, L


def _points(g, model, N, dtype=torch.float32):
    w, mu, L = model
    K, d = mu.shape
    u = torch.rand(N, generator=g, device="cuda", dtype=torch.float64)
    y = torch.bucketize(u, w.cumsum(0)[:-1].contiguous()).to(torch.int32)
    order = torch.argsort(y.long(), stable=True)
    n = torch.bincount(y.long(), minlength=K).tolist()
    X = torch.empty(N, d, device="cuda", dtype=dtype)
    at = 0
    for k in range(K):
        e = torch.randn(n[k], d, generator=g, device="cuda", dtype=dtype)
        X[order[at: at + n[k]]] = e @ L[k].T.to(dtype) + mu[k].to(dtype)
        at += n[k]
    return X, y


def _topics(g, d, K, conc):
    a = torch.full((K, d), conc, dtype=torch.float64, device="cuda")
    t = torch._sample_dirichlet(a, generator=g).clamp_min(1e-12)
    return t / t.sum(1, keepdim=True)


def _words(g, theta, y, lengths):
    """(document, word) of every word, the documents taken topic by topic."""
    doc, word = [], []
    for k in range(theta.shape[0]):
        at = torch.nonzero(y == k).flatten()
        own = torch.repeat_interleave(at, lengths[at])
        if own.numel():
            u = torch.rand(own.numel(), generator=g, device="cuda", dtype=torch.float64)
            doc.append(own)
            word.append(torch.searchsorted(theta[k].cumsum(0)[:-1].contiguous(), u, right=True))
    return torch.cat(doc), torch.cat(word)


def _counts(g, N, d, K, words):
    theta = _topics(g, d, K, 0.1)
    y = torch.randint(0, K, (N,), generator=g, device="cuda")
    X = torch.zeros(N * d, device="cuda", dtype=torch.int32)
    doc, word = _words(g, theta, y, torch.full((N,), words, device="cuda", dtype=torch.int64))
    X.scatter_add_(0, doc * d + word, torch.ones_like(doc, dtype=torch.int32))
    return X.view(N, d), y.to(torch.int32)


def _documents(g, N, d, K):
    theta = _topics(g, d, K, 0.05)
    y = torch.randint(0, K, (N,), generator=g, device="cuda")
    lengths = (30.0 * torch.exp(torch.rand(N, generator=g, device="cuda", dtype=torch.float64) * math.log(20.0))).long()
    doc, word = _words(g, theta, y, lengths)
    key, n = torch.unique(doc * d + word, return_counts=True)
    ptr = torch.zeros(N + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.bincount(key // d, minlength=N).cumsum(0)
    return ptr.cpu().numpy(), (key % d).int().cpu().numpy(), n.int().cpu().numpy(), y.to(torch.int32)


# ---------------------------------------------------------------- chains
def _chain(case, stream):
    d, K_max, prec = case["d"], case["K_max"], PREC[case["prec"]]
    if case["kind"] in ("counts", "documents"):
        return P.DPMM(P.PRIOR_DIRICHLET, d, K_max, 10.0, prec=prec, stream=stream.cuda_stream, beta=np.ones(d))
    return P.DPMM(P.PRIOR_NIW, d, K_max, 10.0, prec=prec, stream=stream.cuda_stream, kappa0=1.0, m0=np.zeros(d),
                  nu0=d + 3.0, psi0=np.eye(d))


def _settle(g, chain, y):
    """Start from the generating clusters and fair sub-label coins."""
    y = torch.unique(y, return_inverse=True)[1].to(torch.int32)  # clusters that drew no point are left out
    zb = torch.randint(0, 2, y.shape, generator=g, device="cuda", dtype=torch.uint8)
    chain.set_state(int(y.max()) + 1, y.cpu().numpy(), zb.cpu().numpy())


def _label_buffers(N):
    return torch.empty(N, dtype=torch.int32, pin_memory=True), torch.empty(N, dtype=torch.uint8, pin_memory=True)


def _batch_sizes(case):
    r = np.random.default_rng(case["sizes"])
    n = case["problems"]
    N = np.exp(r.uniform(math.log(case["N_min"]), math.log(case["N_max"]), n)).astype(int)
    return [(int(a), int(b), int(k)) for a, b, k in zip(N, r.choice([2, 8, 32, 64], n), r.integers(2, 31, n))]


def _assign_params(g, model):
    """Parameters of a fitted model, 3 slots a cluster: the cluster, and two sub-clusters half
    a standard deviation to either side of its mean."""
    w, mu, L = model
    K, d = mu.shape
    e = torch.randn(K, d, generator=g, device="cuda", dtype=torch.float64)
    off = 0.5 * (L @ (e / e.norm(dim=1, keepdim=True)).unsqueeze(2)).squeeze(2)
    W = torch.linalg.inv(L).transpose(1, 2)  # upper triangular, precision = W W^T
    m = torch.stack([mu, mu - off, mu + off], 1).reshape(3 * K, d)
    logw = torch.stack([w.log(), torch.full_like(w, math.log(0.45)), torch.full_like(w, math.log(0.55))], 1).reshape(-1)
    W3 = W.unsqueeze(1).expand(K, 3, d, d).reshape(3 * K, d, d)
    return dict(logw=logw, mu=m, W=W3, logdetW=torch.diagonal(W3, dim1=1, dim2=2).log().sum(1))


def _assign_inputs(case, seed):
    g = _gen(seed)
    model = _model(g, case["d"], case["K"], 5.0, even=True)
    params = _assign_params(g, model)
    X0, y0 = _points(g, model, case["N"])  # the points that the model was fitted to
    X, _ = _points(g, model, case["N"])    # the new ones
    return g, params, X0, y0, X


def _statistics_inputs(case, seed):
    g = _gen(seed)
    X, y = _points(g, _model(g, case["d"], case["K"], 5.0), case["N"])
    return X, y, torch.randint(0, 2, y.shape, generator=g, device="cuda", dtype=torch.uint8)


def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.Stream()
    if kind == "statistics":
        X, z, zb = _statistics_inputs(case, seed)
        K, d = case["K"], case["d"]
        out = [torch.empty(n, dtype=torch.float64, device="cuda") for n in (2 * K, 2 * K * d, 2 * K * d * d)]
        return dict(case=case, X=X, z=z, zb=zb, out=out)
    if kind == "batch":
        g = _gen(seed)
        chains, streams, sizes = [], [], _batch_sizes(case)
        for p, (N, d, K) in enumerate(sizes):
            s = torch.cuda.Stream()
            X, y = _points(g, _model(g, d, K, 5.0), N)
            torch.cuda.synchronize()
            c = _chain(dict(kind="gauss", d=d, K_max=64, prec="fp32" if d <= 8 else "tf32" if d <= 32 else "x3"), s)
            c.set_data(X)
            c.set_problem(p)
            _settle(g, c, y)
            chains.append(c)
            streams.append(s)
        z, zb = _label_buffers(sum(N for N, _, _ in sizes))
        return dict(case=case, chains=chains, streams=streams, sizes=sizes, z=z, zb=zb)
    if kind == "assign":
        g, params, X0, y0, X = _assign_inputs(case, seed)
        torch.cuda.synchronize()
        c = _chain(case, stream)
        c.set_data(X0)
        _settle(g, c, y0)
        c.set_params(case["K"], {k: v.cpu().numpy() for k, v in params.items()})
        c.set_mask(2)  # labels and statistics under the model's parameters
        z, zb = _label_buffers(case["N"])
        return dict(case=case, chain=c, stream=stream, X=X, z=z, zb=zb)
    g = _gen(seed)
    N, d = case["N"], case["d"]
    c = _chain(case, stream)
    z, zb = _label_buffers(N)
    state = dict(case=case, chain=c, stream=stream, z=z, zb=zb)
    if kind == "documents":
        ptr, idx, n, y = _documents(g, N, d, case["K"])
        c.set_data_csr(ptr, idx, n)
    elif kind == "counts":
        X, y = _counts(g, N, d, case["K"], case["words"])
        torch.cuda.synchronize()
        c.set_data(X)
    else:
        model = _model(g, d, case["K"], 6.0 if d == 2 else 5.0 if d <= 32 else 4.0)
        X, y = _points(g, model, N, torch.float64 if case["prec"] == "fp64" else torch.float32)
        torch.cuda.synchronize()
        c.set_data(X)
    _settle(g, c, y)
    if kind == "stream":
        # two more sets of values at the same points' clusters, in page-locked host memory
        host = []
        for _ in range(2):
            h = torch.empty(N, d, pin_memory=True)
            h.copy_(X + 0.1 * torch.randn(N, d, generator=g, device="cuda"))
            host.append(h)
        c.stage_data(host[0])
        state.update(host=host, turn=0)
    return state


# ---------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "statistics":
        P.dpmm_suffstats_noalloc(state["X"], state["z"], state["zb"], case["K"], *state["out"])
        return dict(zip(("n", "sx", "sxx"), state["out"]))
    if kind == "batch":
        P.dpmm_sweep_batch([c.h for c in state["chains"]], case["iters"], SEED)
        at = 0
        for c, (N, _, _) in zip(state["chains"], state["sizes"]):
            P.dpmm_get_labels(c.h, N, state["z"][at: at + N], state["zb"][at: at + N])
            at += N
        return dict(z=state["z"], zbar=state["zb"], K=np.array([c.K for c in state["chains"]], np.int32))
    c = state["chain"]
    if kind == "assign":
        c.update_data(state["X"])
        c.sweep(1, SEED)
    elif kind == "stream":
        c.sweep(1, SEED)
        state["turn"] ^= 1
        c.stage_data(state["host"][state["turn"]])  # copied while this sweep runs
    else:
        c.sweep(case["iters"], SEED)
    P.dpmm_get_labels(c.h, case["N"], state["z"], state["zb"])
    out = dict(z=state["z"], zbar=state["zb"], K=c.K)
    if kind != "stream" and case["d"] <= 256 and not (case["prec"] == "x3"):
        n, sx, sxx = c.stats()
        out["n"], out["sx"] = _table(n, case["K_max"]), _table(sx, case["K_max"])
        if sxx is not None:
            out["sxx"] = _table(sxx, case["K_max"])
    return out


def _table(rows, K_max):
    """The rows of the slots in use as a table of all K_max clusters' slots, zero beyond K, so
    that its shape does not hang on how many clusters a chain has come to."""
    full = np.zeros((3 * K_max,) + rows.shape[1:])
    full[: rows.shape[0]] = rows
    return full


# ---------------------------------------------------------------- what a pass cannot do without
def _sweep_work(kind, prec, d, N, K, words=0):
    """Every point read once and its two labels written; the cluster and two sub-cluster
    scores of each point and its share of the second moments."""
    if kind == "counts":
        return N * d * ESZ[prec] + 5 * N, 2.0 * N * d * (K + 2)
    if kind == "documents":
        nnz = 160.0 * N
        return 8 * nnz + 13 * N, 2.0 * nnz * (K + 2)
    return N * d * ESZ[prec] + 5 * N, float(N) * d * d * (2 * K + 5)


def work(case):
    kind = case["kind"]
    if kind == "statistics":
        N, d, K = case["N"], case["d"], case["K"]
        return dict(bytes=N * (4 * d + 5) + 16 * K * (1 + d + d * d), flops=1.0 * N * d * (d + 1))
    if kind == "batch":
        got = [_sweep_work("gauss", "fp32", d, N, K) for N, d, K in _batch_sizes(case)]
        return dict(bytes=case["iters"] * sum(b for b, _ in got), flops=case["iters"] * sum(f for _, f in got))
    b, f = _sweep_work(kind, case["prec"], case["d"], case["N"], case["K"])
    n = case.get("iters", 1)
    if kind in ("stream", "assign"):  # the new values are read from where the caller has them
        b += 4 * case["N"] * case["d"]
    return dict(bytes=n * b, flops=n * f)


# ---------------------------------------------------------------- the same in 64 bits
def _philox(c0, c1, c2, k0):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors of 32-bit words."""
    m = 0xFFFFFFFF

    def mul(a, b):  # high and low words of a 32 x 32 bit product, without leaving int64
        t = (b & 0xFFFF) * a
        s = (b >> 16) * a + (t >> 16)
        return (s >> 16) & m, ((s << 16) | (t & 0xFFFF)) & m

    c = [c0, torch.full_like(c0, c1), c2, torch.zeros_like(c0)]
    k1 = 0
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c


def _gumbel(word):
    u = (2 * (word >> 9) + 1).double() * 2.0 ** -24
    return -torch.log(-torch.log(u))


def exact(case, seed):
    if case["kind"] == "statistics":
        X, z, zb = _statistics_inputs(case, seed)
        K, d = case["K"], case["d"]
        slot = 2 * z.long() + zb.long()
        sx, sxx = [], []
        for s in range(2 * K):
            Y = X[slot == s].double()
            sx.append(Y.sum(0))
            sxx.append(Y.T @ Y)
        return dict(n=torch.bincount(slot, minlength=2 * K).double(), sx=torch.stack(sx).reshape(-1),
                    sxx=torch.stack(sxx).reshape(-1))
    if case["kind"] != "assign":
        return None  # a chain's numbers hang on the labels that it has drawn
    _, p, _, _, X = _assign_inputs(case, seed)
    X = X.double()
    N, d, K = case["N"], case["d"], case["K"]
    c = p["logw"] + p["logdetW"]
    i = torch.arange(N, device="cuda")
    best = torch.full((N,), -math.inf, dtype=torch.float64, device="cuda")
    z = torch.zeros(N, dtype=torch.int64, device="cuda")
    for k in range(K):  # Gumbel-max over the clusters (tag 5: two clusters to a Philox block)
        s = c[3 * k] - 0.5 * ((X - p["mu"][3 * k]) @ p["W"][3 * k]).square().sum(1)
        s = s + _gumbel(_philox(i, 0, torch.full_like(i, 5 << 24 | k // 2), SEED)[2 * (k % 2)])
        z = torch.where(s > best, k, z)
        best = torch.maximum(s, best)
    w = _philox(i, 0, torch.full_like(i, 6 << 24), SEED)
    zb = torch.empty_like(z)
    n, sx, sxx = [], [], []
    for k in range(K):
        at = torch.nonzero(z == k).flatten()
        Y = X[at]
        s = [c[3 * k + 1 + h] - 0.5 * ((Y - p["mu"][3 * k + 1 + h]) @ p["W"][3 * k + 1 + h]).square().sum(1)
             + _gumbel(w[2 * h][at]) for h in (0, 1)]
        zb[at] = (s[1] > s[0]).long()
        for part in (Y, Y[zb[at] == 0], Y[zb[at] == 1]):
            n.append(float(part.shape[0]))
            sx.append(part.sum(0))
            sxx.append(part.T @ part)
    pad = 3 * (case["K_max"] - K)
    full = [np.concatenate([a, np.zeros((pad,) + a.shape[1:])]) for a in
            (np.array(n), torch.stack(sx).cpu().numpy(), torch.stack(sxx).cpu().numpy())]
    return dict(z=None, zbar=None, K=None, n=full[0], sx=full[1], sxx=full[2])
