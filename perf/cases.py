"""Performance cases of the framework: what a program that uses it has it do.

Every case goes through the binding (paper_1209_0410_gb300.hc) as a user's
program calls it.  Rows are drawn on the device from the mixture the rest of
the repository uses (64 isotropic Gaussian clusters, centres uniform in [0,
255], sigma 20, rounded and clipped; float32 rows are those values / 255) and
queries are rows plus N(0, 8) noise.

kinds
  query    one batch of queries on a built index: hc_query, or with ordered
           hc_query_ordered with a workspace kept between calls
  build    hc_build over rows on the device; the outputs are the index's lists
  multi    many uneven indexes answered by one persistent launch (MultiPlan)
  learned  a depth per query from the predictor, then hc_query_depths
  labels   hc_probe_labels: the training labels of the predictor
  fit      one training run of the predictor (MLP.fit) from given weights
  brute    hc_bruteforce: the exact answer recall is measured against
  serve    requests submitted to a server and collected (host buffers)
"""
import math

import numpy as np
import torch

from paper_1209_0410_gb300 import hc

DEV = "cuda"
CLUSTERS = 64


# ------------------------------------------------------------------ the cases
def _query(name, n, nq, p, k=10, d=128, dtype="u8", curves=8, m=16, parts=1, ordered=True):
    return dict(name=name, kind="query", n=n, d=d, dtype=dtype, curves=curves, m=m, parts=parts,
                nq=nq, k=k, p=p, ordered=ordered)


def listed():
    return [
        # one user looks something up: the latency of a single search
        _query("query_one", 100_000, 1, 128, ordered=False),
        # the small configuration: 1,000 queries on 100,000 rows
        _query("query_small", 100_000, 1_000, 64, ordered=False),
        # the headline batch: 100,000 queries on 10M rows, answered in key order
        _query("query_scale", 10_000_000, 100_000, 128),
        # float32 descriptors, sizes that are no multiple of anything
        _query("query_scale_f32", 4_000_037, 33_333, 128, dtype="f32"),
        # partitioned Hypercurves: 8 partitions at their Pessimist depth
        _query("query_partitions", 10_000_000, 100_000, 32, parts=8),
        # the index of the headline configuration, built from resident rows
        dict(name="build_scale", kind="build", n=10_000_000, d=128, dtype="u8", curves=8, m=16,
             parts=1),
        # 64 independent indexes of uneven sizes, types and batches in one launch
        dict(name="multi_uneven", kind="multi", indexes=64, n_min=10_000, n_max=2_000_000,
             nq_max=4096, p=64, shapes=11),
        # a batch whose depths the predictor chooses
        dict(name="learned_query", kind="learned", n=10_000_000, nq=100_000, k=10, p_hi=512),
        # labels for training the predictor: the depth that reproduces p = 512
        dict(name="labels", kind="labels", n=10_000_000, nq=50_000, k=10, p_max=512),
        # one epoch of training at the minibatch the learned workload uses
        dict(name="fit", kind="fit", n=262_144, batch=4096, epochs=1),
        # exact ground truth for a recall sample
        dict(name="brute_scale", kind="brute", n=10_000_000, d=128, dtype="u8", nq=2_000, k=10),
        # sixteen clients' requests outstanding at a server
        dict(name="serve", kind="serve", n=10_000_000, requests=16, nq=1024, k=10, p=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "query", "query", "build", "build", "multi", "learned",
                       "labels", "fit", "brute", "brute", "serve"])
    n = _log_int(rng, 20_000, 8_000_000)
    if kind in ("query", "build"):
        dtype = rng.choice(["u8", "u8", "f32"])
        d = rng.choice([64, 96, 128, 128, 128, 256])
        m = rng.choice([16, 16, 16, 8])
        curves = min(16, d // m)
        parts = rng.choice([1, 1, 1, 2, 4, 8])
        n = _log_int(rng, 20_000, 4_000_000 if dtype == "f32" or d > 128 or m < 16 else 8_000_000)
        if kind == "build":
            return dict(kind=kind, n=n, d=d, dtype=dtype, curves=curves, m=m, parts=parts)
        p = max(4, _log_int(rng, 16, 512) // parts)
        row = d * (4 if dtype == "f32" else 1)
        most = int(12e9 / (curves * parts * 2 * p * row))
        nq = max(1, min(_log_int(rng, 1, 100_000), most))
        return dict(kind=kind, n=n, d=d, dtype=dtype, curves=curves, m=m, parts=parts, nq=nq,
                    k=rng.choice([1, 10, 10, 10, 37, 100]), p=p, ordered=rng.random() < 0.5)
    if kind == "multi":
        return dict(kind=kind, indexes=rng.randint(3, 24), n_min=10_000,
                    n_max=_log_int(rng, 50_000, 1_000_000), nq_max=_log_int(rng, 64, 4096),
                    p=_log_int(rng, 16, 128), shapes=rng.randrange(1 << 20))
    if kind == "learned":
        return dict(kind=kind, n=n, nq=_log_int(rng, 32, 100_000), k=10, p_hi=512)
    if kind == "labels":
        return dict(kind=kind, n=n, nq=_log_int(rng, 500, 50_000), k=rng.choice([1, 10, 10, 50]),
                    p_max=rng.choice([64, 100, 128, 512]))
    if kind == "fit":
        batch = rng.choice([256, 1000, 2048, 4096])
        return dict(kind=kind, n=batch * rng.randint(4, 48) + rng.randint(0, batch - 1),
                    batch=batch, epochs=1)
    if kind == "brute":
        dtype = rng.choice(["u8", "u8", "f32"])
        return dict(kind=kind, n=_log_int(rng, 10_000, 300_000 if dtype == "f32" else 3_000_000),
                    d=rng.choice([64, 128, 128, 256]), dtype=dtype, nq=_log_int(rng, 1, 2000),
                    k=rng.choice([1, 10, 10, 100]))
    return dict(kind=kind, n=n, requests=rng.randint(2, 16), nq=_log_int(rng, 1, 1024), k=10,
                p=rng.choice([32, 128, 200]))


# ------------------------------------------------------------------- inputs
def _rows(g, n, d):
    """(n, d) uint8 rows of the clustered mixture."""
    centres = torch.rand((CLUSTERS, d), generator=g, device=DEV) * 255.0
    out = torch.empty((n, d), dtype=torch.uint8, device=DEV)
    for a in range(0, n, 1 << 20):
        b = min(n, a + (1 << 20))
        which = torch.randint(0, CLUSTERS, (b - a,), generator=g, device=DEV)
        x = torch.randn((b - a, d), generator=g, device=DEV).mul_(20.0).add_(centres[which])
        out[a:b] = x.round_().clamp_(0, 255).to(torch.uint8)
    return out


def _queries(g, rows, nq):
    src = torch.randint(0, rows.shape[0], (nq,), generator=g, device=DEV)
    x = rows[src].float()
    x += torch.randn(x.shape, generator=g, device=DEV) * 8.0
    return x.round_().clamp_(0, 255).to(torch.uint8)


def _vectors(seed, n, d, nq, dtype):
    """Rows and queries of one index, by the seed alone."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    rows = _rows(g, n, d)
    q = _queries(g, rows, nq) if nq else None
    if dtype == "f32":
        rows = rows.float().div_(255.0)
        q = q.float().div_(255.0) if nq else None
    return rows, q


def _multi_shapes(case):
    """(n, d, dtype, nq, k) of every index: n and nq log-uniform."""
    rng = np.random.default_rng(case["shapes"])
    out = []
    for _ in range(case["indexes"]):
        u = rng.random(2)
        n = case["n_min"] * (case["n_max"] / case["n_min"]) ** u[0]
        out.append((int(n), int(rng.choice([64, 128, 256])), str(rng.choice(["u8", "f32"])),
                    max(1, int(case["nq_max"] ** u[1])), int(rng.choice([1, 10, 100]))))
    return out


FEATURES = 32          # 4 per curve, 8 curves
# typical feature values: key gaps of about 100 octaves, distances of about 14
FEATURE_MEAN = np.tile(np.float32([100, 100, 14, 14.5]), FEATURES // 4)
FEATURE_SD = np.tile(np.float32([8, 8, 1, 0.5]), FEATURES // 4)


def _weights(seed, bias):
    """He-style weights of the 32 -> 64 -> 64 -> 1 predictor, output near bias."""
    rng = np.random.default_rng(seed)
    parts = [rng.normal(0, math.sqrt(2 / 32), 32 * 64), np.zeros(64),
             rng.normal(0, math.sqrt(2 / 64), 64 * 64), np.zeros(64),
             rng.normal(0, 0.5 / math.sqrt(64), 64), np.full(1, bias)]
    return np.concatenate(parts).astype(np.float32)


def _samples(case, seed):
    """Features and depth labels of a training set, labels following the features."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    z = torch.randn((case["n"], FEATURES), generator=g, device=DEV)
    feats = z * torch.from_numpy(FEATURE_SD).to(DEV) + torch.from_numpy(FEATURE_MEAN).to(DEV)
    w = torch.randn((FEATURES,), generator=g, device=DEV) / math.sqrt(FEATURES)
    log_p = 7.0 + (z * w).sum(1) + 0.3 * torch.randn((case["n"],), generator=g, device=DEV)
    return feats.contiguous(), log_p.exp2().clamp(1, 512).to(torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("query", "build"):
        nq = case["nq"] if kind == "query" else 0
        s["rows"], s["q"] = _vectors(seed, case["n"], case["d"], nq, case["dtype"])
        if kind == "query":
            s["index"] = hc.hc_build(s["rows"], case["curves"], case["m"],
                                     partitions=case["parts"])
            if case["ordered"]:
                need = hc.hc_query_ordered_workspace(s["index"], nq)
                s["workspace"] = torch.empty(need, dtype=torch.uint8, device=DEV)
    elif kind == "multi":
        shapes = _multi_shapes(case)
        jobs = []
        total = {t: sum(nq * k for _, _, dt, nq, k in shapes if dt == t) for t in ("u8", "f32")}
        # every job answers into its stretch of one buffer per type
        s["out"] = {"u8": (torch.empty(total["u8"], dtype=torch.int32, device=DEV),
                           torch.empty(total["u8"], dtype=torch.int32, device=DEV)),
                    "f32": (torch.empty(total["f32"], dtype=torch.int32, device=DEV),
                            torch.empty(total["f32"], dtype=torch.float32, device=DEV))}
        at = {"u8": 0, "f32": 0}
        for i, (n, d, dt, nq, k) in enumerate(shapes):
            rows, q = _vectors(seed * 1009 + i, n, d, nq, dt)
            job = hc.MultiJob(hc.hc_build(rows, d // 16, 16), q, k, case["p"])
            ids, dist = s["out"][dt]
            a, b = at[dt], at[dt] + nq * k
            job.ids, job.dist, at[dt] = ids[a:b].view(nq, k), dist[a:b].view(nq, k), b
            jobs.append(job)
        s["plan"] = hc.MultiPlan(jobs, dict(warps_per_block=8, blocks_per_sm=3, tile=1,
                                            use_graph=True))
    elif kind in ("learned", "labels"):
        s["rows"], s["q"] = _vectors(seed, case["n"], 128, case["nq"], "u8")
        s["index"] = hc.hc_build(s["rows"], 8, 16)
        if kind == "learned":
            s["mlp"] = hc.MLP(FEATURES)
            s["mlp"].set_params(_weights(seed, 7.0), FEATURE_MEAN, 1.0 / FEATURE_SD)
    elif kind == "fit":
        s["feats"], s["labels"] = _samples(case, seed)
        s["theta"] = _weights(seed, 0.0)
        s["mlp"] = hc.MLP(FEATURES, max_batch=case["batch"])
        s["seed"] = seed
    elif kind == "brute":
        s["rows"], s["q"] = _vectors(seed, case["n"], case["d"], case["nq"], case["dtype"])
    else:
        s["rows"], q = _vectors(seed, case["n"], 128, case["nq"] * case["requests"], "u8")
        s["index"] = hc.hc_build(s["rows"], 8, 16)
        s["requests"] = np.split(q.cpu().numpy(), case["requests"])
        s["server"] = hc.Server([s["index"]], 64 << 20)
    return s


# --------------------------------------------------------------------- a pass
class _Lists:
    """A device array of an index, as hc_index_describe gives its address."""

    def __init__(self, ptr, count, typestr):
        self.__cuda_array_interface__ = dict(shape=(count,), typestr=typestr, version=3,
                                             data=(ptr, False), strides=None)


def _index_lists(index):
    info, off = hc.hc_index_describe(index)
    out = [torch.as_tensor(_Lists(info["keys_hi_dev"], int(off[-1]), "<i8"), device=DEV),
           torch.as_tensor(_Lists(info["ids_dev"], int(off[-1]), "<i4"), device=DEV)]
    if info["keys_lo_dev"]:
        out.append(torch.as_tensor(_Lists(info["keys_lo_dev"], int(off[-1]), "<i8"), device=DEV))
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "query":
        if case["ordered"]:
            return hc.hc_query_ordered(state["index"], state["q"], case["k"], case["p"],
                                       workspace=state["workspace"])
        return hc.hc_query(state["index"], state["q"], case["k"], case["p"])
    if kind == "build":
        if state.get("index") is not None:      # the index this one replaces
            state["index"].free(torch.cuda.current_stream())
        state["index"] = hc.hc_build(state["rows"], case["curves"], case["m"],
                                     partitions=case["parts"])
        return _index_lists(state["index"])
    if kind == "multi":
        state["plan"].run()
        return state["out"]
    if kind == "learned":
        p = state["mlp"].predict_depths(state["index"], state["q"], 0.0, 1, case["p_hi"])
        return (p,) + tuple(hc.hc_query_depths(state["index"], state["q"], case["k"], p))
    if kind == "labels":
        return hc.hc_probe_labels(state["index"], state["q"], case["k"], case["p_max"])
    if kind == "fit":
        mlp = state["mlp"]
        mlp.set_params(state["theta"], np.zeros(FEATURES, np.float32),
                       np.ones(FEATURES, np.float32))
        losses = mlp.fit(state["feats"], state["labels"], case["epochs"], case["batch"], 1e-3,
                         seed=state["seed"])
        theta, mu, isd = mlp.get_params()
        return theta, mu, isd, np.float32(losses)
    if kind == "brute":
        return hc.hc_bruteforce(state["rows"], state["q"], case["k"])
    server = state["server"]
    tickets = [server.submit(0, q, case["k"], case["p"]) for q in state["requests"]]
    out = []
    for t in tickets:
        got = None
        while got is None:
            got = server.poll(t, timeout_us=1_000_000)
        out.append(got)
    return out


# ----------------------------------------------------------------- its work
def _index_bytes(n, d, dtype, curves, m):
    return n * d * (4 if dtype == "f32" else 1) + n * curves * (12 if m == 16 else 20)


def _query_work(n, d, dtype, curves, m, parts, nq, k, p):
    row = d * (4 if dtype == "f32" else 1)
    rows = nq * curves * parts * min(2 * p, n // parts)
    # the window rows and their ids, or every row and entry once if that is less
    read = min(rows * (row + 4), _index_bytes(n, d, dtype, curves, m))
    return read + nq * row + nq * k * 8, 3.0 * rows * d


def work(case):
    kind = case["kind"]
    if kind == "query":
        b, f = _query_work(*(case[x] for x in ("n", "d", "dtype", "curves", "m", "parts", "nq",
                                               "k", "p")))
    elif kind == "build":
        b, f = _index_bytes(*(case[x] for x in ("n", "d", "dtype", "curves", "m"))), 0.0
    elif kind == "multi":
        parts = [_query_work(n, d, dt, d // 16, 16, 1, nq, k, case["p"])
                 for n, d, dt, nq, k in _multi_shapes(case)]
        b, f = sum(x[0] for x in parts), sum(x[1] for x in parts)
    elif kind == "learned":
        # the weights centre the predictor on depth 128
        b, f = _query_work(case["n"], 128, "u8", 8, 16, 1, case["nq"], case["k"], 128)
        f += 2.0 * 6208 * case["nq"]
    elif kind == "labels":
        b, f = _query_work(case["n"], 128, "u8", 8, 16, 1, case["nq"], 0, case["p_max"])
        b += 4 * case["nq"]
    elif kind == "fit":
        used = case["n"] // case["batch"] * case["batch"] * case["epochs"]
        b, f = case["n"] * (FEATURES * 4 + 4), 6.0 * 6208 * used
    elif kind == "brute":
        row = case["d"] * (4 if case["dtype"] == "f32" else 1)
        b = (case["n"] + case["nq"]) * row + case["nq"] * case["k"] * 8
        f = 2.0 * case["n"] * case["nq"] * case["d"]
    else:
        b, f = _query_work(case["n"], 128, "u8", 8, 16, 1, case["nq"] * case["requests"],
                           case["k"], case["p"])
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------ 64-bit reference
def _signed_order(x):
    """A uint64 bit pattern in int64, so that signed order is unsigned order."""
    return x ^ -(1 << 63)


def _hilbert_words(x, m):
    """High and low words of the Hilbert key of each row of x ((n, m) int64 in
    [0, 255]): Skilling's transpose, bit planes read from the top, axis 0 first."""
    x = [x[:, i].clone() for i in range(m)]
    for q in range(7, 0, -1):
        low = (1 << q) - 1
        for i in range(m):
            bit = (x[i] >> q) & 1
            t = torch.where(bit == 1, 0, (x[0] ^ x[i]) & low)
            x[0] = torch.where(bit == 1, x[0] ^ low, x[0] ^ t)
            if i:
                x[i] = x[i] ^ t
    for i in range(1, m):
        x[i] = x[i] ^ x[i - 1]
    c = x[m - 1] >> 1
    for s in (1, 2, 4):
        c = c ^ (c >> s)
    hi, lo = torch.zeros_like(c), torch.zeros_like(c)
    for q in range(7, -1, -1):
        for i in range(m):
            hi = (hi << 1) | ((lo >> 63) & 1)
            lo = (lo << 1) | (((x[i] ^ c) >> q) & 1)
    return hi, lo


def _key_words(x, c, m):
    """The words of curve c's keys, most significant first (m = 8 or m = 16)."""
    y = x[:, c * m:(c + 1) * m]
    if y.dtype != torch.uint8:
        y = (y * 255.0).round().clamp(0, 255)
    hi, lo = _hilbert_words(y.to(torch.int64), m)
    if m <= 8:                       # the whole key is in the low word
        hi, lo = lo, hi
    return _signed_order(hi), _signed_order(lo)


def _exact_query(rows, q, curves, m, parts, k, p):
    """Distances of the k nearest of every query's windows, in 64 bits."""
    n, nq = rows.shape[0], q.shape[0]
    windows = []
    for c in range(curves):
        qh, ql = _key_words(q, c, m)
        for j in range(parts):
            a, b = j * n // parts, (j + 1) * n // parts
            h, lo = _key_words(rows[a:b], c, m)
            order = torch.sort(lo, stable=True).indices
            order = order[torch.sort(h[order], stable=True).indices]
            h, lo = h[order], lo[order]
            pos = torch.searchsorted(h, qh)
            # equal high words: on to the first entry whose low word is not below
            while True:
                at = pos.clamp(max=b - a - 1)
                step = (pos < b - a) & (h[at] == qh) & (lo[at] < ql)
                if not bool(step.any()):
                    break
                pos = pos + step.long()
            e = pos[:, None] + torch.arange(-p, p, device=DEV)
            ok = (e >= 0) & (e < b - a)
            windows.append(torch.where(ok, order[e.clamp(0, b - a - 1)] + a, -1).to(torch.int32))
            del h, lo, order, e, ok
    windows = torch.cat(windows, 1)
    out = torch.full((nq, k), math.inf, dtype=torch.float64, device=DEV)
    step = max(1, int(2e8 / (windows.shape[1] * q.shape[1])))
    for a in range(0, nq, step):
        w = windows[a:a + step].long().sort(1).values
        again = torch.zeros_like(w, dtype=torch.bool)
        again[:, 1:] = w[:, 1:] == w[:, :-1]
        x = rows[w.clamp(min=0)].double() - q[a:a + step, None, :].double()
        dist = x.square().sum(-1).masked_fill(again | (w < 0), math.inf)
        best = dist.topk(min(k, dist.shape[1]), dim=1, largest=False).values
        out[a:a + step, :best.shape[1]] = best
    return out


def _exact_brute(rows, q, k):
    out = []
    for a in range(0, q.shape[0], 64):
        best = None
        for b in range(0, rows.shape[0], 1 << 18):
            # |q|^2 + |x|^2 - 2 q.x in 64 bits
            x, y = rows[b:b + (1 << 18)].double(), q[a:a + 64].double()
            dist = (y.square().sum(1)[:, None] + x.square().sum(1)[None] - 2.0 * (y @ x.T))
            best = dist if best is None else torch.cat([best, dist], 1)
            best = best.topk(min(k, best.shape[1]), dim=1, largest=False).values
        out.append(best.clamp(min=0))
    return torch.cat(out)


def _splitmix64(z):
    z = z + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _exact_fit(case, seed):
    """One training run in float64: targets, normalisation, epoch orders, Adam."""
    feats, labels = (t.cpu().numpy() for t in _samples(case, seed))
    x, t = feats.astype(np.float64), np.log2(np.maximum(labels, 1).astype(np.float64))
    mu, isd = x.mean(0), 1.0 / np.maximum(x.std(0, ddof=1), 1e-3)
    xn = torch.from_numpy((x - mu) * isd).to(DEV)
    t = torch.from_numpy(t).to(DEV)
    theta = torch.from_numpy(_weights(seed, 0.0).astype(np.float64)).to(DEV).requires_grad_()
    cut = np.cumsum([32 * 64, 64, 64 * 64, 64, 64, 1])
    m, v = torch.zeros_like(theta), torch.zeros_like(theta)
    b, step, losses = case["batch"], 0, []
    for e in range(case["epochs"]):
        i = np.arange(case["n"], dtype=np.uint64)
        keys = _splitmix64(np.uint64(seed) ^ (np.uint64(e) << np.uint64(40)) ^ i)
        order = torch.from_numpy(np.argsort(keys >> np.uint64(32), kind="stable")).to(DEV)
        logged = []
        for j in range(case["n"] // b):
            at = order[j * b:(j + 1) * b]
            w1, b1, w2, b2, w3, b3 = (theta[a:z] for a, z in zip([0, *cut[:-1]], cut))
            h = torch.relu(xn[at] @ w1.view(32, 64) + b1)
            h = torch.relu(h @ w2.view(64, 64) + b2)
            loss = (h @ w3 + b3 - t[at]).square().mean()
            grad, = torch.autograd.grad(loss, theta)
            step += 1
            with torch.no_grad():
                m = 0.9 * m + 0.1 * grad
                v = 0.999 * v + 0.001 * grad * grad
                theta -= 1e-3 * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-8)
            if j % 50 == 0:
                logged.append(float(loss))
        losses.append(float(np.mean(logged)))
    return theta.detach(), mu, isd, np.float64(losses)


def exact(case, seed):
    kind = case["kind"]
    if kind == "fit":
        return _exact_fit(case, seed)
    if kind in ("query", "brute") and case["dtype"] == "f32":
        rows, q = _vectors(seed, case["n"], case["d"], case["nq"], "f32")
        if kind == "brute":
            return None, _exact_brute(rows, q, case["k"])
        return None, _exact_query(rows, q, *(case[x] for x in ("curves", "m", "parts", "k", "p")))
    if kind == "multi":
        dist = []
        for i, (n, d, dt, nq, k) in enumerate(_multi_shapes(case)):
            if dt == "f32":
                rows, q = _vectors(seed * 1009 + i, n, d, nq, dt)
                dist.append(_exact_query(rows, q, d // 16, 16, 1, k, case["p"]).reshape(-1))
        return {"f32": (None, torch.cat(dist))} if dist else None
    return None          # the other outputs are whole numbers
