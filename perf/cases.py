"""The measured workloads of the library: what a user's program runs through
the public entry points of paper_2201_02460_gb300.epi, over the sizes it is
used at.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs and handles a program holds before the call
    run(state)           one pass through the entry points, whole outputs
    work(case)           bytes and flops a pass cannot do without
    exact(case, seed)    the outputs in 64-bit arithmetic, where that is quick
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2201_02460_gb300 import epi

# work of the largest listed case, in combination-samples x 3^order: no drawn
# search or batch passes it
_MAX_WORK = math.comb(500, 4) * 8192 * 81
# passes of the orders without a tensor-core path, and of the thresholded
# output, are kept to about this share of it
_MAX_WORK_SLOW = _MAX_WORK / 40

_ctx = None


def _context():
    """The program's one library context (torch's current stream)."""
    global _ctx
    if _ctx is None:
        _ctx = epi.Context(0)
    return _ctx


def listed():
    return [
        # an interactive pair scan of a candidate-gene panel: the smallest
        # call, where launches and latency count (the repository's order-2
        # configuration)
        dict(name="pairs_panel", kind="search", order=2, n=200, m=1600, cases=800, top_n=10, plant=2),
        # a pair scan of a filtered chip, ragged and unbalanced
        dict(name="pairs_wide", kind="search", order=2, n=6007, m=5003, cases=1877, top_n=100, plant=2),
        # genotypes just read into host memory, to the best triples: dataset
        # creation and an ordinary search of odd size, as a program's first
        # call on each new study
        dict(name="triples_from_host", kind="fresh", order=3, n=401, m=2507, cases=907, top_n=20, plant=3),
        # the order-3 headline search (2000 SNPs x 4000 samples, top 100)
        dict(name="triples_wide", kind="search", order=3, n=2000, m=4000, cases=2000, top_n=100, plant=3),
        # the order-4 headline search (500 SNPs x 8192 samples): the largest
        dict(name="quads_large", kind="search", order=4, n=500, m=8192, cases=4096, top_n=100, plant=0),
        # order 5 on a short list of SNPs, ragged and unbalanced
        dict(name="quints_short", kind="search", order=5, n=93, m=2001, cases=811, top_n=100, plant=5),
        # the highest order (the published order-8 workload: 23 SNPs x 2048)
        dict(name="octets", kind="search", order=8, n=23, m=2048, cases=1024, top_n=100, plant=0),
        # many studies of uneven shape and mixed orders 2-4 in one call (the
        # batched configuration with its SNP counts divided by four)
        dict(name="batch_mixed", kind="batch", count=64, n_lo=25, n_hi=250, m_lo=1000, m_hi=16000, top_n=20, mix=4),
        # every significant triple instead of a top list: all with
        # G = 2 m MI at or above a fixed level
        dict(name="triples_significant", kind="threshold", order=3, n=1000, m=4000, cases=2000, g_min=76.0,
             capacity=4096, plant=3),
        # ranking candidate sets: network inference on one chunk of rows
        dict(name="network_rank", kind="mlp_forward", rows=1 << 22, n_in=30),
        # fitting the network: loss and gradients of one training batch
        dict(name="network_gradients", kind="mlp_gradients", rows=8192, n_in=30),
        # order-5 proposals on a new study: lower-order tables, candidate
        # ranking by a network with four-way features, exact re-score
        dict(name="proposals", kind="proposer", n=200, m=2000, cases=1000, triples=4096, budget=1_000_000,
             top_n=100, n_in=30),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# SNP ranges by order of drawn searches
_N_RANGE = {2: (60, 8000), 3: (40, 2000), 4: (24, 500), 5: (16, 120), 6: (12, 44), 7: (11, 32), 8: (11, 25)}


def _draw_shape(rng, order, cap, m_lo=400, m_hi=16000):
    """SNPs, samples and cases of an order-`order` study of at most `cap` work."""
    while True:
        n = _log_int(rng, *_N_RANGE[order])
        m = _log_int(rng, m_lo, m_hi)
        if math.comb(n, order) * m * 3 ** order <= cap:
            return n, m, max(1, min(m - 1, int(m * rng.uniform(0.2, 0.8))))


def draw(rng):
    kind = rng.choice(["search"] * 6 + ["fresh", "batch", "threshold", "mlp_forward", "mlp_gradients", "proposer"])
    if kind == "search":
        order = rng.choice([2, 3, 3, 4, 4, 5, 6, 7, 8])
        if order <= 4:
            n, m, c = _draw_shape(rng, order, _MAX_WORK)
        elif order == 5:
            n, m, c = _draw_shape(rng, order, _MAX_WORK / 4, 400, 4000)
        else:
            n, m, c = _draw_shape(rng, order, _MAX_WORK_SLOW, 400, 2600)
        return dict(kind=kind, order=order, n=n, m=m, cases=c, top_n=rng.choice([1, 10, 20, 100, 250]),
                    plant=order if order <= 5 else 0)
    if kind == "fresh":
        order = rng.choice([2, 3])
        n, m, c = _draw_shape(rng, order, _MAX_WORK / 50)
        return dict(kind=kind, order=order, n=n, m=m, cases=c, top_n=rng.choice([1, 10, 20, 100]), plant=order)
    if kind == "batch":
        n_hi = _log_int(rng, 40, 250)
        m_hi = _log_int(rng, 1500, 16000)
        return dict(kind=kind, count=rng.randint(2, 64), n_lo=max(8, n_hi // 10), n_hi=n_hi, m_lo=max(300, m_hi // 16),
                    m_hi=m_hi, top_n=rng.choice([1, 10, 20, 50]), mix=rng.randint(0, 9999))
    if kind == "threshold":
        order = rng.choice([2, 3, 3, 4])
        n, m, c = _draw_shape(rng, order, _MAX_WORK_SLOW)
        return dict(kind=kind, order=order, n=n, m=m, cases=c, g_min={2: 38.0, 3: 76.0, 4: 150.0}[order],
                    capacity=rng.choice([1000, 4096, 10000]), plant=order)
    if kind == "mlp_forward":
        return dict(kind=kind, rows=_log_int(rng, 1, 1 << 23), n_in=rng.choice([25, 30]))
    if kind == "mlp_gradients":
        return dict(kind=kind, rows=_log_int(rng, 100, 1 << 16), n_in=rng.choice([25, 30]))
    n = _log_int(rng, 30, 200)
    m = _log_int(rng, 400, 4000)
    return dict(kind=kind, n=n, m=m, cases=max(1, min(m - 1, int(m * rng.uniform(0.3, 0.7)))),
                triples=_log_int(rng, 16, min(4096, math.comb(n, 3))), budget=_log_int(rng, 1000, 1_000_000),
                top_n=rng.choice([10, 100]), n_in=rng.choice([25, 30]))


# ------------------------------------------------------------------ inputs --

def _genotypes(n, m, cases, plant, seed):
    """Hardy-Weinberg genotypes uint8 [n, m] (minor-allele frequencies
    U[0.05, 0.5]) and phenotypes uint8 [m] with exactly `cases` ones, on the
    GPU; with plant = q, q SNPs of frequency 0.5 whose genotype parity shifts
    an individual's chance to be a case (no lower-order effect)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 2_654_435_761 % (1 << 62) + 17)
    maf = 0.05 + 0.45 * torch.rand(n, 1, generator=g, device="cuda")
    where = torch.randperm(n, generator=g, device="cuda")[:plant]
    maf[where] = 0.5
    geno = torch.zeros(n, m, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        geno += torch.rand(n, m, generator=g, device="cuda") < maf
    liability = torch.rand(m, generator=g, device="cuda")
    if plant:
        liability += 0.5 * (geno[where].to(torch.int64).sum(0) & 1)
    pheno = torch.zeros(m, dtype=torch.uint8, device="cuda")
    pheno[torch.topk(liability, cases).indices] = 1
    return geno, pheno


def _rows(rows, n_in, seed):
    """Feature rows (log-scores, each in about [-10, -1]) and standardised targets."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 2_654_435_761 % (1 << 62) + 29)
    X = -5.0 + 1.5 * torch.randn(rows, n_in, generator=g, device="cuda")
    t = torch.randn(rows, generator=g, device="cuda")
    return X, t


def _network(n_in, seed):
    """A network as training leaves it: weights and the input standardisation."""
    net = epi.MLP(_context(), n_in, 256, seed=1 + seed)
    net.set_input_norm(np.full(n_in, -5.0, np.float32), np.full(n_in, 1.0 / 1.5, np.float32))
    return net


def _batch_shapes(case):
    """(SNPs, samples, cases, order) of a batch's studies."""
    rng = np.random.default_rng(case["mix"])
    shapes = []
    for _ in range(case["count"]):
        m = int(rng.integers(case["m_lo"], case["m_hi"] + 1))
        shapes.append((int(rng.integers(case["n_lo"], case["n_hi"] + 1)), m, int(round(m * rng.uniform(0.3, 0.7))),
                       int(rng.integers(2, 5))))
    return shapes


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case)
    if kind in ("search", "threshold"):
        geno, pheno = _genotypes(case["n"], case["m"], case["cases"], case["plant"], seed)
        state["ds"] = epi.Dataset(_context(), geno, pheno)
    elif kind == "fresh":
        geno, pheno = _genotypes(case["n"], case["m"], case["cases"], case["plant"], seed)
        state["geno"], state["pheno"] = geno.cpu().numpy(), pheno.cpu().numpy()
        _context()
    elif kind == "batch":
        state["sets"], state["orders"] = [], []
        for i, (n, m, c, order) in enumerate(_batch_shapes(case)):
            geno, pheno = _genotypes(n, m, c, 0, seed * 1000 + i)
            state["sets"].append(epi.Dataset(_context(), geno, pheno))
            state["orders"].append(order)
    elif kind in ("mlp_forward", "mlp_gradients"):
        state["net"] = _network(case["n_in"], seed)
        state["X"], state["t"] = _rows(case["rows"], case["n_in"], seed)
    elif kind == "proposer":
        state["geno"], state["pheno"] = _genotypes(case["n"], case["m"], case["cases"], 0, seed)
        state["net"] = _network(case["n_in"], seed)
    else:
        raise ValueError(kind)
    return state


def _outputs(r):
    return dict(combs=r.combs, rank=r.rank, mi=r.mi, mi_f32=r.mi_f32, counts=r.counts)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "search":
        return _outputs(epi.search(state["ds"], case["order"], case["top_n"]))
    if kind == "fresh":
        ds = epi.Dataset(_context(), state["geno"], state["pheno"])
        out = _outputs(epi.search(ds, case["order"], case["top_n"]))
        ds.close()
        return out
    if kind == "batch":
        res = epi.search_batched(_context(), state["sets"], state["orders"], [case["top_n"]] * len(state["sets"]))
        # every dataset's records and tables, one array per field
        outs = [_outputs(r) for r in res]
        return {f: np.concatenate([o[f].reshape(-1) for o in outs]) for f in outs[0]}
    if kind == "threshold":
        cap = case["capacity"]
        r, found = epi.search_threshold(state["ds"], case["order"], case["g_min"] / (2.0 * case["m"]), cap)
        # zero-filled to the capacity, so that every input gives the same shapes
        return dict(found=found, **{f: np.concatenate([a, np.zeros((cap - len(a),) + a.shape[1:], a.dtype)])
                                    for f, a in _outputs(r).items()})
    if kind == "mlp_forward":
        return state["net"].forward(state["X"])
    if kind == "mlp_gradients":
        g, loss = state["net"].gradients(state["X"], state["t"])
        return dict(grad=g, loss=loss)
    ds = epi.Dataset(_context(), state["geno"], state["pheno"])
    r, _ = epi.proposer_search(ds, state["net"], case["triples"], case["budget"], case["top_n"], with_counts=True)
    ds.close()
    return _outputs(r)


# -------------------------------------------------------------------- work --

def _search_work(n, m, order, top_n):
    """A table needs 2^order counted cells per class (the others follow by
    subtraction from the sub-tables), each over its class's individuals."""
    records = min(top_n, math.comb(n, order)) * (56 + 8 * 3 ** order)
    return dict(bytes=2 * n * m / 8 + m / 8 + records, flops=2.0 * 2 ** order * m * math.comb(n, order))


def work(case):
    kind = case["kind"]
    if kind in ("search", "fresh"):
        w = _search_work(case["n"], case["m"], case["order"], case["top_n"])
        if kind == "fresh":
            w["bytes"] += case["n"] * case["m"] + case["m"]
        return w
    if kind == "threshold":
        return _search_work(case["n"], case["m"], case["order"], 0)
    if kind == "batch":
        ws = [_search_work(n, m, k, case["top_n"]) for n, m, _, k in _batch_shapes(case)]
        return dict(bytes=sum(w["bytes"] for w in ws), flops=sum(w["flops"] for w in ws))
    h = 256
    if kind == "mlp_forward":
        params = case["n_in"] * h + h * h + 3 * h + 1
        return dict(bytes=4 * case["rows"] * (case["n_in"] + 1) + 2 * params,
                    flops=2.0 * case["rows"] * (case["n_in"] * h + h * h + h))
    if kind == "mlp_gradients":
        params = case["n_in"] * h + h * h + 3 * h + 1
        return dict(bytes=4 * case["rows"] * (case["n_in"] + 1) + 6 * params,
                    flops=2.0 * case["rows"] * (2 * case["n_in"] * h + 3 * h * h + 3 * h))
    n, m = case["n"], case["m"]
    orders = 4 if case["n_in"] == 30 else 3
    lower = sum(2.0 * 2 ** k * m * math.comb(n, k) for k in range(1, orders + 1))
    cands = case["triples"] * math.comb(n - 3, 2)
    flops = lower + 2.0 * cands * (case["n_in"] * h + h * h + h) + 2.0 * 32 * m * min(case["budget"], cands)
    return dict(bytes=n * m + m + case["top_n"] * (56 + 8 * 243), flops=flops)


# ------------------------------------------------------------------- exact --

def _xlogx(x):
    return torch.special.xlogy(x, x)


def _mi64(tables, m1, m0):
    """Mutual information (nats, float64) of counts [..., 2, cells]."""
    m = float(m1 + m0)
    t = tables.to(torch.float64)
    joint = _xlogx(t / m).sum((-1, -2))
    cell = _xlogx(t.sum(-2) / m).sum(-1)
    klass = sum(y / m * math.log(y / m) for y in (m1, m0) if y)
    return joint - cell - klass


def _exact_search(geno, pheno, order, top_n):
    """The best top_n combinations of order 2 or 3 by float64 MI, ties by rank."""
    n, m = geno.shape
    m1 = int(pheno.sum())
    classes = [(pheno == 1), (pheno == 0)]
    hot = [torch.stack([(geno[:, c] == g) for g in range(3)], 1).to(torch.float32) for c in classes]  # [n,3,mc]
    best_mi, best_rank, best_comb, best_tab = [], [], [], []
    prefixes = [()] if order == 2 else [(i,) for i in range(n - 2)]
    for pre in prefixes:
        lo = pre[0] + 1 if pre else 0
        rows = n - lo
        chunk = max(1, (1 << 22) // max(1, rows * 3 ** order)) if order == 2 else rows
        for a0 in range(0, rows, chunk):
            a1 = min(rows, a0 + chunk)
            tabs = []
            for h in hot:
                left = h[lo + a0:lo + a1]                                    # [A,3,mc]
                if pre:
                    left = (h[pre[0]][None, :, None, :] * left[:, None]).reshape(a1 - a0, 9, -1)
                right = h[lo:].reshape(rows * 3, -1)
                t = (left.reshape((a1 - a0) * left.shape[1], -1) @ right.T)   # exact: counts below 2^24
                tabs.append(t.reshape(a1 - a0, left.shape[1], rows, 3).permute(0, 2, 1, 3).reshape(
                    a1 - a0, rows, 3 ** order))
            tab = torch.stack(tabs, 2)                                        # [A,rows,2,cells]
            ia = torch.arange(lo + a0, lo + a1, device=geno.device)
            ja = torch.arange(lo, n, device=geno.device)
            ok = (ja[None, :] > ia[:, None]).nonzero()
            if ok.numel() == 0:
                continue
            tab = tab[ok[:, 0], ok[:, 1]]
            mi = _mi64(tab, m1, m - m1)
            comb = torch.stack([torch.full_like(ok[:, 0], p) for p in pre] + [ia[ok[:, 0]], ja[ok[:, 1]]], 1)
            rank = math.comb(n, order) - 1 - sum(
                _binom(n - 1 - comb[:, t], order - t) for t in range(order))
            keep = torch.topk(mi, min(mi.numel(), top_n + 64)).indices
            best_mi.append(mi[keep]); best_rank.append(rank[keep])
            best_comb.append(comb[keep]); best_tab.append(tab[keep])
    mi, rank = torch.cat(best_mi), torch.cat(best_rank)
    comb, tab = torch.cat(best_comb), torch.cat(best_tab)
    o = np.lexsort((rank.cpu().numpy(), -mi.cpu().numpy()))[:top_n]
    o = torch.as_tensor(o, device=mi.device)
    f = mi[o].cpu().numpy()
    return dict(combs=comb[o].cpu().numpy(), rank=rank[o].cpu().numpy().astype(np.uint64), mi=f, mi_f32=f,
                counts=tab[o].round().to(torch.int64).cpu().numpy().astype(np.uint32))


def _binom(a, b):
    out = torch.ones_like(a)
    for i in range(b):
        out = out * (a - i) // (i + 1)
    return out.clamp_min(0)


def _exact_network(case, seed):
    net = _network(case["n_in"], seed)
    theta = torch.as_tensor(net.params(), dtype=torch.float64, device="cuda")
    net.close()
    h, n_in = 256, case["n_in"]
    sizes = [(h, n_in), (h,), (h, h), (h,), (h,), (1,)]
    at, p = 0, []
    for s in sizes:
        p.append(theta[at:at + math.prod(s)].reshape(s).clone().requires_grad_(True))
        at += math.prod(s)
    X, t = _rows(case["rows"], n_in, seed)

    def forward(x):
        x = (x.to(torch.float64) + 5.0) * float(np.float32(1.0 / 1.5))
        a = torch.relu(x @ p[0].T + p[1])
        a = torch.relu(a @ p[2].T + p[3])
        return a @ p[4] + p[5]
    return forward, p, X, t


def exact(case, seed):
    kind = case["kind"]
    if kind in ("search", "fresh"):
        tables = math.comb(case["n"], case["order"])
        if case["order"] > 3 or tables * 3 ** case["order"] > 6e8 or case["order"] == 2 and case["n"] > 3000:
            return None
        geno, pheno = _genotypes(case["n"], case["m"], case["cases"], case["plant"], seed)
        with torch.no_grad():
            out = _exact_search(geno, pheno, case["order"], case["top_n"])
        # the whole-number outputs are compared as they are
        return dict(combs=None, rank=None, mi=out["mi"], mi_f32=out["mi_f32"], counts=None)
    if kind == "mlp_forward":
        forward, _, X, _ = _exact_network(case, seed)
        with torch.no_grad():
            return torch.cat([forward(x) for x in X.split(1 << 18)])
    if kind == "mlp_gradients":
        forward, p, X, t = _exact_network(case, seed)
        loss = ((forward(X) - t.to(torch.float64)) ** 2).mean()
        loss.backward()
        grad = torch.cat([q.grad.reshape(-1) for q in p])
        return dict(grad=grad.cpu().numpy(), loss=float(loss))
    return None
