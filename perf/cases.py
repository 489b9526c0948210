"""Performance cases: what programs have this library do, over its real range.

Every case is one pass of such a program through the public entry points of
``paper_1807_03847_gb300``: a certified ranking on a handle that is kept, a
ranking from a graph in host memory, an update batch, a served stream of
batches, another stopping criterion, or a check of given bounds.  Graphs are
made on the GPU from the seed alone: Erdos-Renyi, R-MAT (a, b, c, d = .57,
.19, .19, .05) and Chung-Lu (Pareto expected degrees, exponent 2.1, capped at
sqrt of their sum, vertex ids in random order), symmetrised and deduplicated.

``exact`` restates the paper's Algorithm 1 (and the continuation after a
batch, Algorithm 2's result) in plain 64-bit torch.
"""
import math

import numpy as np
import torch

import paper_1807_03847_gb300 as K

EPS = 1e-9  # separation slack of every workload
DEV = "cuda"

# Walk length r that rankings of these families end at (eps = 1e-9), for work():
# the recurrence reads the adjacency once per level, and no graph above the
# cache size stays on the chip between levels.
LEVELS = {"er": 20, "rmat": 8, "chunglu": 12}
CACHE_BYTES = 126e6


def listed():
    return [
        # the smallest calls: a small graph ranked again and again (parameter
        # studies, ego networks); latency and launches count
        {"name": "rank-er16k", "do": "rank", "graph": "er", "n": 16384, "deg": 16.0, "k": 100, "precision": 0,
         "directed": False, "half_alpha": False},
        # an ordinary social-network-sized graph, the paper's precision
        {"name": "rank-rmat22", "do": "rank", "graph": "rmat", "n": 1 << 22, "deg": 32.0, "k": 1000, "precision": 0,
         "directed": False, "half_alpha": False},
        # a larger one in FP32-certified mode (walk vectors about the size of L2)
        {"name": "rank-rmat24-fp32cert", "do": "rank", "graph": "rmat", "n": 1 << 24, "deg": 32.0, "k": 1000,
         "precision": 1, "directed": False, "half_alpha": False},
        # the largest: 134 M vertices, int64 offsets, walk vectors far above L2
        {"name": "rank-chunglu27", "do": "rank", "graph": "chunglu", "n": 1 << 27, "deg": 16.0, "k": 100,
         "precision": 0, "directed": False, "half_alpha": False},
        # the same family in FP32-certified mode, an odd size, int32 offsets
        {"name": "rank-chunglu25-fp32cert", "do": "rank", "graph": "chunglu", "n": 33554393, "deg": 16.0, "k": 100,
         "precision": 1, "directed": False, "half_alpha": False},
        # a directed graph (l_r = c_r), ordinary size, top-100
        {"name": "rank-directed-rmat21", "do": "rank", "graph": "rmat", "n": 1999993, "deg": 16.0, "k": 100,
         "precision": 0, "directed": True, "half_alpha": False},
        # one-shot use: a graph in pinned host memory, ranked once
        {"name": "oneshot-rmat21", "do": "oneshot", "graph": "rmat", "n": 1 << 21, "deg": 32.0, "k": 1000,
         "precision": 0, "directed": False, "half_alpha": False},
        # the full certified order of all vertices (the ranking criterion)
        {"name": "full-ranking-er18", "do": "criterion", "criterion": 1, "graph": "er", "n": 262147, "deg": 16.0, "k": 0,
         "precision": 0, "directed": False, "half_alpha": False},
        # a small batch on a graph without hubs: few walk counts change
        {"name": "update-er20-16", "do": "update", "graph": "er", "n": 1 << 20, "deg": 16.0, "k": 100, "precision": 0,
         "directed": False, "half_alpha": False, "m": 16},
        # a batch on the serving graph (hubs: whole levels are repaired)
        {"name": "update-rmat23-1000", "do": "update", "graph": "rmat", "n": 1 << 23, "deg": 32.0, "k": 100,
         "precision": 0, "directed": False, "half_alpha": False, "m": 1000},
        # a stream of uneven batches through the serving loop, FP32-certified levels
        {"name": "serve-rmat20-fp32cert", "do": "serve", "graph": "rmat", "n": 1 << 20, "deg": 32.0, "k": 100,
         "precision": 2, "directed": False, "half_alpha": False, "batches": 6, "max_m": 10000},
        # bounds that a program holds already, certified without allocation
        {"name": "certify-rmat22", "do": "certify", "graph": "rmat", "n": 1 << 22, "deg": 32.0, "k": 1000,
         "precision": 0, "directed": False, "half_alpha": False},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case: the same kinds of work, sizes over the whole range."""
    do = rng.choice(["rank", "rank", "rank", "rank", "oneshot", "criterion", "update", "update", "serve", "certify"])
    hi = {"rank": 6e7, "oneshot": 5e6, "criterion": 2e6, "update": 8e6, "serve": 2e6, "certify": 1e7}[do]
    n = int(_log(rng, 3000 if do in ("rank", "oneshot") else 30000, hi))
    if do == "rank" and n > 1 << 24:
        graph = "chunglu"
    else:
        graph = rng.choice(["er", "er", "chunglu"] if do == "criterion" else ["er", "rmat", "chunglu"])
    deg = {"er": rng.choice([8.0, 16.0]), "rmat": rng.choice([16.0, 32.0]), "chunglu": 16.0}[graph]
    case = {"do": do, "graph": graph, "n": n, "deg": deg, "k": int(_log(rng, 10, 1500)),
            "precision": 0 if do == "criterion" else rng.choice([0, 0, 2]),
            "directed": do in ("rank", "update") and graph != "chunglu" and rng.random() < 0.25,
            "half_alpha": do == "rank" and rng.random() < 0.3}
    if do == "criterion":
        case["criterion"] = rng.choice([1, 1, 2])
        case["k"] = 0
    elif do == "update":
        case["m"] = int(_log(rng, 1, 10000))
    elif do == "serve":
        case["batches"] = rng.randint(2, 6)
        case["max_m"] = int(_log(rng, 30, 10000))
    return case


# ---- graphs ------------------------------------------------------------------
ID_BITS = 31  # keys are (row << 31) | column


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(0x5EED0000 + int(seed))
    return g


def _pairs(case, seed):
    """Generated pairs (u, v), int64, in blocks."""
    n, kind = case["n"], case["graph"]
    total = int(n * case["deg"] / 2) if not case["directed"] else int(n * case["deg"])
    g = _gen(seed)
    if kind == "chunglu":
        # vertex i of the weight order has weight x_m ((i + 0.5) / n)^(-1/tau), capped;
        # an endpoint is drawn by the inverse of the weights' running sum
        tau = 1.1
        x_m = case["deg"] * (tau - 1.0) / tau
        cap = math.sqrt(case["deg"] * n)
        i0 = n * (x_m / cap) ** tau  # the first i0 vertices are at the cap
        b = 1.0 - 1.0 / tau
        tail = x_m * n ** (1.0 / tau) * (n ** b - i0 ** b) / b
        p_cap = i0 * cap / (i0 * cap + tail)
        ids = torch.randperm(n, generator=g, device=DEV, dtype=torch.int32)
    step = 1 << 27
    for a in range(0, total, step):
        m = min(step, total - a)
        if kind == "er":
            yield (torch.randint(0, n, (m,), generator=g, device=DEV), torch.randint(0, n, (m,), generator=g, device=DEV))
        elif kind == "rmat":
            u = torch.zeros(m, dtype=torch.int64, device=DEV)
            v = torch.zeros(m, dtype=torch.int64, device=DEV)
            for _ in range(max(1, (n - 1).bit_length())):
                x = torch.rand(m, generator=g, device=DEV)
                u.mul_(2).add_(x >= 0.76)
                v.mul_(2).add_(((x >= 0.57) & (x < 0.76)) | (x >= 0.95))
            if n & (n - 1):  # a size between two scales: its first n vertices
                keep = (u < n) & (v < n)
                u, v = u[keep], v[keep]
            yield u, v
        else:
            ends = []
            for _ in range(2):
                x = torch.rand(m, generator=g, device=DEV)
                f = torch.rand(m, generator=g, device=DEV)  # the bits below x's last one
                t = (x - p_cap) / (1.0 - p_cap)
                y = (t * (n ** b - i0 ** b) + i0 ** b).clamp_(min=i0 ** b)
                width = y.pow(1.0 / b - 1.0) * ((n ** b - i0 ** b) / b * 2.0 ** -23)
                i = torch.where(x < p_cap, f * i0, y.pow(1.0 / b)).long()
                i += torch.where(x < p_cap, 0.0, f * width).long()
                ends.append(ids[i.clamp_(0, n - 1)].long())
                del x, f, t, y, width, i
            yield ends[0], ends[1]


def _csr_of_keys(n, keys):
    """(rowptr, col) of sorted (row << 31 | column) keys."""
    rows = torch.bincount(keys >> ID_BITS, minlength=n)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(rows, 0, out=rowptr[1:])
    return rowptr, (keys & ((1 << ID_BITS) - 1)).int()


def _csr_of_edges(n, keys):
    """Symmetric CSR of sorted (lo << 31 | hi) edge keys: a row holds its
    smaller neighbours (from the edges turned round), then its larger ones."""
    mask = (1 << ID_BITS) - 1
    turned = torch.unique(((keys & mask) << ID_BITS) | (keys >> ID_BITS))
    small = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    large = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(turned >> ID_BITS, minlength=n), 0, out=small[1:])
    torch.cumsum(torch.bincount(keys >> ID_BITS, minlength=n), 0, out=large[1:])
    m = keys.numel()
    col = torch.empty(2 * m, dtype=torch.int32, device=DEV)
    at = torch.arange(m, device=DEV)
    step = 1 << 28
    for a in range(0, m, step):
        e = slice(a, min(a + step, m))
        col[at[e] + small[1:][keys[e] >> ID_BITS]] = (keys[e] & mask).int()
        col[at[e] + large[turned[e] >> ID_BITS]] = (turned[e] & mask).int()
    return small + large, col


def _keys(case, seed):
    """Sorted keys: edges (lo << 31 | hi), or arcs of a directed graph."""
    parts = []
    for u, v in _pairs(case, seed):
        keep = u != v
        if not case["directed"]:
            u, v = torch.minimum(u, v), torch.maximum(u, v)
        parts.append(((u << ID_BITS) | v)[keep])
        del u, v, keep
    keys = parts[0] if len(parts) == 1 else torch.cat(parts)
    del parts
    return torch.unique(keys)


def _csr(case, keys):
    return _csr_of_keys(case["n"], keys) if case["directed"] else _csr_of_edges(case["n"], keys)


def _deg_max(rowptr):
    return int((rowptr[1:] - rowptr[:-1]).max())


def _batch(case, keys, m, g):
    """m updates, half deletions of existing edges and half insertions of new
    uniform pairs: sorted keys of the deleted and of the inserted edges."""
    n = case["n"]
    m = max(1, min(m, keys.numel() // 4))
    ins = (m + 1) // 2
    gone = keys[torch.unique(torch.randint(0, keys.numel(), (m - ins,), generator=g, device=DEV))]
    u = torch.randint(0, n, (2 * ins + 64,), generator=g, device=DEV)
    v = torch.randint(0, n, (2 * ins + 64,), generator=g, device=DEV)
    keep = u != v
    if not case["directed"]:
        u, v = torch.minimum(u, v), torch.maximum(u, v)
    new = torch.unique(((u << ID_BITS) | v)[keep])
    at = torch.searchsorted(keys, new).clamp_(max=keys.numel() - 1)
    new = new[keys[at] != new]
    return gone, new[torch.randperm(new.numel(), generator=g, device=DEV)[:ins]].sort().values


def _host_batch(gone, new, g):
    """(src, dst, is_insert) as host arrays, in a random order."""
    keys = torch.cat([gone, new])
    ins = torch.cat([torch.zeros_like(gone), torch.ones_like(new)])
    order = torch.randperm(keys.numel(), generator=g, device=DEV)
    keys, ins = keys[order].cpu().numpy(), ins[order].cpu().numpy()
    return ((keys >> ID_BITS).astype(np.int32), (keys & ((1 << ID_BITS) - 1)).astype(np.int32), ins.astype(np.uint8))


def _minus(keys, gone):
    keep = torch.ones(keys.numel(), dtype=torch.bool, device=DEV)
    keep[torch.searchsorted(keys, gone)] = False
    return keys[keep]


def _applied(keys, gone, new):
    return torch.cat([_minus(keys, gone), new]).sort().values


def _batches(case, seed, keys):
    """The case's batches, each drawn on the graph that the ones before it
    leave: (gone, new) each, and the graphs' keys after each."""
    g = _gen(seed + 7919)
    if case["do"] == "update":
        sizes = [case["m"]]
    else:  # sizes log-uniform in [1, max_m]
        r = torch.rand(case["batches"], generator=g, device=DEV).tolist()
        sizes = [max(1, int(math.exp(x * math.log(case["max_m"])))) for x in r]
    out, after = [], []
    for m in sizes:
        b = _batch(case, keys, m, g)
        keys = _applied(keys, *b)
        out.append(b)
        after.append(keys)
    return out, after, g


# ---- a pass --------------------------------------------------------------------
class _State:
    def __del__(self):
        if hasattr(self, "server"):  # a server is released before the handles it serves
            self.server.close()


def _alpha(case, deg_max):
    return 0.5 / max(1, deg_max) if case["half_alpha"] else 0.0


def prepare(case, seed):
    s = _State()
    s.case = case
    n, do = case["n"], case["do"]
    keys = _keys(case, seed)
    s.k = min(case["k"], n)
    dynamic = do in ("update", "serve")
    if dynamic:
        batches, _, g = _batches(case, seed, keys)
        # a pass applies the batches and then takes them back
        s.batches = [_host_batch(gone, new, g) for gone, new in batches]
        s.batches += [_host_batch(new, gone, g) for gone, new in reversed(batches)]
        del batches
    rowptr, col = _csr(case, keys)
    del keys
    deg_max = _deg_max(rowptr)
    s.alpha = _alpha(case, deg_max)
    opts = dict(precision=case["precision"], undirected=0 if case["directed"] else 1)
    if dynamic:
        opts.update(keep_history=1, deg_bound=deg_max + 64)
    s.opts = opts
    s.lower = torch.empty(n, dtype=torch.float64, device=DEV)
    s.upper = torch.empty(n, dtype=torch.float64, device=DEV)
    if do == "oneshot":  # the graph in pinned host memory
        s.rowptr = torch.empty(rowptr.shape, dtype=rowptr.dtype, pin_memory=True)
        s.col = torch.empty(col.shape, dtype=col.dtype, pin_memory=True)
        s.rowptr.copy_(rowptr)
        s.col.copy_(col)
        return s
    s.h = K.Katz(rowptr, col, K.katz_default_opts(**opts))
    del rowptr, col
    if do == "certify":
        s.h.rank(s.alpha, s.k, EPS)
        K.katz_get_bounds(s.h.h, lower=s.lower, upper=s.upper)
        s.h.close()
        s.ids = torch.empty(s.k, dtype=torch.int32, device=DEV)
        s.certified = torch.empty(1, dtype=torch.int32, device=DEV)
    elif dynamic:
        s.h.rank(s.alpha, s.k, EPS)
        if do == "serve":
            s.server = K.Server()
            s.server.attach(s.h, s.k)
        run(s)  # the walk length settles at the largest that any of the graphs needs
    return s


def run(s):
    do, h = s.case["do"], getattr(s, "h", None)
    if do == "rank":
        info = h.rank(s.alpha, s.k, EPS)
        ids = h.ranking(s.k)
        K.katz_get_bounds(h.h, lower=s.lower, upper=s.upper)
        return {"r": info.r, "ids": ids, "lower": s.lower, "upper": s.upper}
    if do == "oneshot":
        h = K.Katz(s.rowptr, s.col, K.katz_default_opts(**s.opts))
        info = h.rank(s.alpha, s.k, EPS)
        ids = h.ranking(s.k)
        K.katz_get_bounds(h.h, lower=s.lower, upper=s.upper)
        h.close()
        return {"r": info.r, "ids": ids, "lower": s.lower, "upper": s.upper}
    if do == "criterion":
        info = h.rank_by(s.case["criterion"], s.alpha, EPS)
        out = {"r": info.r, "lower": s.lower, "upper": s.upper}
        if s.case["criterion"] == K.KATZ_CRIT_RANKING:
            out["ids"] = h.ranking(s.case["n"])
        K.katz_get_bounds(h.h, lower=s.lower, upper=s.upper)
        return out
    if do == "update":
        out = {}
        for i, (src, dst, ins) in enumerate(s.batches):
            info = h.update(src, dst, ins)
            out["r%d" % i] = info.r
            out["ids%d" % i] = h.ranking(s.k)
        K.katz_get_bounds(h.h, lower=s.lower, upper=s.upper)
        out["lower"], out["upper"] = s.lower, s.upper
        return out
    if do == "serve":
        tickets = [s.server.submit(h, src, dst, ins) for src, dst, ins in s.batches]
        answers = [s.server.wait(t) for t in tickets]
        return {"status": np.array([a[0] for a in answers]), "r": np.array([a[2].info.r for a in answers]),
                "ids": np.stack([a[1] for a in answers])}
    K.katz_certify_topk_noalloc(s.lower, s.upper, s.k, EPS, s.ids, s.certified, torch.cuda.current_stream())
    return {"ids": s.ids, "certified": s.certified}


def work(case):
    n, do = case["n"], case["do"]
    nnz = 0.97 * n * case["deg"]
    levels = LEVELS[case["graph"]]
    if do == "certify":  # both bounds of every node
        return {"bytes": 16.0 * n, "flops": 2.0 * n}
    csr = 4.0 * nnz + 4.0 * n
    # per level the adjacency, s_{r-1}, s_r and c; once where all of it stays in L2
    per_level = csr + 32.0 * n
    streamed = per_level * levels if per_level > CACHE_BYTES else per_level
    passes = {"rank": 1, "oneshot": 1, "criterion": 1, "update": 2, "serve": 2 * case.get("batches", 0)}[do]
    if case["graph"] == "er" and do == "update":  # few rows change: the vectors' reads and the touched rows
        return {"bytes": passes * 24.0 * n, "flops": passes * 4.0 * n}
    return {"bytes": passes * streamed + 16.0 * n, "flops": passes * 2.0 * nnz * levels}


# ---- the same in 64 bits ---------------------------------------------------------
class _Exact:
    """Algorithm 1 on one graph, level by level, all nodes kept."""

    def __init__(self, case, keys, alpha, D):
        self.rowptr, col = _csr(case, keys)
        self.n, self.case, self.D = case["n"], case, D
        self.alpha = alpha if alpha > 0 else 1.0 / (D + 1.0)
        self.col = col
        self.s = torch.ones(self.n, dtype=torch.float64, device=DEV)
        self.c = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        self.r = 0

    def step(self):
        y = torch.empty_like(self.s)
        cuts = [0]  # rows in blocks of at most about 2^28 arcs
        while cuts[-1] < self.n:
            at = self.rowptr[cuts[-1]] + (1 << 28)
            cuts.append(max(cuts[-1] + 1, int(torch.searchsorted(self.rowptr, at, right=True)) - 1))
            cuts[-1] = min(cuts[-1], self.n)
        for a, b in zip(cuts, cuts[1:]):
            j0, j1 = int(self.rowptr[a]), int(self.rowptr[b])
            block = torch.sparse_csr_tensor(self.rowptr[a:b + 1] - j0, self.col[j0:j1].long(),
                                            torch.ones(j1 - j0, dtype=torch.float64, device=DEV), size=(b - a, self.n))
            y[a:b] = torch.mv(block, self.s) if j1 > j0 else 0.0
        self.s = self.alpha * y
        self.c = self.c + self.s
        self.r += 1

    def bounds(self):
        gamma = self.D / (1.0 - self.alpha * self.D)
        lower = self.c if self.case["directed"] else self.c + self.alpha * self.s
        return lower, self.c + self.alpha * gamma * self.s

    def holds(self, k):
        """The stopping criterion at this level (top-k; k = n: every pair; 0: score)."""
        lower, upper = self.bounds()
        if k == 0:
            return bool((upper - lower < EPS).all())
        order = torch.sort(lower, descending=True, stable=True).indices
        l, u = lower[order], upper[order]
        return bool((u[1:k] - EPS < l[: k - 1]).all()) and bool((u[k:] - EPS < l[k - 1]).all())

    def until(self, k, r=1):
        while self.r < r or not self.holds(k):
            self.step()
            if self.r > 128:
                raise RuntimeError("not separated")
        return self


def exact(case, seed):
    do, n = case["do"], case["n"]
    if do == "certify" or do == "serve":
        return None  # whole numbers only
    keys = _keys(case, seed)
    rowptr = _csr(case, keys)[0]
    deg_max = _deg_max(rowptr)
    alpha = _alpha(case, deg_max)
    k = min(case["k"], n)
    if do == "criterion" and case["criterion"] == 1:
        k = n
    if do != "update":
        e = _Exact(case, keys, alpha, deg_max).until(k)
        lower, upper = e.bounds()
        out = {"r": e.r, "ids": None, "lower": lower, "upper": upper}
        if do == "criterion" and case["criterion"] != 1:
            del out["ids"]
        return out
    # the walk length of a handle never falls: the largest that either graph needs
    _, after, _ = _batches(case, seed, keys)
    r = _Exact(case, after[0], alpha, deg_max + 64).until(k).r
    e = _Exact(case, keys, alpha, deg_max + 64).until(k, r)
    lower, upper = e.bounds()
    return {"r0": e.r, "ids0": None, "r1": e.r, "ids1": None, "lower": lower, "upper": upper}
