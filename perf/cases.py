"""The work a program has this library do, as cases that can be timed.

Kinds of a case (its ``kind``), each one call or one short sequence of calls
of the public binding:

- ``eval``: support and Eq. (1) of a population held on the device, on a handle
  whose pair table is built (``ebic_eval_population_dev``).
- ``host``: the same through host buffers on a handle that was only loaded
  (``ebic_eval_population`` as the README calls it, falling counts included).
- ``batch``: many problems of uneven size in one launch (``ebic_batch_eval``).
- ``search``: a whole EBIC run, Steps 1-5 (``ebic_run_generations``).
- ``rows``: Steps 6-7, the rows of found series (``ebic_extract_rows[_approx]``).
- ``predict`` / ``train``: the surrogate's scoring and its Adam steps.
- ``matrix``: a new matrix placed, its pair table built, a first population
  evaluated, everything released.

Matrices are drawn on the GPU: normal or log-normal background with planted
order-preserving biclusters, every second one decreasing.  Populations are half
ordered subsequences of the plants (a third of them with one foreign column
inserted) and half random series, like a population halfway through a search.
"""
import math

import numpy as np
import torch

import paper_1801_03039_gb300 as eb

F, EMB, H = 80, 64, 256          # the surrogate's layer widths
LR = 1e-3


def listed():
    return [
        # the smallest call: one fitness pass of the 200 x 20 configuration
        dict(name="eval-tiny-200x20", kind="eval", rows=200, cols=20, pop=100, len_min=2, len_max=6,
             both=False, missing=0.0, tuned=False),
        # one fitness pass of the paper's synthetic scale
        dict(name="eval-paper-1000x100", kind="eval", rows=1000, cols=100, pop=600, len_min=3,
             len_max=20, both=False, missing=0.0, tuned=False),
        # the expression-shaped pass bench.py times, with the launch shape the autotuner picks
        dict(name="eval-expression-20000x200", kind="eval", rows=20000, cols=200, pop=4096,
             len_min=3, len_max=30, both=False, missing=0.0, tuned=True),
        # ragged sizes, missing values, rising plus falling rows
        dict(name="eval-both-7777x123", kind="eval", rows=7777, cols=123, pop=1501, len_min=2,
             len_max=25, both=True, missing=0.02, tuned=False),
        # the paper's scalability shape through the host call, no pair table
        dict(name="host-25000x100", kind="host", rows=25000, cols=100, pop=2000, len_min=3,
             len_max=20, missing=0.0),
        # 64 problems of uneven size (restarts and datasets side by side)
        dict(name="batch-64-uneven", kind="batch", problems=64, rows_min=500, rows_max=50000,
             cols_min=20, cols_max=500, pop_min=256, pop_max=2048, len_max=30),
        # the paper-scale search: P = 600, 1,000 generations
        dict(name="search-paper-1000x100", kind="search", rows=1000, cols=100, pop=600, len_min=3,
             len_max=20, generations=1000),
        # the start of a search on the expression shape, the largest population
        dict(name="search-expression-20000x200", kind="search", rows=20000, cols=200, pop=4096,
             len_min=3, len_max=30, generations=20),
        # Steps 6-7 on a full top-rank list, negative trends included
        dict(name="rows-20000x200", kind="rows", rows=20000, cols=200, pop=100, len_min=3,
             len_max=20, falling=True, breaks=0),
        # scores of one screened generation's candidates (P = 600, 8 per attempt)
        dict(name="predict-38432", kind="predict", cols=100, n=38432, len_min=3, len_max=20),
        # surrogate training at the minibatch bench.py uses
        dict(name="train-4096x24", kind="train", cols=100, n=120000, len_min=3, len_max=20,
             batch=4096, steps=24),
        # a new dataset: placed, table built, first population evaluated, released
        dict(name="matrix-20000x200", kind="matrix", rows=20000, cols=200, pop=1000, len_min=3,
             len_max=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "host", "batch", "search", "rows", "predict", "train",
                       "matrix"])
    if kind == "batch":
        return dict(kind=kind, problems=rng.randint(4, 40), rows_min=rng.randint(200, 600),
                    rows_max=_log(rng, 2000, 45000), cols_min=rng.randint(15, 30),
                    cols_max=_log(rng, 60, 450), pop_min=rng.randint(100, 300),
                    pop_max=_log(rng, 400, 2000), len_max=rng.randint(8, 30))
    if kind in ("predict", "train"):
        c = dict(kind=kind, cols=rng.randint(20, 200), len_min=rng.randint(2, 4),
                 len_max=rng.randint(6, 20))
        if kind == "predict":
            return dict(c, n=_log(rng, 250, 36000))
        return dict(c, n=_log(rng, 20000, 110000), batch=_log(rng, 200, 4096),
                    steps=rng.randint(4, 20))
    cols = _log(rng, 20, 190)
    len_max = min(cols, rng.randint(6, 30))
    c = dict(kind=kind, rows=_log(rng, 150, 19000), cols=cols, pop=_log(rng, 60, 4000),
             len_min=rng.randint(2, 4), len_max=len_max)
    if kind == "eval":
        c.update(both=rng.random() < 0.3, missing=rng.choice([0.0, 0.0, 0.02]),
                 tuned=rng.random() < 0.5)
    elif kind == "host":
        c.update(missing=rng.choice([0.0, 0.0, 0.02]), pop=_log(rng, 60, 2000))
    elif kind == "search":
        c.update(pop=_log(rng, 60, 900), generations=_log(rng, 10, 300),
                 rows=_log(rng, 150, 10000))
    elif kind == "rows":
        c.update(pop=_log(rng, 5, 100), falling=rng.random() < 0.6,
                 breaks=rng.choice([0, 0, 1, 2]))
    else:
        c.update(pop=_log(rng, 60, 1000))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _matrix(g, rng, R, C, missing=0.0, lognormal=False):
    """A [R, C] fp32 matrix on the GPU and the column orders of its plants."""
    A = torch.randn(R, C, generator=g, device="cuda")
    plants = []
    for b in range(int(rng.integers(3, 7))):
        nr = int(rng.integers(max(4, R // 100), max(8, R // 25) + 1))
        nc = int(rng.integers(min(4, C), max(4, min(30, C // 3)) + 1))
        rows = torch.randperm(R, generator=g, device="cuda")[:nr]
        order = torch.randperm(C, generator=g, device="cuda")[:nc]
        v = torch.randn(len(rows), nc, generator=g, device="cuda").sort(dim=1).values
        if b % 2:
            v = v.flip(1)
        A[rows[:, None], order[None, :]] = v
        plants.append(order.flip(0) if b % 2 else order)
    if lognormal:
        A = A.exp()
    if missing > 0.0:
        A[torch.rand(R, C, generator=g, device="cuda") < missing] = float("nan")
    return A, plants


def _series(g, n, C, lmin, lmax, plants=(), planted=0.5):
    """n series of distinct columns: padded columns [n, lmax] and lengths [n]."""
    dev = "cuda"
    pad = torch.rand(n, C, generator=g, device=dev).argsort(dim=1)[:, :lmax]
    if pad.shape[1] < lmax:
        pad = torch.cat([pad, pad.new_zeros(n, lmax - pad.shape[1])], dim=1)
    length = torch.randint(lmin, min(lmax, C) + 1, (n,), generator=g, device=dev)
    if not plants:
        return pad, length
    width = torch.tensor([len(p) for p in plants], device=dev)
    W = int(width.max())
    table = torch.zeros(len(plants), W, dtype=torch.long, device=dev)
    other = torch.zeros(len(plants), C, dtype=torch.long, device=dev)
    n_other = torch.zeros(len(plants), dtype=torch.long, device=dev)
    for i, p in enumerate(plants):
        table[i, :len(p)] = p
        rest = torch.ones(C, dtype=torch.bool, device=dev)
        rest[p] = False
        rest = rest.nonzero().flatten()
        other[i, :len(rest)] = rest
        n_other[i] = len(rest)
    which = torch.randint(0, len(plants), (n,), generator=g, device=dev)
    w = width[which]
    top = torch.clamp(w, max=lmax)
    low = torch.clamp(top, max=lmin)
    plen = low + (torch.rand(n, generator=g, device=dev) * (top - low + 1)).long().clamp(max=C)
    plen = torch.minimum(plen, top)
    key = torch.rand(n, W, generator=g, device=dev)
    key[torch.arange(W, device=dev)[None, :] >= w[:, None]] = 2.0
    rank = key.argsort(dim=1).argsort(dim=1)
    pos = torch.where(rank < plen[:, None], torch.arange(W, device=dev)[None, :], W)
    pos = pos.sort(dim=1).values[:, :lmax].clamp(max=W - 1)
    sub = table[which[:, None], pos]
    if sub.shape[1] < lmax:
        sub = torch.cat([sub, sub.new_zeros(n, lmax - sub.shape[1])], dim=1)
    # a third of them get one foreign column
    ins = (torch.rand(n, generator=g, device=dev) < 1 / 3) & (plen < min(lmax, C)) & \
        (n_other[which] > 0)
    at = (torch.rand(n, generator=g, device=dev) * (plen + 1)).long()
    alien = other[which, (torch.rand(n, generator=g, device=dev) * n_other[which]).long().clamp(max=C - 1)]
    t = torch.arange(lmax, device=dev)[None, :]
    left = (t - 1).clamp(min=0).expand(n, lmax)
    with_alien = torch.where(t < at[:, None], sub, torch.where(t == at[:, None], alien[:, None],
                                                               sub.gather(1, left)))
    sub = torch.where(ins[:, None], with_alien, sub)
    plen = plen + ins.long()
    use = torch.rand(n, generator=g, device=dev) < planted
    return torch.where(use[:, None], sub, pad), torch.where(use, plen, length)


def _cbf(pad, length):
    """Offsets [P + 1] and concatenated columns, int32, on the GPU."""
    off = torch.zeros(len(length) + 1, dtype=torch.int32, device="cuda")
    off[1:] = length.cumsum(0)
    keep = torch.arange(pad.shape[1], device="cuda")[None, :] < length[:, None]
    return off, pad[keep].to(torch.int32).contiguous()


def _sigma(R):
    return max(10, R // 400)


def _data(case, seed):
    """Matrix and population of a single-matrix case."""
    g, rng = _gen(seed), np.random.default_rng(seed)
    A, plants = _matrix(g, rng, case["rows"], case["cols"], case.get("missing", 0.0),
                        lognormal=case["rows"] > 5000)
    pad, length = _series(g, case["pop"], case["cols"], min(case["len_min"], case["cols"]),
                          min(case["len_max"], case["cols"]), plants)
    return A, pad, length


def _batch_data(case, seed):
    """(matrix, padded columns, lengths) of every problem of a batch; the sizes
    are the case's, the values the seed's."""
    g, rng = _gen(seed), np.random.default_rng(seed)
    sizes = np.random.default_rng(case["problems"])
    for _ in range(case["problems"]):
        R = int(sizes.integers(case["rows_min"], case["rows_max"] + 1))
        C = int(sizes.integers(case["cols_min"], case["cols_max"] + 1))
        P = int(sizes.integers(case["pop_min"], case["pop_max"] + 1))
        A, plants = _matrix(g, rng, R, C)
        pad, length = _series(g, P, C, 3, min(case["len_max"], C), plants)
        yield A, pad, length


def _params(case, seed):
    """Flat fp32 surrogate parameters of the library's layout, He-scaled."""
    rng, C = np.random.default_rng(seed), case["cols"]
    w1 = rng.standard_normal((F, H)) * math.sqrt(2 / 67)
    w1[67:] = 0.0
    parts = [0.1 * rng.standard_normal((C, EMB)), w1, 0.05 * rng.standard_normal(H),
             rng.standard_normal((H, H)) * math.sqrt(2 / H), 0.05 * rng.standard_normal(H),
             rng.standard_normal(H) / math.sqrt(H), np.zeros(1)]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def _sur_data(case, seed):
    """The 1,000-row matrix behind a surrogate and its series."""
    g, rng = _gen(seed), np.random.default_rng(seed)
    A, plants = _matrix(g, rng, 1000, case["cols"])
    lmax = min(case["len_max"], case["cols"])
    pad, length = _series(g, case["n"], case["cols"], case["len_min"], lmax, plants)
    fit = torch.empty(0, dtype=torch.float64)
    if case["kind"] == "train":
        # fitness of the right kind: a heavy tail above many zeros
        z = torch.randn(case["n"], generator=g, device="cuda", dtype=torch.float64)
        fit = torch.where(z > 0.3, length * torch.exp(z), torch.zeros_like(z)).contiguous()
    return A, pad, length, fit


# ---------------------------------------------------------------------------
# what a program keeps between calls
# ---------------------------------------------------------------------------
class State:
    """Handles and buffers of one prepared case, released with the object."""

    def __init__(self, case):
        self.case = case
        self.handles, self.batch, self.sur = [], None, None

    def __del__(self):
        if self.batch is not None:
            eb.ebic_batch_free(self.batch)
        if self.sur is not None:
            eb.ebic_surrogate_free(self.sur)
        for h in self.handles:
            eb.ebic_free(h)

    def load(self, A):
        torch.cuda.current_stream().synchronize()
        h = eb.ebic_load_matrix_dev(A.contiguous())
        self.handles.append(h)
        return h

    def population(self, pad, length):
        self.off, self.cols = _cbf(pad, length)
        self.P, self.total = len(length), int(self.cols.numel())
        self.outputs()

    def outputs(self):
        self.inc = torch.zeros(self.P, dtype=torch.int32, device="cuda")
        self.dec = torch.zeros(self.P, dtype=torch.int32, device="cuda")
        self.fit = torch.zeros(self.P, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    s = State(case)
    kind = case["kind"]
    if kind == "batch":
        items, s.out = [], []
        for A, pad, length in _batch_data(case, seed):
            h = s.load(A)
            off, cols = _cbf(pad, length)
            P = len(length)
            inc = torch.zeros(P, dtype=torch.int32, device="cuda")
            fit = torch.zeros(P, dtype=torch.float64, device="cuda")
            s.out.append((inc, fit, off, cols))
            items.append((off, cols, P, int(cols.numel()), _sigma(A.shape[0]), inc, fit))
        s.batch = eb.ebic_batch_create(s.handles, items, eb.BATCH_AUTOTUNE | eb.BATCH_GRAPH |
                                       eb.BATCH_BUILD_TABLES)
        return s
    if kind in ("predict", "train"):
        A, pad, length, fit = _sur_data(case, seed)
        h = s.load(A)
        s.sur = eb.ebic_surrogate_create(h, pad.shape[1], seed)
        eb.ebic_surrogate_params(s.sur, _params(case, seed))
        s.seq, s.len = pad.to(torch.int16).contiguous(), length.to(torch.int32).contiguous()
        s.stride, s.target = pad.shape[1], fit
        s.y = torch.empty(case["n"], dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        return s
    A, pad, length = _data(case, seed)
    s.sigma = _sigma(case["rows"])
    if kind == "matrix":
        s.A = A.contiguous()
        s.population(pad, length)
        return s
    h = s.load(A)
    if kind == "search":
        s.params = eb.ebic_default_params(
            pop_size=case["pop"], len_min=min(case["len_min"], case["cols"]),
            len_max=pad.shape[1], iterations=case["generations"], sigma=s.sigma, toprank_size=100,
            tournament_k=2, seed=seed)
        s.top = np.full((100, pad.shape[1]), -1, np.int32)
        s.top_len, s.top_fit = np.zeros(100, np.int32), np.zeros(100)
        return s
    if kind in ("host", "rows"):
        off, cols = _cbf(pad, length)
        s.off, s.cols = off.cpu().numpy(), cols.cpu().numpy()
        if kind == "rows":
            s.found = np.full(case["pop"] * case["rows"], -1, np.int32)
        return s
    s.population(pad, length)
    eb.ebic_build_pair_table(h)
    s.mode = eb.SUPPORT_INC_PLUS_DEC if case["both"] else eb.SUPPORT_INC
    if case["tuned"]:
        eb.ebic_autotune_eval(h, s.off, s.cols, s.P, s.total, s.sigma, s.mode, s.inc,
                              s.dec if case["both"] else None, s.fit, flags=eb.TUNE_COLD_L2)
    return s


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "eval":
        dec = s.dec if case["both"] else None
        eb.ebic_eval_population_dev(s.handles[0], s.off, s.cols, s.P, s.total, s.sigma, s.mode,
                                    s.inc, dec, s.fit)
        return {"inc": s.inc, "dec": dec, "fitness": s.fit}
    if kind == "host":
        inc, dec, fit = eb.ebic_eval_population(s.handles[0], s.off, s.cols, s.sigma)
        return {"inc": inc, "dec": dec, "fitness": fit}
    if kind == "batch":
        eb.ebic_batch_eval(s.batch)
        return {"inc": torch.cat([o[0] for o in s.out]), "fitness": torch.cat([o[1] for o in s.out])}
    if kind == "search":
        top, fit, st = eb.ebic_run_generations(s.handles[0], s.params)
        k = len(top)
        s.top_len[:k] = [len(x) for x in top]
        s.top_fit[:k] = fit
        for i, x in enumerate(top):
            s.top[i, :len(x)] = x
        return {"found": k, "length": s.top_len, "series": s.top, "fitness": s.top_fit,
                "generations": st["generations_done"],
                "evaluations": st["evaluations_total"], "hits": st["tabu_hits_total"]}
    if kind == "rows":
        mode = eb.ROWS_RISING_OR_FALLING if case["falling"] else eb.ROWS_RISING
        if case["breaks"]:
            rows = eb.ebic_extract_rows_approx(s.handles[0], s.off, s.cols, case["breaks"], mode)
        else:
            rows = eb.ebic_extract_rows(s.handles[0], s.off, s.cols, mode)
        np.concatenate(rows, out=s.found[:sum(map(len, rows))])
        return {"count": np.array([len(r) for r in rows]), "rows": s.found}
    if kind == "predict":
        eb.ebic_surrogate_predict(s.sur, s.seq, s.len, s.stride, case["n"], s.y)
        return {"y": s.y}
    if kind == "train":
        loss = eb.ebic_surrogate_train(s.sur, case["steps"], case["batch"], LR, s.seq, s.len,
                                       s.stride, s.target, case["n"])
        return {"loss": np.float32(loss), "params": eb.ebic_surrogate_params(s.sur)}
    h = eb.ebic_load_matrix_dev(s.A)
    eb.ebic_build_pair_table(h)
    eb.ebic_eval_population_dev(h, s.off, s.cols, s.P, s.total, s.sigma, eb.SUPPORT_INC, s.inc, None,
                                s.fit)
    eb.ebic_free(h)
    return {"inc": s.inc, "fitness": s.fit}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _mean_len(case):
    return (case["len_min"] + min(case["len_max"], case["cols"])) / 2


def work(case):
    """bytes: inputs and outputs once.  flops: row comparisons (an early exit
    per row leaves e - 1 of them for a random series) or multiply-adds x 2."""
    kind = case["kind"]
    if kind == "batch":
        n = case["problems"]
        R = (case["rows_min"] + case["rows_max"]) / 2
        C = (case["cols_min"] + case["cols_max"]) / 2
        P = (case["pop_min"] + case["pop_max"]) / 2
        L = (3 + case["len_max"]) / 2
        return {"bytes": n * (4 * R * C + P * (4 * L + 16)), "flops": n * P * R * (math.e - 1)}
    if kind in ("predict", "train"):
        n = case["n"] if kind == "predict" else case["batch"] * case["steps"]
        par = case["cols"] * EMB + F * H + H * H + 3 * H + 1
        mac = n * (F * H + H * H + H)
        io = n * (2 * _mean_len(case) + 8)
        if kind == "predict":
            return {"bytes": 4 * par + io, "flops": 2 * mac}
        return {"bytes": 12 * par * 2 + io + 8 * case["n"], "flops": 6 * mac}
    R, C, P = case["rows"], case["cols"], case["pop"]
    cbf = P * (4 * _mean_len(case) + 4)
    if kind == "search":
        g = case["generations"] + 1
        return {"bytes": 4 * R * C + g * P * (2 * _mean_len(case) + 12),
                "flops": g * P * R * (math.e - 1)}
    if kind == "rows":
        return {"bytes": 4 * R * C + cbf + 4 * P * R / 40, "flops": P * R * (math.e - 1)}
    tests = P * R * (math.e - 1) * (2 if kind == "host" or case.get("both") else 1)
    out = P * (16 if kind == "host" or case.get("both") else 12)
    table = C * C * R / 8 if kind == "matrix" else 0
    return {"bytes": 4 * R * C + table + cbf + out,
            "flops": tests + (C * C * R if kind == "matrix" else 0)}


# ---------------------------------------------------------------------------
# the same in 64 bits, by plain torch
# ---------------------------------------------------------------------------
def _alive(A, pad, length, falling=False):
    """[P, R] booleans: row k rises (or falls) strictly along series i."""
    At = A.t().contiguous()
    keep = At.new_ones((len(length), A.shape[0]), dtype=torch.bool)
    for t in range(pad.shape[1] - 1):
        on = (t + 1 < length).nonzero().flatten()
        for part in on.split(512):
            a, b = At[pad[part, t]], At[pad[part, t + 1]]
            keep[part] &= (a > b) if falling else (a < b)
    return keep


def _fitness(n, length, sigma):
    n = n.double()
    f = torch.log((n - 1).clamp(min=1)) * torch.exp2((n - sigma).clamp(max=0)) * length
    return torch.where(n > 1, f, torch.zeros_like(f))


def _mlp(par, C, x, seq, length, len_scale):
    """Scores by the flat fp64 parameters; x: the two column-statistics features."""
    emb, w1, b1, w2, b2, w3, b3 = torch.split(
        par, [C * EMB, F * H, H, H * H, H, H, 1])
    on = (torch.arange(seq.shape[1], device=seq.device)[None, :] < length[:, None]).double()
    e = (emb.view(C, EMB)[seq] * on[:, :, None]).sum(1)
    stats = (x[seq] * on[:, :, None]).sum(1) / length.clamp(min=1)[:, None].double()
    f = torch.cat([e, stats, (length.double() / len_scale)[:, None]], dim=1)
    h1 = torch.relu(f @ w1.view(F, H)[:67] + b1)
    h2 = torch.relu(h1 @ w2.view(H, H) + b2)
    return h2 @ w3 + b3


def _philox(c0, c1, c2, seed):
    """Words 0 and 1 of Philox-4x32-10 for counters (c0, c1, c2, 0), key seed."""
    m32 = np.uint64(0xFFFFFFFF)
    x = [c0.astype(np.uint64), np.full_like(c0, c1, np.uint64), np.full_like(c0, c2, np.uint64),
         np.zeros_like(c0, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = x[0] * np.uint64(0xD2511F53), x[2] * np.uint64(0xCD9E8D57)
        x = [(p1 >> np.uint64(32)) ^ x[1] ^ np.uint64(k0), p1 & m32,
             (p0 >> np.uint64(32)) ^ x[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x[0], x[1]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("search", "rows"):
        return None                     # whole runs and whole numbers
    if kind == "batch":
        fits = []
        for A, pad, length in _batch_data(case, seed):
            n = _alive(A, pad, length).sum(1)
            fits.append(_fitness(n, length, _sigma(A.shape[0])))
        return {"inc": None, "fitness": torch.cat(fits)}
    if kind in ("predict", "train"):
        A, pad, length, fit = _sur_data(case, seed)
        C, L = case["cols"], pad.shape[1]
        A = A.double()
        x = torch.stack([A.mean(0), A.std(0, unbiased=False)], dim=1)
        par = torch.from_numpy(_params(case, seed)).cuda().double()
        if kind == "predict":
            y = [_mlp(par, C, x, pad[i:i + 8192], length[i:i + 8192], L)
                 for i in range(0, case["n"], 8192)]
            return {"y": torch.cat(y)}
        t = torch.log1p(fit)
        t = (t - t.mean()) / t.std(unbiased=False)
        m, v, n, B = torch.zeros_like(par), torch.zeros_like(par), case["n"], case["batch"]
        for k in range(1, case["steps"] + 1):
            hi, lo = _philox(np.arange(B), k, 0x5EED, seed)
            idx = torch.from_numpy((((hi << np.uint64(32)) | lo) % np.uint64(n)).astype(np.int64)).cuda()
            par.requires_grad_(True)
            loss = ((_mlp(par, C, x, pad[idx], length[idx], L) - t[idx]) ** 2).mean()
            gr, = torch.autograd.grad(loss, par)
            par = par.detach()
            m, v = 0.9 * m + 0.1 * gr, 0.999 * v + 0.001 * gr * gr
            par = par - LR * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
        return {"loss": loss.detach().item(), "params": par}
    A, pad, length = _data(case, seed)
    n = _alive(A, pad, length).sum(1)
    if case.get("both"):
        n = n + _alive(A, pad, length, falling=True).sum(1)
    out = {"inc": None, "fitness": _fitness(n, length, _sigma(case["rows"]))}
    if kind == "host" or case.get("both"):
        out["dec"] = None
    return out
