"""Workloads that the store's speed is measured on.

A case is one call, or one step of a training loop, on a table that has been
restored from a checkpoint (rows and Adagrad state imported), through
`EmbeddingStore`.  Table and batch shapes follow `workloads/configs.py` (the
recommendation, knowledge-graph, graph-network, tiered and YCSB-shaped
workloads and the tiny check) with smaller tables, so that several fit the
card, and the range of dims the tests cover.

A training loop runs Get(batch t), the model, apply(batch t), Get(batch t+1),
...  A pass is taken from the middle of it: the Get of the batch has been made,
its gradients are in hand, and the pass applies them and makes the next Get.
The next Get asks for the same keys, so what it returns are the updated rows
of every lookup.
"""
import functools
import math

import numpy as np
import torch

from paper_2504_01506_gb300 import EmbeddingStore

LR = 0.01
EPS = 1e-8
ROW_SIGMA = 0.01      # rows of a trained table
GRAD_SIGMA = 1e-3     # gradients per lookup
RELATION_BASE = 1 << 62
CHUNK_FLOATS = 1 << 27  # floats of rows per import call while a table is restored


def listed():
    return [
        # Serving: the features of 16 samples (26 tables) are looked up; nothing but latency.
        dict(name="serve_get", kind="get", tables=26, keys=26 * 40_000, dim=128, n=416, alpha=1.2),
        # The repository's tiny check as a training step: a small model's whole table, narrow rows.
        dict(name="tiny_step", kind="step", tables=1, keys=100_000, dim=16, n=4_096, alpha=1.05),
        # A small recommendation model: 512 samples x 26 features, dim 32.
        dict(name="small_step", kind="step", tables=26, keys=26 * 40_000, dim=32, n=512 * 26, alpha=1.2),
        # Word-vector training at dim 50 (rows that are no multiple of 16 bytes), an odd batch, and after the
        # apply the batch's rows and their state are exported, as a loop with delta checkpoints does.
        dict(name="odd_delta", kind="delta", tables=1, keys=1_999_993, dim=50, n=100_003, alpha=1.0),
        # Wide rows (dims above 128 take more than one vector a lane), a mid-sized batch.
        dict(name="wide_step", kind="step", tables=1, keys=1_500_000, dim=512, n=65_536, alpha=0.8),
        # Knowledge-graph embedding: heads and tails Zipf(0.9), relations, uniform negatives; dim 100.
        dict(name="kg_step", kind="kg", tables=1, keys=16_000_000, dim=100, n=200_000, alpha=0.9),
        # Recommendation training: 65,536 samples x 26 features, dim 128.
        dict(name="dlrm_step", kind="step", tables=26, keys=26 * 1_000_000, dim=128, n=65_536 * 26, alpha=1.2),
        # Graph-network minibatch: 8,192 seeds with 10 + 250 sampled neighbours each, dim 64.
        dict(name="gnn_step", kind="step", tables=1, keys=25_000_000, dim=64, n=8_192 * 261, alpha=1.0 / 1.1),
        # YCSB-shaped batch: half the operations read, half write (upsert), Zipf(0.99) keys, 1 KiB values.
        dict(name="ycsb_mix", kind="mix", tables=1, keys=5_000_000, dim=256, n=1_048_576, alpha=0.99),
        # Planning a batch: its distinct keys and their counts.
        dict(name="dedup", kind="dedup", tables=26, keys=26 * 1_000_000, dim=16, n=65_536 * 26, alpha=1.2),
        # A table larger than its HBM cache: look-ahead of the next batch beside the apply, then its Get.
        dict(name="tiered_step", kind="tiered", tables=1, keys=2_000_000, dim=128, n=131_072, alpha=1.1),
        # The same step through the host-buffer calls: keys and gradients from pinned memory, rows back to it.
        dict(name="host_step", kind="host", tables=26, keys=26 * 100_000, dim=128, n=8_192 * 26, alpha=1.2),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """Batch sizes from a few dozen lookups to two million, dims 4 to 1024 (odd ones and ones that are no multiple
    of 4 among them), uniform to strongly skewed keys, one table or 26, every kind of call."""
    kind = rng.choice(["get", "step", "step", "step", "step", "kg", "delta", "mix", "dedup", "tiered", "host"])
    if rng.random() < 0.3:
        dim = rng.choice([5, 10, 18, 25, 50, 67, 75, 90, 130, 150, 202])
    else:
        dim = rng.choice([4, 8, 12, 16, 24, 32, 48, 64, 64, 100, 128, 128, 200, 256, 300, 512, 768, 1024])
    hi = {"tiered": 131_072, "host": 212_992, "delta": 400_000, "kg": 800_000}.get(kind, 2_138_112)
    most = 27_000_000 if kind == "host" else 200_000_000  # floats of one batch
    n = _spread(rng, 8_192 if kind == "tiered" else 64, min(hi, most // dim))
    keys = _spread(rng, 20_000, min(25_000_000, 3_000_000_000 // dim))
    if kind == "tiered":
        keys = min(keys, 256_000_000 // dim)
    tables = 26 if kind in ("get", "step", "dedup", "host") and rng.random() < 0.4 else 1
    alpha = rng.choice([0.0, 0.6, 0.8, 0.9, 0.99, 1.05, 1.2, 1.3])
    return dict(kind=kind, tables=tables, keys=keys // tables * tables, dim=dim, n=max(n, 26) // tables * tables,
                alpha=alpha)


# --- inputs -----------------------------------------------------------------

RELATIONS = 15_000
TIER_BATCHES = 32  # distinct batches in turn: together they hold more rows than the cache


def _gen(seed, stream):
    g = torch.Generator("cuda")
    g.manual_seed((seed * 1_000_003 + stream * 7_919 + 17) & 0x7FFF_FFFF_FFFF)
    return g


def _zipf(count, keys, alpha, gen):
    """`count` draws from P(r) ~ (r + 1)^-alpha over [0, keys), the ranks scattered over the range."""
    if alpha == 0.0:
        return torch.randint(keys, (count,), generator=gen, device="cuda")
    w = torch.arange(1, keys + 1, device="cuda", dtype=torch.float64).pow_(-alpha)
    cdf = torch.cumsum(w, 0)
    u = torch.rand(count, generator=gen, device="cuda", dtype=torch.float64) * cdf[-1]
    rank = torch.searchsorted(cdf, u).clamp_(max=keys - 1)
    step = max(1, int(keys * 0.6180339887) | 1)
    while math.gcd(step, keys) != 1:
        step += 2
    return (rank * step + keys // 3) % keys


def _total(case):
    return case["keys"] + (RELATIONS if case["kind"] == "kg" else 0)


def _key_of(case, i):
    """The 64-bit key of table entry i (a tensor of indices): table * 2^32 + row, relations above 2^62."""
    if case["kind"] == "kg":
        return torch.where(i < case["keys"], i, RELATION_BASE + (i - case["keys"]))
    per = case["keys"] // case["tables"]
    return (torch.div(i, per, rounding_mode="floor") << 32) + i % per


def _lookups(case, seed, batch=0):
    """Table entries that one batch looks up."""
    gen = _gen(seed, 100 + batch)
    n, keys = case["n"], case["keys"]
    if case["kind"] == "kg":  # heads, relations, tails, negatives
        q = n // 4
        parts = [_zipf(q, keys, case["alpha"], gen),
                 keys + torch.randint(RELATIONS, (q,), generator=gen, device="cuda"),
                 _zipf(q, keys, case["alpha"], gen),
                 torch.randint(keys, (n - 3 * q,), generator=gen, device="cuda")]
        return torch.cat(parts)
    if case["kind"] == "dedup":  # a known number of distinct entries, each looked up once or more
        few = torch.randperm(keys, generator=gen, device="cuda")[:_planned(case)]
        i = torch.cat([few, few[_zipf(n - few.numel(), few.numel(), case["alpha"], gen)]])
        return i[torch.randperm(n, generator=gen, device="cuda")]
    t = case["tables"]
    per = keys // t
    i = _zipf(n, per, case["alpha"], gen)
    if t > 1:  # sample-major: the lookups of a sample are adjacent, each table's hot rows in another place
        f = torch.arange(n, device="cuda") % t
        i = f * per + (i + f * (per // t)) % per
    return i


def _planned(case):
    """Distinct keys of a batch to deduplicate."""
    return max(1, min(case["keys"], int(0.18 * case["n"])))


def _chunks(case):
    step = max(1, min(CHUNK_FLOATS // case["dim"], _max_batch(case)))
    return [(a, min(a + step, _total(case))) for a in range(0, _total(case), step)]


def _max_batch(case):
    return case["n"] if case["kind"] == "tiered" else max(case["n"], 262_144)


def _table(case, seed, k, a, b):
    """Rows and Adagrad state of entries a .. b-1 (chunk k) of the checkpoint: sums of some squared gradients."""
    gen = _gen(seed, 10_000 + k)
    shape = (b - a, case["dim"])
    rows = torch.empty(shape, device="cuda").normal_(0.0, ROW_SIGMA, generator=gen)
    state = torch.empty(shape, device="cuda").uniform_(GRAD_SIGMA ** 2, 50 * GRAD_SIGMA ** 2, generator=gen)
    return rows, state


def _normal(case, seed, stream, n, sigma):
    return torch.empty((n, case["dim"]), device="cuda").normal_(0.0, sigma, generator=_gen(seed, stream))


def _reads(case, seed):
    """Which operations of a mixed batch read (half of them; the others write)."""
    return torch.randperm(case["n"], generator=_gen(seed, 3), device="cuda") < case["n"] // 2


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    store = EmbeddingStore(dim=case["dim"], capacity=_total(case), max_batch=_max_batch(case), lr=LR, eps=EPS, seed=1,
                           hbm_cache_rows=2 * n + 64 if kind == "tiered" else 0)
    for k, (a, b) in enumerate(_chunks(case)):
        rows, state = _table(case, seed, k, a, b)
        store.import_(_key_of(case, torch.arange(a, b, device="cuda")), rows, state)
    s = {"kind": kind, "store": store}
    if kind == "tiered":
        s["batches"] = [_key_of(case, _lookups(case, seed, j)) for j in range(TIER_BATCHES)]
        s["at"] = 0
        s["grads"] = _normal(case, seed, 2, n, GRAD_SIGMA)
        store.get(s["batches"][0])
        return s
    entries = _lookups(case, seed)
    keys = _key_of(case, entries)
    if kind == "mix":
        read = _reads(case, seed)
        s["read"], s["write"] = keys[read], keys[~read]
        s["values"] = _normal(case, seed, 4, s["write"].numel(), ROW_SIGMA)
    elif kind == "host":
        s["keys"] = keys.cpu().pin_memory()
        s["grads"] = _normal(case, seed, 2, n, GRAD_SIGMA).cpu().pin_memory()
        s["out"] = torch.empty((n, case["dim"])).pin_memory()
        store.get_host(s["keys"], s["out"])
    else:
        s["keys"] = keys
        if kind in ("step", "kg", "delta"):
            s["grads"] = _normal(case, seed, 2, n, GRAD_SIGMA)
            store.get(keys)
    return s


def run(state):
    store, kind = state["store"], state["kind"]
    if kind == "get":
        return store.get(state["keys"])
    if kind in ("step", "kg"):
        store.apply_grad(state["keys"], state["grads"])
        return store.get(state["keys"])
    if kind == "delta":
        store.apply_grad(state["keys"], state["grads"])
        return store.export(state["keys"])
    if kind == "mix":
        rows = store.get(state["read"])
        store.put(state["write"], state["values"])
        return rows, store.get(state["write"])
    if kind == "dedup":
        return store.dedup(state["keys"])
    if kind == "tiered":
        b = state["batches"]
        now, nxt = b[state["at"]], b[(state["at"] + 1) % len(b)]
        state["at"] = (state["at"] + 1) % len(b)
        store.lookahead(nxt)
        store.apply_grad(now, state["grads"])
        return store.get(nxt)
    store.apply_grad_host(state["keys"], state["grads"])
    store.get_host(state["keys"], state["out"])
    return state["out"]


# --- what a pass cannot do without ------------------------------------------

@functools.lru_cache(maxsize=64)
def _distinct(keys, alpha, n):
    """Expected number of distinct entries of n draws."""
    if n <= 0:
        return 0.0
    p = np.arange(1, keys + 1, dtype=np.float64) ** -alpha
    return float(-np.expm1(-n * (p / p.sum())).sum())


def _expected_distinct(case, n):
    if case["kind"] == "kg":
        q = n // 4
        zipf = _distinct(case["keys"], case["alpha"], 2 * q) + _distinct(case["keys"], 0.0, n - 3 * q)
        return zipf + _distinct(RELATIONS, 0.0, q)
    t = case["tables"]
    return t * _distinct(case["keys"] // t, case["alpha"], n // t)


def work(case):
    """Keys, gradients and values read once, outputs written once, each distinct row (and in an apply its state)
    read and, where it changes, written once, and one 16-byte index entry per distinct key."""
    kind, n, d = case["kind"], case["n"], case["dim"]
    u = _planned(case) if kind == "dedup" else _expected_distinct(case, n)
    if kind == "get":
        return {"bytes": n * (8 + 4 * d) + u * (16 + 4 * d), "flops": 0.0}
    if kind == "dedup":
        return {"bytes": n * 8 + u * (16 + 12), "flops": 0.0}
    if kind == "mix":
        h = n / 2
        v = _expected_distinct(case, n // 2)
        return {"bytes": n * 8 + 3 * h * 4 * d + v * (32 + 8 * d), "flops": 0.0}
    flops = n * d + 6 * u * d
    if kind == "delta":  # the rows and state exported are those just written
        return {"bytes": n * (8 + 12 * d) + u * (16 + 16 * d), "flops": flops}
    if kind == "tiered":  # the next batch's rows are read too
        return {"bytes": n * (16 + 8 * d) + u * (32 + 20 * d), "flops": flops}
    return {"bytes": n * (8 + 8 * d) + u * (16 + 16 * d), "flops": flops}


def tolerance(case):
    """Gets, Puts and dedups move values and are exact.  Updated rows and state are 32-bit sums and one Adagrad step:
    another order of a run's sum moves them by a few roundings (5e-8 off 64 bits as measured, either way)."""
    if case["kind"] in ("get", "mix", "dedup"):
        return "exact"
    return {"rel": 3e-7, "max": 3e-5}


def exact(case, seed):
    kind, n, d = case["kind"], case["n"], case["dim"]
    if kind == "dedup":
        return None
    batch = _lookups(case, seed)
    wanted = _lookups(case, seed, 1) if kind == "tiered" else batch
    uniq = torch.unique(torch.cat([batch, wanted]))
    w = torch.empty((uniq.numel(), d), device="cuda", dtype=torch.float64)
    G = torch.empty_like(w)
    for k, (a, b) in enumerate(_chunks(case)):
        rows, state = _table(case, seed, k, a, b)
        lo, hi = int(torch.searchsorted(uniq, a)), int(torch.searchsorted(uniq, b))
        w[lo:hi] = rows[uniq[lo:hi] - a].double()
        G[lo:hi] = state[uniq[lo:hi] - a].double()
    at = torch.searchsorted(uniq, batch)
    if kind == "get":
        return w[at]
    if kind == "mix":
        read = _reads(case, seed)
        rows = w[at[read]]
        vals = _normal(case, seed, 4, int((~read).sum()), ROW_SIGMA).double()
        put = at[~read]  # the later write of a key wins
        last = torch.full((uniq.numel(),), -1, device="cuda", dtype=torch.int64)
        last.scatter_reduce_(0, put, torch.arange(put.numel(), device="cuda"), "amax")
        return rows, vals[last[put]]
    g = torch.zeros_like(w)
    grads = _normal(case, seed, 2, n, GRAD_SIGMA)
    step = max(1, (1 << 27) // d)
    for a in range(0, n, step):
        g.index_add_(0, at[a:a + step], grads[a:a + step].double())
    hit = torch.zeros(uniq.numel(), device="cuda", dtype=torch.bool)
    hit[at] = True
    # lr and eps as the table holds them, in 32 bits
    lr, eps = float(np.float32(LR)), float(np.float32(EPS))
    G += g * g
    w -= torch.where(hit[:, None], lr * g / (G.sqrt() + eps), torch.zeros_like(g))
    if kind == "delta":
        return w[at], G[at]
    return w[torch.searchsorted(uniq, wanted)]
