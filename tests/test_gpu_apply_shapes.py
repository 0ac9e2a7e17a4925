"""Where the apply, Get, Put and export change kernel or split: batch sizes at
the edges of the one-cluster plan and of the one-kernel reduce, row ids of one
to three sort passes, dims at the edges of lane groups, segments and vector
widths, runs cut into several nodes, and row buffers of every alignment.

Gradients are small multiples of 2^-10, so every run's sum is exact in any
order: rows and state must equal the fp32 oracle's bit for bit whatever the
order of the additions.
"""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import assert_bits, dev, host, make_pair, torch_cuda

pytestmark = pytest.mark.gpu


def _grads(rng, n, dim):
    return (rng.integers(-8, 9, size=(n, dim)) * 2.0**-10).astype(np.float32)


def _cfg(dim):
    cfg = W.tiny()
    cfg.dim = dim
    return cfg


def _shifted(a, floats):
    """A device copy of `a` that starts `floats` floats after a 256-byte boundary."""
    torch = torch_cuda()
    buf = torch.empty(a.size + floats, dtype=torch.float32, device="cuda:0")
    view = buf[floats:].view(a.shape)
    view.copy_(torch.from_numpy(a))
    return view


def _check_table(store, ref, keys, what):
    u = np.unique(keys)
    w, G = store.export(dev(u))
    rw, rG = ref.export(u)
    assert_bits(host(w), rw, f"rows: {what}")
    assert_bits(host(G), rG, f"state: {what}")
    assert np.array_equal(host(store.find(dev(u))), ref.find(u)), f"row ids: {what}"


# 1, a warp, one block and its neighbours, blocks of 1 lookup a thread up to the
# cluster's 16, 2 lookups a thread up to the largest plan, and one past it
PLAN_SIZES = [1, 33, 1023, 1024, 1025, 2049, 5000, 16384, 16385, 32767, 32768, 32769]


@pytest.mark.parametrize("capacity", [600, 40_000, 3_000_000])  # row ids of 10, 16 and 22 bits: 1, 2 and 3 passes
@pytest.mark.parametrize("mix", ["zipf", "distinct", "one key"])
def test_plan_edges(capacity, mix):
    torch_cuda()
    store, ref = make_pair(_cfg(4), capacity=capacity, max_batch=max(PLAN_SIZES), lr=0.125, eps=1e-8)
    rng = np.random.default_rng(capacity)
    universe = rng.choice(1 << 40, min(capacity - 10, 40_000), replace=False).astype(np.int64)
    known = universe[: len(universe) * 3 // 4]  # the others get their rows in an apply
    for s in range(0, len(known), max(PLAN_SIZES)):
        store.insert(dev(known[s:s + max(PLAN_SIZES)]))
        ref.insert(known[s:s + max(PLAN_SIZES)])
    seen = []
    for n in PLAN_SIZES:
        if mix == "zipf":
            keys = universe[np.minimum(rng.zipf(1.3, n) - 1, len(universe) - 1)]
        elif mix == "distinct":
            keys = rng.permutation(np.resize(universe, n))
        else:
            keys = np.full(n, universe[n % len(universe)])
        keys[n // 2] = -1 if n == 5000 else keys[n // 2]  # the reserved key: skipped, and reported
        grads = _grads(rng, n, 4)
        store.apply_grad(dev(keys), dev(grads))
        ok = keys != -1
        ref.apply_grad(keys[ok], grads[ok])
        if not ok.all():
            assert store.sync() != 0
            store.clear_status()
        assert store.last_unique() == len(np.unique(keys[ok])), f"distinct rows of {n} lookups"
        seen.append(keys[ok])
        assert store.size() == ref.size()
    _check_table(store, ref, np.concatenate(seen), mix)
    assert store.sync() == 0
    store.close()


def test_plan_without_insertion_skips_absent_keys():
    torch_cuda()
    store, ref = make_pair(_cfg(8), capacity=5000, max_batch=9000, insert_on_miss=False, lr=0.125)
    rng = np.random.default_rng(5)
    universe = rng.choice(1 << 40, 6000, replace=False).astype(np.int64)
    store.insert(dev(universe[:4000]))
    ref.insert(universe[:4000])
    keys = universe[rng.integers(0, 6000, 9000)]
    grads = _grads(rng, 9000, 8)
    store.apply_grad(dev(keys), dev(grads))
    assert store.sync() != 0  # some keys are not in the table
    store.clear_status()
    there = np.isin(keys, universe[:4000])
    ref.apply_grad(keys[there], grads[there])
    _check_table(store, ref, keys[there], "apply beside absent keys")
    store.close()


# one float, both sides of 32 vectors of 4, 8 and 16 bytes, whole and ragged segments, the widest
DIMS = [1, 2, 3, 6, 31, 33, 50, 64, 66, 100, 128, 130, 132, 200, 256, 260, 512, 1000, 1024]


@pytest.mark.parametrize("dim", DIMS)
def test_rows_of_every_width(dim):
    torch = torch_cuda()
    sizes = [700, 33_000]  # the one-kernel reduce, and a kernel per run length
    store, ref = make_pair(_cfg(dim), capacity=4000, max_batch=max(sizes), lr=0.125, eps=1e-8)
    rng = np.random.default_rng(dim)
    universe = rng.choice(1 << 40, 3990, replace=False).astype(np.int64)
    p = 1.0 / np.arange(1, 3991) ** 0.9
    p /= p.sum()
    for n in sizes:
        keys = universe[rng.choice(3990, n, p=p)]
        want, _, _ = ref.get(keys)
        assert_bits(host(store.get(dev(keys))), want, f"Get, {n} lookups")
        for shift in (0, 2, 1) if dim <= 256 else (0,):  # 16-, 8- and 4-byte aligned row buffers
            grads = _grads(rng, n, dim)
            store.apply_grad(dev(keys), _shifted(grads, shift))
            ref.apply_grad(keys, grads)
            out = _shifted(np.zeros((n, dim), np.float32), shift)
            store.get(dev(keys), out=out)
            want, _, _ = ref.get(keys)
            assert_bits(host(out), want, f"Get after the apply, {n} lookups, shift {shift}")
        values = rng.standard_normal((n, dim), dtype=np.float32)
        store.put(dev(keys), _shifted(values, 2 if dim <= 256 else 0))
        ref.put(keys, values)
        _check_table(store, ref, keys, f"{n} lookups")
    uniq = universe[::-1].copy()
    rows, state = (rng.random((3990, dim), dtype=np.float32) for _ in range(2))
    store.import_(dev(uniq), dev(rows), dev(state))
    w, G = store.export(dev(uniq))
    assert_bits(host(w), rows, "imported rows")
    assert_bits(host(G), state, "imported state")
    assert store.sync() == 0
    store.close()


@pytest.mark.parametrize("n", [32_768, 100_000, (1 << 19) + 77])
@pytest.mark.parametrize("dim", [4, 64, 132])
def test_hot_runs_of_several_nodes(n, dim):
    """Runs of thousands of chunks (several nodes of 256, trees of several
    levels), of 257 chunks, of one node, and short ones around them."""
    torch_cuda()
    store, ref = make_pair(_cfg(dim), capacity=2000, max_batch=n, lr=0.125, eps=1e-8)
    rng = np.random.default_rng(n + dim)
    universe = rng.choice(1 << 40, 1990, replace=False).astype(np.int64)
    store.insert(dev(universe))
    ref.insert(universe)
    chunk = 64 if n >= 1 << 19 else 16
    lens = [n // 2, min(n // 4, 257 * chunk), 17 * chunk, 16 * chunk + 1, 33, 32, 5, 4]
    keys = np.repeat(universe[: len(lens)], lens)
    keys = rng.permutation(np.concatenate([keys, universe[rng.integers(8, 1990, n - len(keys))]]))
    for _ in range(2):  # the second apply starts from the counters the first left
        grads = _grads(rng, n, dim)
        store.apply_grad(dev(keys), dev(grads))
        ref.apply_grad(keys, grads)
    _check_table(store, ref, keys, f"{n} lookups")
    assert store.sync() == 0
    store.close()


@pytest.mark.parametrize("n", [40, 3000, 300_000])
def test_put_of_hot_keys_keeps_the_last_value(n):
    torch_cuda()
    store, ref = make_pair(_cfg(8), capacity=3000, max_batch=n)
    rng = np.random.default_rng(n)
    universe = rng.choice(1 << 40, 2990, replace=False).astype(np.int64)
    for alpha in (1.05, 1.6):
        keys = universe[np.minimum(rng.zipf(alpha, n) - 1, 2989)]
        values = rng.standard_normal((n, 8), dtype=np.float32)
        store.put(dev(keys), dev(values))
        ref.put(keys, values)
        _check_table(store, ref, keys, f"Put of {n}")
    store.close()


@pytest.mark.parametrize("dim", [4, 50, 128, 260])
@pytest.mark.parametrize("n", [1, 9, 2432, 2433, 4865, 16_384, 16_385])
def test_get_gives_new_keys_rows(n, dim):
    """Gets with no new key, new keys in one warp, some everywhere, and all new, on
    both sides of the sizes whose miss path runs inside the Get's kernel; each
    Get starts from the counters the one before left."""
    torch_cuda()
    store, ref = make_pair(_cfg(dim), capacity=60_000, max_batch=n)
    rng = np.random.default_rng(n + dim)
    fresh = iter(rng.choice(1 << 40, 55_000, replace=False).astype(np.int64))
    known = np.array([next(fresh) for _ in range(50)], np.int64)
    store.insert(dev(known[: min(n, 50)]))
    ref.insert(known[: min(n, 50)])
    known = known[: min(n, 50)]
    for share in (0.0, 0.0, 1.0 / n, 0.3, 0.0, 1.0):
        keys = known[rng.integers(0, len(known), n)]
        new = np.array([next(fresh) for _ in range(int(np.ceil(n * share * 0.8)))], np.int64)
        at = rng.choice(n, int(round(n * share)), replace=False)
        if len(at):
            keys[at] = new[rng.integers(0, len(new), len(at))]  # some of them more than once
        want, _, _ = ref.get(keys)
        assert_bits(host(store.get(dev(keys))), want, f"Get, {share:.2f} of the lookups new")
        assert store.size() == ref.size()
        assert np.array_equal(host(store.find(dev(keys))), ref.find(keys))
    grads = _grads(rng, n, dim)
    store.apply_grad(dev(keys), dev(grads))
    ref.apply_grad(keys, grads)
    _check_table(store, ref, keys, "apply after the Gets")
    assert store.sync() == 0
    store.close()


@pytest.mark.parametrize("dim", [3, 64, 128, 512])
@pytest.mark.parametrize("n", [65, 2432, 9728, 16_384])
def test_get_whose_new_keys_are_in_few_blocks(n, dim):
    """The blocks that met a new key rank the new keys of their own lookups and
    share the rows: new keys in the first lookups, in the last ones (more of them
    than a warp takes at a time), in two far ends, one alone, and again and again
    the same one."""
    torch_cuda()
    store, ref = make_pair(_cfg(dim), capacity=4000, max_batch=n, state_init=0.25)
    rng = np.random.default_rng(n + dim)
    known = rng.choice(1 << 40, 500, replace=False).astype(np.int64)
    for s in range(0, 500, n):
        store.insert(dev(known[s:s + n]))
        ref.insert(known[s:s + n])
    fresh = iter((1 << 41) + rng.permutation(4000).astype(np.int64))
    few, end = min(40, n), min(300, n)
    for at in (np.arange(few), np.arange(n - end, n), np.r_[np.arange(few // 2), np.arange(n - few // 2, n)],
               np.array([n // 2]), None, np.array([], np.int64)):
        keys = known[rng.integers(0, 500, n)]
        if at is None:
            keys[rng.permutation(n)[: n // 2]] = next(fresh)
        else:
            keys[at] = [next(fresh) for _ in range(len(at))]
        want, _, _ = ref.get(keys)
        assert_bits(host(store.get(dev(keys))), want, "Get")
        assert store.size() == ref.size()
        _check_table(store, ref, keys, "after the Get")
    assert store.sync() == 0
    store.close()


@pytest.mark.parametrize("dim", [1, 6, 50, 64, 128, 132, 512])
@pytest.mark.parametrize("n", [700, 8192, 32_768])
def test_apply_gives_new_keys_rows_before_it_reduces_them(n, dim):
    """Applies whose keys are new (all of them, or some) in runs of every length,
    through the one-cluster plan: each row starts from its init values and state,
    whichever kernel (by n and dim) and run length reduces it; the next apply
    finds none new; and a full table gives the first keys rows and skips the rest."""
    torch_cuda()
    lens = [n // 3, 9 * 16 + 1, 33, 32, 20, 5, 4, 4, 3, 2, 2]  # 16 lookups a chunk of a long run
    opts = dict(max_batch=n, lr=0.125, eps=1e-8, state_init=0.25)
    store, ref = make_pair(_cfg(dim), capacity=3 * n, **opts)
    rng = np.random.default_rng(n + dim)
    fresh = (1 << 41) + rng.permutation(6 * n).astype(np.int64)
    used = 0
    known = np.zeros(0, np.int64)
    for share in (1.0, 0.0, 0.2):
        runs = fresh[used:used + len(lens)]
        ones = fresh[used + len(lens):used + n]
        used += n
        keys = np.concatenate([np.repeat(runs, lens), ones])[:n]
        if share < 1:
            at = rng.permutation(n)[: int(n * (1 - share))]
            keys = rng.permutation(keys)
            keys[at] = known[rng.integers(0, len(known), len(at))]
        keys = rng.permutation(keys)
        grads = _grads(rng, n, dim)
        store.apply_grad(dev(keys), dev(grads))
        ref.apply_grad(keys, grads)
        assert store.size() == ref.size() and store.last_unique() == len(np.unique(keys))
        _check_table(store, ref, keys, f"{share:.1f} of the lookups new")
        known = np.unique(np.concatenate([known, keys]))
    assert store.sync() == 0
    store.close()
    room = n // 2 + 3
    store, ref = make_pair(_cfg(dim), capacity=room, **opts)
    keys = fresh[used:used + n]
    grads = _grads(rng, n, dim)
    store.apply_grad(dev(keys), dev(grads))
    assert store.sync() == 5  # MLKV_ERR_FULL
    store.clear_status()
    ref.apply_grad(keys[:room], grads[:room])
    assert store.size() == ref.size() == room
    _check_table(store, ref, keys[:room], "a table filled by an apply")
    store.close()


@pytest.mark.parametrize("dim,edge", [(16, 1 << 16), (20, 200_000), (32, 400_000), (96, 400_000), (100, 200_000)])
@pytest.mark.parametrize("insert", [True, False])
def test_get_at_the_edge_of_the_asynchronous_copies(dim, edge, insert):
    """One lookup fewer and as many as where a Get leaves the kernel that moves
    rows by asynchronous copies, known keys beside new (or absent) ones."""
    torch_cuda()
    store, ref = make_pair(_cfg(dim), capacity=30_000, max_batch=edge, insert_on_miss=insert)
    rng = np.random.default_rng(dim)
    universe = rng.choice(1 << 40, 29_000, replace=False).astype(np.int64)
    store.insert(dev(universe[:20_000]))
    ref.insert(universe[:20_000])
    for n, known in ((edge - 1, 25_000), (edge, 29_000)):
        keys = universe[rng.integers(0, known, n)]
        want, _, _ = ref.get(keys)
        got = host(store.get(dev(keys)))
        assert np.array_equal(np.isnan(got), np.isnan(want))
        assert_bits(np.nan_to_num(got), np.nan_to_num(want), f"Get of {n}")
        if not insert:
            assert store.sync() == 7  # MLKV_ERR_NOT_FOUND
            store.clear_status()
        assert store.size() == ref.size()
    assert store.sync() == 0
    store.close()


@pytest.mark.parametrize("n,dim,shift", [(4096, 256, 1), (4096, 1024, 0), (16_384, 256, 0), (32_768, 128, 0)])
def test_trees_of_the_most_segments(n, dim, shift):
    """One run of all of the batch's lookups, then runs just past 32, in as many
    row segments as the one-kernel reduce takes: the combine trees' counters, of
    every level, and again from what the first apply left."""
    torch_cuda()
    store, ref = make_pair(_cfg(dim), capacity=2000, max_batch=n, lr=0.125, eps=1e-8)
    rng = np.random.default_rng(n + dim)
    universe = rng.choice(1 << 40, 1990, replace=False).astype(np.int64)
    store.insert(dev(universe))
    ref.insert(universe)
    for keys in (np.full(n, universe[3]), np.resize(np.repeat(universe, 33), n), np.full(n, universe[5])):
        grads = _grads(rng, n, dim)
        store.apply_grad(dev(keys), _shifted(grads, shift))
        ref.apply_grad(keys, grads)
        _check_table(store, ref, keys, "one apply")
    assert store.sync() == 0
    store.close()


@pytest.mark.parametrize("n", [62_914, 62_915])
def test_get_into_host_memory_at_the_edge_of_the_asynchronous_copies(n):
    """One row fewer and as many bytes as where a Get whose rows go to host memory leaves them."""
    torch = torch_cuda()
    store, ref = make_pair(_cfg(100), capacity=30_000, max_batch=n)
    rng = np.random.default_rng(n)
    universe = rng.choice(1 << 40, 29_000, replace=False).astype(np.int64)
    store.insert(dev(universe[:20_000]))
    ref.insert(universe[:20_000])
    keys = universe[rng.integers(0, 29_000, n)]
    out = torch.empty((n, 100), dtype=torch.float32).pin_memory()
    store.get_host(torch.from_numpy(keys).pin_memory(), out)
    assert store.sync() == 0
    torch.cuda.synchronize()
    want, _, _ = ref.get(keys)
    assert_bits(out.numpy(), want, "Get into host memory")
    store.close()
