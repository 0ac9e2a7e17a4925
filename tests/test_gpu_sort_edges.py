"""The sort and the dedup's output at the edges of their tiles: batches of one
lookup fewer and more than tiles of 2,048 (the sort below 2^19 lookups) and
4,096 (the dedup's output), the first batch past the one-cluster plan, runs that
start in one tile and end several tiles later, and keys without a row (sorted
last, in no run).

Gradients are small multiples of 2^-10, so every run's sum is exact in any
order: rows and state must equal the fp32 oracle's bit for bit."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_helpers import assert_bits, dev, host, make_pair, torch_cuda

pytestmark = pytest.mark.gpu

N_KEYS = 30_000
# row ids of one, two and three passes (the last with an odd digit width)
CAPACITIES = [31_000, 200_000, 3_000_000]


def _keys(rng, universe, n, mix):
    if mix == "one key":
        return np.full(n, universe[-1], dtype=np.int64)
    if mix == "distinct":  # shuffled, every key as often as any other (to one)
        return rng.permutation(np.resize(universe, n))
    k = universe[rng.integers(0, 5, n)]  # runs over several tiles between runs of one
    one = rng.random(n) < 0.2
    k[one] = rng.choice(universe, int(one.sum()))
    return k


@pytest.mark.parametrize("mix", ["one key", "distinct", "few hot"])
def test_dedup_tile_edges(mix):
    torch_cuda()
    sizes = [1, 2, 2047, 2048, 2049, 4095, 4096, 4097, 8192, 12_289, 40_961]
    store, _ = make_pair(W.tiny(), capacity=CAPACITIES[1], max_batch=max(sizes))
    rng = np.random.default_rng(11)
    universe = rng.choice(1 << 40, N_KEYS, replace=False).astype(np.int64)
    store.insert(dev(universe))
    for n in sizes:
        keys = _keys(rng, universe, n, mix)
        for lost in (0, n // 3, n):  # lookups whose key has no row
            k = keys.copy()
            k[rng.permutation(n)[:lost]] = -5
            present = k[k != -5]
            uniq, counts = store.dedup(dev(k))
            uniq, counts = host(uniq), host(counts)
            ou, oc, _ = oracle.dedup(present)
            o, g = np.argsort(ou), np.argsort(uniq)
            assert np.array_equal(uniq[g], ou[o]), f"keys, {n} lookups, {lost} without a row"
            assert np.array_equal(counts[g].astype(np.int64), oc[o]), f"counts, {n} lookups, {lost} without a row"
            if len(uniq):
                assert np.all(np.diff(host(store.find(dev(uniq)))) > 0), "in row order"
    assert store.sync() == 0


@pytest.mark.parametrize("capacity", CAPACITIES)
@pytest.mark.parametrize("mix", ["one key", "distinct", "few hot"])
def test_apply_tile_edges(capacity, mix):
    torch_cuda()
    sizes = [32_769, 34_815, 34_816, 34_817, 100_003, (1 << 19) - 2047, (1 << 19) - 1, 1 << 19]
    cfg = W.tiny()
    cfg.dim = 2
    store, ref = make_pair(cfg, capacity=capacity, max_batch=max(sizes), lr=0.125, eps=1e-8)
    rng = np.random.default_rng(12)
    universe = rng.choice(1 << 40, N_KEYS, replace=False).astype(np.int64)
    store.insert(dev(universe))
    ref.insert(universe)
    for n in sizes:
        keys = _keys(rng, universe, n, mix)
        grads = (rng.integers(-8, 9, size=(n, cfg.dim)) * 2.0**-10).astype(np.float32)
        store.apply_grad(dev(keys), dev(grads))
        ref.apply_grad(keys, grads)
        assert store.last_unique() == len(np.unique(keys)), f"distinct rows, {n} lookups"
        w, G = store.export(dev(universe))
        rw, rG = ref.export(universe)
        assert_bits(host(w), rw, f"rows, {n} lookups")
        assert_bits(host(G), rG, f"state, {n} lookups")
    assert store.sync() == 0
