"""Graphs with more pairs than edges, near the sizes where a rule turns on one
or the other, against the oracle and the counts of each graph alone."""
import numpy as np
import pytest
import torch

import oracle
from paper_1907_09575_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tc():
    from paper_1907_09575_gb300 import tc as _tc
    _tc.load()
    oracle.build()
    return _tc


def random_pairs(n, pairs, seed):
    rng = np.random.default_rng(seed)
    return rng.integers(0, n, pairs).astype(np.int32), rng.integers(0, n, pairs).astype(np.int32), n


def repeated(scale, pairs, times, seed):
    s, d = inputs.rmat(seed, scale, pairs)
    order = np.random.default_rng(seed).permutation(times * pairs)
    return np.tile(s, times)[order], np.tile(d, times)[order], 1 << scale


def build(tc, hs, hd, n):
    return tc.preprocess(torch.from_numpy(hs).cuda(), torch.from_numpy(hd).cuda(), n)


# more than 2^19 pairs, at most 2^19 edges: zones by the pairs, a batch's size by the edges
MANY = {"random": lambda: random_pairs(800, 600_000, 1),
        "rmat": lambda: (*inputs.rmat(3, 15, 560_000), 1 << 15),
        "repeated": lambda: repeated(14, 140_000, 4, 2),
        "small": lambda: random_pairs(500, 20_000, 3)}


@pytest.mark.parametrize("members", [["random"], ["rmat"], ["repeated"], ["small", "random", "repeated"],
                                     ["repeated", "small"], ["random", "rmat", "random"]])
@pytest.mark.parametrize("tuning", [{}, {"table_mode": 1}, {"small_max_outdeg": 16, "slice_max": 64}])
def test_batch(tc, members, tuning):
    t = tc.Tuning()
    for k, v in tuning.items():
        setattr(t, k, v)
    made = {k: MANY[k]() for k in members}
    want = {k: oracle.count(*made[k]) for k in made}
    graphs = [build(tc, *made[k]) for k in members]
    alone = 0
    for k, g in zip(members, graphs):
        assert g.count(tuning=t) == want[k]
        alone += sum(g.count_stats()["probes"])
    b = tc.Batch(graphs, tuning=t)
    assert b.count().tolist() == [want[k] for k in members]
    if "slice_max" not in tuning:                  # a CTA unit a slice, a warp's pivots have none
        assert sum(b.count_stats()["probes"]) == alone
    if not tuning:
        b.autotune(reps=1)
        assert b.count().tolist() == [want[k] for k in members]
    b.free()
    for g in graphs:
        g.free()


@pytest.mark.parametrize("pairs", [(1 << 21) - 1, 1 << 21, 1 << 22, (1 << 22) + 1])
@pytest.mark.parametrize("components", [False, True])
def test_units_are_planned_once(tc, pairs, components):
    """The units preprocessing built are those the first default count asks
    for, whatever share of the pairs are edges."""
    n = 1 << 15
    rng = np.random.default_rng(pairs)
    s, d = (torch.from_numpy(rng.integers(0, n // 8, pairs).astype(np.int32)).cuda() for _ in range(2))
    s[: pairs // 2], d[: pairs // 2] = s[pairs // 2: 2 * (pairs // 2)].clone(), d[pairs // 2: 2 * (pairs // 2)].clone()
    g = tc.preprocess_components(s, d, [0, n // 2, n]) if components else tc.preprocess(s, d, n)
    assert g.stats()["m"] < 1 << 21
    torch.cuda.synchronize()
    tc.profile_enable()
    got = int(tc.count_components(g).sum()) if components else g.count()
    launched = tc.profile_read()
    tc.profile_enable(False)
    assert "k_unit_fill" not in launched, launched
    t = tc.tuning_default()
    t.warp_unit_tasks = 5
    assert g.count(tuning=t) == got
    g.free()


def build_ms(tc, s, d, n):
    best = 1e9
    for _ in range(3):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        tc.preprocess(s, d, n).free()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("shape", ["one pair", "16 vertices", "hub", "blocks", "shuffled"])
def test_large_inputs_of_few_edges(tc, shape):
    """More than 2^26 pairs (the sorted path) with few distinct ones: the graph
    is that of the distinct pairs, and one counter's share of the duplicates
    does not hold up the rest."""
    pairs = (1 << 26) + 77
    gen = torch.Generator(device="cuda").manual_seed(5)
    at = torch.arange(pairs, device="cuda")
    if shape == "one pair":
        hs, hd, n = np.array([3], np.int32), np.array([7], np.int32), 10
    elif shape == "16 vertices":
        i, j = np.triu_indices(16, 1)
        hs, hd, n = i.astype(np.int32), j.astype(np.int32), 16
    elif shape == "hub":                      # every edge's larger id is the hub's
        hs, n = np.arange(4000, dtype=np.int32), 4001
        hd = np.full(4000, 4000, np.int32)
    else:
        hs, hd = inputs.rmat(7, 14, 100_000)
        n = 1 << 14
    if shape == "blocks":                     # each pair's copies beside one another
        pick = at * hs.size // pairs
    else:
        pick = torch.randint(0, hs.size, (pairs,), generator=gen, device="cuda")
        pick[: hs.size] = torch.arange(hs.size, device="cuda")
    s, d = (torch.from_numpy(x).cuda()[pick] for x in (hs, hd))
    del pick
    swap = (at & 1).bool()
    s, d = torch.where(swap, s, d), torch.where(swap, d, s)
    del at, swap
    want, want_t, facts = oracle.count(hs, hd, n, per_vertex=True, stats=True)
    g = tc.preprocess(s, d, n)
    total, t = g.count(per_vertex=True)
    assert total == want and np.array_equal(t.cpu().numpy().astype(np.uint64), want_t)
    assert (g.stats()["m"], g.stats()["max_deg"]) == (facts["m"], facts["max_deg"])
    g.free()
    mine = build_ms(tc, s, d, n)
    s, d = (torch.randint(0, 1 << 20, (pairs,), generator=gen, dtype=torch.int32, device="cuda") for _ in range(2))
    assert mine < 2 * build_ms(tc, s, d, 1 << 20)
