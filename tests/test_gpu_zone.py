"""Dense zones of the count (rows' top labels as bit blocks), against the
oracle: the hubs' number around the zone size and several zones, more blocks
than there is room for, every way of counting a graph that has them."""
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


def hub_graph(hubs, leaves, per_leaf, density, seed):
    """`leaves` vertices joined to per_leaf random hubs each, the hubs to one
    another with the given density; ids scattered."""
    rng = np.random.default_rng(seed)
    n = hubs + leaves
    ids = rng.permutation(n).astype(np.int32)
    a = rng.integers(0, hubs, (leaves, per_leaf))
    s = [np.repeat(np.arange(hubs, n), per_leaf)]
    d = [a.ravel()]
    k = int(density * hubs * (hubs - 1) / 2)
    s.append(rng.integers(0, hubs, k))
    d.append(rng.integers(0, hubs, k))
    s, d = np.concatenate(s), np.concatenate(d)
    return ids[s], ids[d], n


def check(tc, hs, hd, n):
    want, want_t = oracle.count(hs, hd, n, per_vertex=True)
    s, d = torch.from_numpy(hs).cuda(), torch.from_numpy(hd).cuda()
    g = tc.preprocess(s, d, n)
    total, t = g.count(per_vertex=True)
    assert total == want and np.array_equal(t.cpu().numpy().astype(np.uint64), want_t)
    assert g.count() == want
    probes = sum(g.count_stats()["probes"])
    b = tc.Batch([g, g])
    assert b.count().tolist() == [want, want]
    assert sum(b.count_stats()["probes"]) == 2 * probes
    b.free()
    t2 = tc.tuning_default()
    t2.table_mode, t2.small_max_outdeg = 1, 16
    assert g.count(tuning=t2) == want
    g.offload()
    total, t, ts = g.count_tiled(1 << 30, per_vertex=True)
    assert total == want and np.array_equal(t, want_t) and ts["probes"] == probes
    g.free()
    return want


@pytest.mark.parametrize("hubs", [200, 2047, 2048, 2049, 4097, 9001])
@pytest.mark.parametrize("density", [0.02, 0.4])
def test_hubs(tc, hubs, density):
    assert check(tc, *hub_graph(hubs, 6000, 80, density, hubs)) > 0


def test_more_blocks_than_room(tc):
    # rows of 36 hubs each: a block a row against one block for 128 edges
    assert check(tc, *hub_graph(400, 30000, 36, 0.5, 3)) > 0


@pytest.mark.parametrize("scale,pairs", [(16, 1 << 21), (18, 1 << 23), (20, (1 << 24) + 1)])
def test_rmat(tc, scale, pairs):
    # the last one is preprocessed step by step
    hs, hd = inputs.rmat(scale, scale, pairs)
    check(tc, hs, hd, 1 << scale)


def test_components(tc):
    parts = [hub_graph(300, 3000, 50, 0.3, 1), hub_graph(2500, 4000, 70, 0.1, 2), hub_graph(50, 100, 40, 0.9, 3)]
    prefix = np.concatenate([[0], np.cumsum([p[2] for p in parts])])
    hs, hd = (np.concatenate([p[e] + b for p, b in zip(parts, prefix)]).astype(np.int32) for e in (0, 1))
    g = tc.preprocess_components(torch.from_numpy(hs).cuda(), torch.from_numpy(hd).cuda(), prefix)
    got = tc.count_components(g).tolist()
    assert got == [oracle.count(p[0].astype(np.int32), p[1].astype(np.int32), p[2]) for p in parts]
    g.free()


@pytest.mark.parametrize("k", [5795, 6001])
def test_dense_graph_beyond_the_persistent_form(tc, k):
    """K_k of more than 2^24 pairs: few rows, nearly all of them in several
    zones; making their blocks takes less than the deduplication."""
    i, j = torch.triu_indices(k, k, 1, device="cuda")
    p = torch.randperm(i.numel(), generator=torch.Generator().manual_seed(k)).cuda()
    s, d = (x[p].to(torch.int32) for x in (i, j))
    assert s.numel() > 1 << 24
    tc.preprocess(s, d, k).free()
    tc.profile_enable()
    g = tc.preprocess(s, d, k)
    times = tc.profile_read()
    tc.profile_enable(False)
    assert times["k_zone_rows"][1] < 0.5 * times["k_dedup_insert"][1], times
    total, t = g.count(per_vertex=True)
    assert total == k * (k - 1) * (k - 2) // 6 and bool((t == (k - 1) * (k - 2) // 2).all())
    g.free()


def launched(tc, call):
    tc.profile_enable()
    out = call()
    torch.cuda.synchronize()
    names = set(tc.profile_read())
    tc.profile_enable(False)
    return out, names


@pytest.mark.parametrize("small_max", [1, 16, 64])
def test_hashed_pivots_use_no_zones(tc, small_max):
    """table_mode 1 is the AND-hash alone, in a graph that has zones too; the
    work counters are those of the last count."""
    hs, hd, n = hub_graph(3000, 6000, 90, 0.2, 8)
    want, want_t = oracle.count(hs, hd, n, per_vertex=True)
    g = tc.preprocess(torch.from_numpy(hs).cuda(), torch.from_numpy(hd).cuda(), n)
    t = tc.tuning_default()
    t.table_mode, t.small_max_outdeg = 1, small_max
    (total, pv), names = launched(tc, lambda: g.count(per_vertex=True, tuning=t))
    assert total == want and np.array_equal(pv.cpu().numpy().astype(np.uint64), want_t)
    assert not names & {"k_zone", "k_light"}, names
    hashed = sum(g.count_stats()["probes"])
    assert g.zone_probes() == 0
    b = tc.Batch([g, g], tuning=t)
    assert b.count().tolist() == [want, want]
    assert sum(b.count_stats()["probes"]) == 2 * hashed
    b.free()
    total, names = launched(tc, g.count)
    assert total == want and {"k_zone", "k_light"} <= names
    assert sum(g.count_stats()["probes"]) == hashed and 0 < g.zone_probes() < hashed
    assert g.count(tuning=t) == want and sum(g.count_stats()["probes"]) == hashed
    g.free()


@pytest.mark.parametrize("hubs,density", [(200, 0.9), (2047, 0.1), (2048, 0.1), (2049, 0.1), (2080, 0.1)])
def test_zone_edges_with_zones(tc, hubs, density):
    """The hubs' number around a zone's labels, in graphs of enough pairs to
    have zones and with pivots that use them."""
    want, names = launched(tc, lambda: check(tc, *hub_graph(hubs, 8000, 80, density, hubs)))
    assert want > 0 and "k_zone" in names


@pytest.mark.parametrize("tuning", [{"small_max_outdeg": 1}, {"slice_max": 64}, {"warp_unit_tasks": 1, "cta_unit_tasks": 1},
                                    {"cta_threads": 64, "slice_max": 100, "merge_max_outdeg": 64},
                                    {"cta_unit_tasks": 100000, "merge_max_outdeg": 8, "small_max_outdeg": 16}])
def test_tunings_with_zones(tc, tuning):
    hs, hd, n = hub_graph(2500, 8000, 80, 0.3, 4)
    want, want_t = oracle.count(hs, hd, n, per_vertex=True)
    t = tc.tuning_default()
    for k, v in tuning.items():
        setattr(t, k, v)
    g = tc.preprocess(torch.from_numpy(hs).cuda(), torch.from_numpy(hd).cuda(), n)
    (total, pv), names = launched(tc, lambda: g.count(per_vertex=True, tuning=t))
    assert "k_zone" in names
    assert total == want and np.array_equal(pv.cpu().numpy().astype(np.uint64), want_t)
    assert g.count(tuning=t) == want
    b = tc.Batch([g, g], tuning=t)
    assert b.count().tolist() == [want, want]
    b.free()
    g.free()
