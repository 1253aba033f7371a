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
