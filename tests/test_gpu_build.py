"""Preprocessing of small graphs in one persistent kernel, against the oracle
at the sizes where its phases change form: the two ends of the one-launch
form, warps and tiles with a ragged end, degrees at a digit's edge, rows at
the edges of the row sort's classes."""
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


def compare(tc, hs, hd, n, offsets=None):
    want, want_t, st = oracle.count(hs, hd, n, per_vertex=True, stats=True)
    g = tc.preprocess(torch.from_numpy(hs).cuda(), torch.from_numpy(hd).cuda(), n, offsets=offsets)
    got, got_t = g.count(per_vertex=True)
    assert got == want and np.array_equal(got_t.cpu().numpy().astype(np.uint64), want_t)
    assert g.count() == want                      # the accumulators' range cleared again
    facts = g.stats()
    for mine, theirs in (("m", "m"), ("max_deg", "max_deg"), ("max_outdeg", "max_outdeg"),
                         ("probes", "wedges_jik"), ("probes_ijk", "wedges_ijk")):
        assert facts[mine] == st[theirs], mine
    g.free()


@pytest.mark.parametrize("pairs,n", [(1, 2), (31, 9), (33, 40), (511, 64), (513, 1023), (2049, 1025),
                                     (65537, 4097), ((1 << 18) + 1, 50_001)])
@pytest.mark.parametrize("offsets", [None, 64])
def test_ragged_sizes(tc, pairs, n, offsets):
    rng = np.random.default_rng(pairs)
    hs, hd = (rng.integers(0, n, pairs).astype(np.int32) for _ in range(2))
    compare(tc, hs, hd, n, offsets)


@pytest.mark.parametrize("pairs", [(1 << 22) - 1, 1 << 22, (1 << 22) + 1])
def test_one_launch_and_two(tc, pairs):
    hs, hd = inputs.rmat(5, 18, pairs)
    compare(tc, hs, hd, 1 << 18)


@pytest.mark.parametrize("hub", [254, 255, 256, 257, 65535, 65536, 65537])
def test_degree_digits(tc, hub):
    """A hub of the given degree above leaves that form a path."""
    leaves = np.arange(1, hub + 1, dtype=np.int32)
    hs = np.concatenate([np.zeros(hub, np.int32), leaves[:-1]])
    hd = np.concatenate([leaves, leaves[1:]])
    compare(tc, hs, hd, hub + 1)


@pytest.mark.parametrize("k", [9, 10, 17, 18, 33, 34, 65, 66, 129, 130, 257, 258, 513, 514, 1025, 1026, 1500])
def test_row_lengths(tc, k):
    """K_k has one row of every length below k; its edges in random order and
    direction, some of them twice, ids scattered."""
    rng = np.random.default_rng(k)
    ids = rng.permutation(3 * k).astype(np.int32)[:k]
    i, j = np.triu_indices(k, 1)
    a, b = ids[i], ids[j]
    flip = rng.random(a.size) < 0.5
    hs, hd = np.where(flip, a, b), np.where(flip, b, a)
    more = rng.integers(0, a.size, a.size // 10)
    order = rng.permutation(a.size + more.size)
    hs, hd = np.concatenate([hs, hd[more]])[order], np.concatenate([hd, hs[more]])[order]
    compare(tc, hs.astype(np.int32), hd.astype(np.int32), 3 * k)


def test_bad_pairs(tc):
    n = 1000
    s, d = (torch.randint(0, n, (5000,), dtype=torch.int32, device="cuda") for _ in range(2))
    for bad in (-1, n, 2**31 - 1):
        t = s.clone()
        t[4321] = bad
        with pytest.raises(tc.TCError) as ei:
            tc.preprocess(t, d, n)
        assert ei.value.status == tc.TC_EINVAL
        with pytest.raises(tc.TCError) as ei:
            tc.triangles_static(t, d, n)
        assert ei.value.status == tc.TC_EINVAL
    s, d = s % 500, d % 500
    d[17] += 500
    with pytest.raises(tc.TCError) as ei:
        tc.preprocess_components(s, d, [0, 500, n])
    assert ei.value.status == tc.TC_EINVAL
