"""hilberta_cut_schedule and hilberta_check_shares, on the host: the shares of every cut item partition its keys, every CTA of
a cluster lists the same cut units first and in the same order (what keeps a cluster from waiting in vain), and
nothing is lost, doubled or given to a CTA that does not run."""
import time

import numpy as np
import pytest

from paper_2509_26538_b200 import binding as hb
from paper_2509_26538_b200 import build

SMS, CLUSTERS = 148, (74, 33, 15)   # what the hardware runs at once of these kernels


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build_library()


def _items(P, S, tiles, rows, block, rng=None):
    """Work items as a bind makes them: `P` prefix rows that see all `S` tokens, tiles of the given sizes (the last one
    wraps around in two ranges), sorted by their number of key blocks."""
    out = []

    def add(start, n, segs):
        segs = [(a, l) for a, l in segs if l > 0]
        for r in range(0, n, rows):
            rec = [start + r, min(rows, n - r), len(segs)] + [a for a, _ in segs] + [0] * (3 - len(segs))
            out.append(rec + [l for _, l in segs] + [0] * (3 - len(segs)) + [sum(-(-l // block) for _, l in segs)])

    add(0, P, [(0, S)])
    at = P
    for t in tiles:
        add(at, t, [(0, P), (at + t // 3, t - t // 3), (at, t // 3)])
        at += t
    assert at == S
    return np.array(sorted(out, key=lambda r: -r[9]), dtype=np.int32)


def _costs(items, forward):
    kv, rows = items[:, 9].astype(np.int64), items[:, 1]
    if not forward:
        return 20 * kv + 60, None
    return np.where(rows > 128, 20 * kv + 40, 19 * kv + 20), np.where(rows > 128, 0, 21 * kv + 40)


def _problem(seed):
    rng = np.random.default_rng(seed)
    P, n_tiles = int(rng.integers(0, 900)), int(rng.integers(1, 40))
    tiles = rng.integers(1, int(rng.choice([40, 400, 3000])), n_tiles)
    forward = bool(rng.integers(2))
    items = _items(P, P + int(tiles.sum()), [int(t) for t in tiles], 256 if forward else 128, 128)
    cost, two = _costs(items, forward)
    order = np.argsort(-cost, kind="stable")
    return items[order], cost[order], None if two is None else two[order], int(rng.choice([1, 2, 3, 5, 9, 24, 96])), 0 if forward else 100


def _verify(items, cost, two, bh, extra):
    n = len(items)
    cluster, cut, n_cta, shares, units, begin, load = hb.cut_schedule(items, cost, two, bh, SMS, CLUSTERS, 128, extra)
    assert cluster in (1, 2, 4, 8) and (cluster > 1) == (cut > 0) and n_cta % cluster == 0
    assert n_cta <= (SMS if cluster == 1 else cluster * CLUSTERS[{2: 0, 4: 1, 8: 2}[cluster]])
    assert begin[0] == 0 and (np.diff(begin) >= 0).all() and begin[-1] == len(units)
    if cut:
        assert hb.check_shares(items[:cut], shares, cluster, 128) == hb.OK
        for i in range(cut):   # and by keys, one by one
            keys = [k for r in shares[i * cluster:(i + 1) * cluster] for a, l in zip(r[3:3 + r[2]], r[6:6 + r[2]]) for k in range(a, a + l)]
            want = [k for a, l in zip(items[i][3:3 + items[i][2]], items[i][6:6 + items[i][2]]) for k in range(a, a + l)]
            assert keys == want
    whole, split, most = set(), {}, 0
    for c in range(n_cta):
        mine = units[begin[c]:begin[c + 1]]
        shared = [(int(a), int(j)) for a, j, b in mine if b == -2]
        assert all(b == -2 for _, _, b in mine[:len(shared)])   # first in the list
        most = max(most, len(shared))
        for a, j in shared:
            i, r = divmod(a - n, cluster)
            assert 0 <= i < cut and r == c % cluster and 0 <= j < bh
        seq = [((a - n) // cluster, j) for a, j in shared]
        if c % cluster == 0:
            for s in seq:
                assert s not in split
                split[s] = c
            leader = seq
        assert seq == leader   # the same units in the same order as the cluster's first CTA
        for a, j, b in mine[len(shared):]:
            assert cut <= a < n
            for h in (j, b) if b >= 0 else (j,):
                assert 0 <= h < bh and (int(a), int(h)) not in whole
                whole.add((int(a), int(h)))
            assert b < 0 or (two is not None and two[a] > 0 and b == j + 1)
    assert len(whole) == (n - cut) * bh and len(split) == cut * bh
    return cluster, cut, most, load


@pytest.mark.parametrize("seed", range(60))
def test_random_problems(seed):
    items, cost, two, bh, extra = _problem(seed)
    _, cut, _, load = _verify(items, cost, two, bh, extra)
    if cut:   # only for a gain over the uncut schedule
        assert load < hb.schedule_units(cost, two, bh, SMS)[2]


def test_the_random_problems_cut_in_every_way():
    seen = {(c, f) for c, cut, most, _, f in ((*_verify(*_problem(s)), _problem(s)[4]) for s in range(60)) if cut}
    assert {c for c, _ in seen} == {2, 4, 8} and {f for _, f in seen} == {0, 100}
    assert max(_verify(*_problem(s))[2] for s in range(60)) >= 2   # several cut units in one CTA


def test_one_dense_tile_and_a_token():
    """16 items of two query tiles and one of a single row, ten heads: three cut units in a CTA."""
    items = _items(1, 4097, [4096], 256, 128)
    cost, two = _costs(items, True)
    order = np.argsort(-cost, kind="stable")
    cluster, cut, most, _ = _verify(items[order], cost[order], two[order], 10, 0)
    assert cluster > 1 and most == 3


@pytest.mark.parametrize("what", ["rows", "gap", "overlap", "last_key", "blocks", "empty", "order"])
def test_one_mistake_in_the_shares_is_caught(what):
    items = _items(300, 3000, [900, 900, 900], 256, 128)[:2]
    cost, two = _costs(items, True)
    cluster, cut, _, shares, *_ = hb.cut_schedule(items, cost, two, 1, SMS, CLUSTERS, 128)
    assert cut == 2 and hb.check_shares(items, shares, cluster, 128) == hb.OK
    s = shares.copy()
    if what == "rows":
        s[1, 1] -= 1
    elif what == "gap":
        s[1, 3] += 1
        s[1, 6] -= 1
    elif what == "overlap":
        s[1, 3] -= 1
        s[1, 6] += 1
    elif what == "last_key":
        s[cluster - 1, 6 + s[cluster - 1, 2] - 1] -= 1
    elif what == "blocks":
        s[0, 9] += 1
    elif what == "empty":
        s[0, 6] = 0
        s[0, 9] = 0
    elif what == "order":
        s[[0, 1]] = s[[1, 0]]
    assert hb.check_shares(items, s, cluster, 128) == hb.ERR_INVALID


def test_argument_errors():
    items = _items(300, 3000, [900, 900, 900], 256, 128)
    cost, two = _costs(items, True)
    for bad in (dict(bh=0), dict(sm_count=0), dict(block=0), dict(clusters=(75, 33, 15))):
        with pytest.raises(hb.HilbertaError):
            hb.cut_schedule(items, cost, two, **{**dict(bh=1, sm_count=SMS, clusters=CLUSTERS, block=128), **bad})
    assert hb.check_shares(items[:1], items[:1], 1, 0) == hb.ERR_INVALID
    assert hb.check_shares(items[:1], items[:1], 1, 128) == hb.OK


def test_few_candidates_are_tried():
    """Time of choice and schedule together against that of a schedule alone (128 x 128 tokens and 512 of text, 3 heads):
    a bind does this for each direction.  7.5 times as long when every candidate was tried, 3.3 with bounds."""
    items = _items(768, 16896, [1008] * 16, 256, 128)
    cost, two = _costs(items, True)

    def best(f):
        took = []
        for _ in range(40):
            t = time.perf_counter()
            f()
            took.append(time.perf_counter() - t)
        return min(took)

    cut = best(lambda: hb.cut_schedule(items, cost, two, 3, SMS, CLUSTERS, 128))
    assert cut <= 5 * best(lambda: hb.schedule_units(cost, two, 3, SMS)), cut
