"""hilberta_schedule_units takes the least loaded CTA each time (of equal ones the lowest number), also while CTAs are
still idle and where units cost nothing: unit by unit against the greedy rule itself."""
import numpy as np
import pytest

from paper_2509_26538_b200 import binding as hb


@pytest.mark.parametrize("n_cta,bh,costs", [
    (1, 3, [5, 4]), (7, 1, [9]), (7, 7, [9]), (7, 8, [9]), (4, 3, [8, 3, 3]),     # fewer units than CTAs, as many, more
    (148, 6, [760, 320, 320, 300]), (148, 37, [90, 80, 70, 60]), (148, 24, [700, 40, 1]),
    (5, 2, [4, 0]), (5, 4, [4, 0]), (5, 2, [0, 0, 0, 0]),                         # units without cost
])
def test_greedy_order(n_cta, bh, costs):
    units, begin, largest = hb.schedule_units(np.array(costs, dtype=np.int64), None, bh, n_cta)
    n = min(n_cta, len(costs) * bh)
    load, want = [0] * n, [[] for _ in range(n)]
    for item in sorted(range(len(costs)), key=lambda i: -costs[i]):
        for head in range(bh):
            c = min(range(n), key=lambda i: (load[i], i))
            load[c] += costs[item]
            want[c].append((item, head, -1))
    got = [[tuple(int(x) for x in u) for u in units[begin[c]:begin[c + 1]]] for c in range(n)]
    assert got == want and largest == max(load)
