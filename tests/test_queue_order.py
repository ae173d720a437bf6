"""Order of the device queue (no GPU): CTAs take it strictly in order, so an order that puts sub-tasks which cannot start
yet before ready ones leaves CTAs waiting.  The queue has the order of a list schedule; served in order by 152 CTAs it
has to stay within Graham's bound for list schedules, longest path + work / CTAs, also with times that are wrong."""
import heapq
import random

import pytest

import paper_1611_06892_gb300 as G

PF, PU, UNMQR, TSMQR, TTMQR = 7, 8, 1, 3, 5


def _times(prog, nblk, spread, seed):
    """Sub-task times in microseconds as measured for FP64 digit products, off by a factor up to 1 + spread per kind."""
    rng = random.Random(seed)
    off = {k: (1.0 + spread) ** rng.uniform(-1, 1) for k in range(16)}
    us = {PF: 62.0, PU: 23.0, UNMQR: 12.0 * nblk, TSMQR: 14.0 * nblk, TTMQR: 12.0 * nblk}
    return [us.get(int(op) & 15, 10.0) * off[int(op) & 15] for op in prog[:, 0]]


@pytest.mark.parametrize("m,n,nb,tree,variant", [(2048, 2048, 256, "auto", "bidiag"), (3001, 1537, 192, "greedy", "bidiag"),
                                                 (8192, 512, 128, "flatts", "rbidiag"), (320, 256, 64, "flattt", "bidiag")])
@pytest.mark.parametrize("spread", [0.0, 0.2])
def test_in_order_service_within_grahams_bound(m, n, nb, tree, variant, spread):
    prog, deps = G.bidiag_plan_program(m, n, nb, 32, G.TREES[tree], G.VARIANTS[variant], resources=19)[:2]
    t = _times(prog, nb // 32, spread, 5)
    end, path = [0.0] * len(t), [0.0] * len(t)
    free = [0.0] * 152
    for y in range(len(t)):
        d = [int(x) for x in deps[int(prog[y, 5]):int(prog[y, 6])]]
        assert all(x < y for x in d)                       # the order is topological
        path[y] = t[y] + max((path[x] for x in d), default=0.0)
        start = max([heapq.heappop(free)] + [end[x] for x in d])
        end[y] = start + t[y]
        heapq.heappush(free, end[y])
    assert max(end) <= max(path) + sum(t) / 152
