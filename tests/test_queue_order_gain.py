"""The device queue against the order it replaced (no GPU): sorted by longest path to the end alone, CTAs that serve the
queue strictly in order wait on sub-tasks of the chain while ready strips stand behind them.  On shapes with more work
than the chain hides, the list schedule's order is 2.6 to 3.2 % shorter in this simulation (exact times, and times off
by 20 % with other seeds); 2 % are required, so the plain order fails."""
import heapq

import pytest

import paper_1611_06892_gb300 as G
from test_queue_order import _times


def _serve(order, t, deps):
    end, free = [0.0] * len(t), [0.0] * 152
    for y in order:
        end[y] = max([heapq.heappop(free)] + [end[x] for x in deps[y]]) + t[y]
        heapq.heappush(free, end[y])
    return max(end)


@pytest.mark.parametrize("n", [4096, 6144])
def test_shorter_than_by_longest_path_alone(n):
    prog, flat = G.bidiag_plan_program(n, n, 256, 32, G.TREES["auto"], G.VARIANTS["bidiag"], resources=19)[:2]
    deps = [[int(x) for x in flat[int(e[5]):int(e[6])]] for e in prog]
    t = _times(prog, 8, 0.0, 5)
    bottom = [0.0] * len(t)
    for y in range(len(t) - 1, -1, -1):
        bottom[y] += t[y]
        for x in deps[y]:
            bottom[x] = max(bottom[x], bottom[y])
    by_path = sorted(range(len(t)), key=lambda y: -bottom[y])
    for spread, seed in [(0.0, 5), (0.2, 5), (0.2, 6), (0.2, 7)]:
        t = _times(prog, 8, spread, seed)
        assert _serve(range(len(t)), t, deps) <= 0.98 * _serve(by_path, t, deps), (spread, seed)
