"""The conflict graph of move lists whose paths meet the same successor again
and again: corridors along a row, crossed between any two of them by vertical
moves in groups of columns (a corridor's successors alternate between the next
corridor and up to `group` vertical moves), and lines crossed by about 32 and
64 moves (the sweeps read the moves of a line 32 at a time). Every batch list
equals the oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def corridor_moves(n, group, rounds, bend):
    """On 9 rows: row 4 is the corridors'; `bend` gives them a vertical leg."""
    out = []
    for i in range(rounds):
        there = [(4, 0, 4 + bend, n - 1), (4, n - 1, 4 - bend, 0)][i % 2]
        out.append(there)
        for c in range(1, n - 1):
            if c % (group + 1):
                out.append((1, c, 7, c) if i % 2 else (7, c, 1, c))
    return out


def line_moves(length):
    """`length` moves that end in one column, and as many that start in one row."""
    out = []
    for i in range(length):
        out.append((i % 5, 3, 9 - i % 4, 3) if i % 3 else (i % 5, 6, 9, 3))
        out.append((2, 8 + i % 7, 2 + i % 2, 20 - i % 3))
    return out


@pytest.mark.parametrize("m,n,moves", [
    *[(9, n, corridor_moves(n, g, 4, b)) for n, g, b in
      [(40, 1, 0), (40, 3, 0), (40, 4, 2), (41, 5, 0), (64, 6, 3), (300, 4, 1), (300, 5, 0), (300, 12, 2), (700, 5, 0)]],
    *[(10, 21, line_moves(k)) for k in (1, 31, 32, 33, 64, 65)],
])
def test_corridors(m, n, moves):
    import oracle
    from paper_2504_06182_gb300.planner import Planner
    mv = np.array(moves, dtype=np.int32)
    steps = int(np.abs(mv[:, 0] - mv[:, 2]).sum() + np.abs(mv[:, 1] - mv[:, 3]).sum())
    rops, rmem = oracle.batch(mv, m, n, cap=steps)
    planner = Planner(arena_bytes=1 << 28)
    ops, mem = planner.batch(torch.from_numpy(mv).cuda(), m, n)
    torch.cuda.synchronize()
    assert np.array_equal(ops.cpu().numpy(), rops) and np.array_equal(mem.cpu().numpy(), rmem)
    planner.close()
