"""The bird planner over its block sizes (64 to 1024 threads, chosen by the
number of grids and their sides) against the oracle: grids with hardly more
atoms than traps, so that the last receivers search to the grid's corners,
targets on the grid's border or inside it, oblong grids."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def tight_grid(rng, m, n, rect, spare):
    r0, c0, r1, c1 = rect
    usable = np.ones((m, n), bool)
    usable[r0:r1, :c0] = usable[r0:r1, c1:] = False     # band rows outside the target columns feed nobody
    cells = rng.permutation(np.flatnonzero(usable))
    grid = np.zeros(m * n, np.uint8)
    grid[cells[: (r1 - r0) * (c1 - c0) + spare]] = 1
    return grid.reshape(m, n)


@pytest.mark.parametrize("count,m,n", [
    (1, 31, 33), (1, 300, 90), (1, 97, 257), (1, 130, 540), (6, 64, 64),      # few grids: a thread per column
    (160, 96, 130), (200, 60, 61), (1400, 40, 33), (3000, 17, 64), (700, 70, 160),
])
def test_bird_block_sizes(count, m, n):
    import paper_2504_06182_gb300 as rr
    from paper_2504_06182_gb300.planner import Planner, pack_instances, plan_batched, unpack_instances
    rng = np.random.default_rng(m * 1000 + n)
    cases = []
    for i in range(8):
        h, w = int(m * rng.uniform(0.3, 0.8)), int(n * rng.uniform(0.4, 0.95))
        r0 = (0, m - h, (m - h) // 2, int(rng.integers(0, m - h + 1)))[i % 4]
        c0 = int(rng.integers(0, n - w + 1))
        rect = (r0, c0, r0 + h, c0 + w)
        grid = tight_grid(rng, m, n, rect, int(rng.integers(0, max(2, m * n // 50))) if i % 3 else 0)
        cases.append((grid, rect, oracle.bird(grid, rect)))
    assert sum(ref.status == 0 and len(ref.moves) > 0 for _, _, ref in cases) >= 6
    planner = Planner(arena_bytes=4 << 30)
    entries, outs = [], []
    dev_grids = [torch.from_numpy(np.ascontiguousarray(g)).cuda() for g, _, _ in cases]
    for q in range(count):
        _, rect, ref = cases[q % 8]
        room = len(ref.moves) + 1
        outs.append(torch.full((room, 4), -1, dtype=torch.int32, device="cuda"))
        entries.append(dict(grid=dev_grids[q % 8], layout=rr.RR_U8, m=m, n=n, rect=rect, moves=outs[-1], cap_moves=room))
    if count == 1:
        for q in range(8):
            st, mv = planner.plan(dev_grids[q], cases[q][1], layout=rr.RR_U8, n=n, bird=True)
            assert st == cases[q][2].status
            assert np.array_equal(mv.cpu().numpy(), cases[q][2].moves)
    else:
        dev = pack_instances(entries)
        plan_batched(planner, dev, count, max(m, n), with_batch=False, bird=True)
        torch.cuda.synchronize()
        for q, r in enumerate(unpack_instances(dev, count)):
            ref = cases[q % 8][2]
            assert r.status == (rr.RR_OK if ref.status == 0 else rr.RR_INFEASIBLE)
            assert r.n_moves == len(ref.moves)
            if q < 64 or q >= count - 16:
                got = outs[q].cpu().numpy()
                assert np.array_equal(got[: len(ref.moves)], ref.moves) and (got[len(ref.moves):] == -1).all()
    planner.close()
