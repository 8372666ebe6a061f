"""Receiver units by their number of contributors (16 fit in a warp's shared
memory, more are read in turn), against the oracle: one receiver short of
`need` atoms, every donor with `surplus` atoms to spare, on both sides of the
band or one, with and without filled outer columns."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def shared_receiver(rng, m, n, h, need, surplus, r0, outer):
    """Target columns outer .. n - outer; the middle one lacks `need` atoms."""
    grid = np.zeros((m, n), np.uint8)
    reservoir = np.r_[0:r0, r0 + h:m]
    mid = n // 2
    for c in range(n):
        if c < outer or c >= n - outer:
            grid[rng.choice(m, int(m * 0.8), replace=False), c] = 1
        elif c == mid:
            grid[rng.choice(m, h - need, replace=False), c] = 1
        else:
            grid[r0:r0 + h, c] = 1
            grid[rng.choice(reservoir, surplus, replace=False), c] = 1
    return grid, (r0, outer, r0 + h, n - outer)


@pytest.mark.parametrize("m,n,h,need,surplus,r0,outer", [
    (48, 40, 24, 1, 1, 12, 0), (48, 40, 24, 16, 1, 12, 0), (48, 40, 24, 17, 1, 12, 0), (48, 40, 24, 24, 1, 0, 0),
    (70, 120, 66, 60, 1, 2, 0), (200, 150, 140, 130, 1, 60, 0), (200, 150, 140, 130, 2, 30, 1), (33, 64, 31, 30, 1, 1, 3),
])
def test_contributors(m, n, h, need, surplus, r0, outer):
    import paper_2504_06182_gb300 as rr
    from paper_2504_06182_gb300.planner import Planner, pack_instances, plan_batched, unpack_instances
    rng = np.random.default_rng(n + need)
    cases = []
    for _ in range(4):
        grid, rect = shared_receiver(rng, m, n, h, need, surplus, r0, outer)
        ref = oracle.plan(grid, rect)
        assert ref.status == 0 and len(ref.moves) >= need
        cases.append((torch.from_numpy(grid).cuda(), rect, ref))
    planner = Planner(arena_bytes=1 << 30)
    for grid, rect, ref in cases:
        st, mv = planner.plan(grid, rect, layout=rr.RR_U8, n=n)
        assert st == rr.RR_OK and np.array_equal(mv.cpu().numpy(), ref.moves)
    count = 400                           # a warp per receiver
    outs = [torch.empty((len(cases[q % 4][2].moves), 4), dtype=torch.int32, device="cuda") for q in range(count)]
    dev = pack_instances([dict(grid=cases[q % 4][0], layout=rr.RR_U8, m=m, n=n, rect=cases[q % 4][1], moves=outs[q],
                               cap_moves=len(outs[q])) for q in range(count)])
    plan_batched(planner, dev, count, max(m, n), with_batch=False)
    torch.cuda.synchronize()
    for q, r in enumerate(unpack_instances(dev, count)):
        assert r.status == rr.RR_OK and r.n_moves == len(outs[q])
        assert np.array_equal(outs[q].cpu().numpy(), cases[q % 4][2].moves)
    planner.close()
