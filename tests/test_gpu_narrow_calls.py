"""Calls over many narrow grids: what they cost beside what they need, and
mixed with wide ones (warps go to the grids that have receivers), against the
oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def entries_of(grids, rects, room):
    import paper_2504_06182_gb300 as rr
    out = []
    for g, rect, k in zip(grids, rects, room):
        mv = torch.empty((max(k, 1), 4), dtype=torch.int32, device="cuda")
        out.append(dict(grid=g, layout=rr.RR_U8, m=g.shape[0], n=g.shape[1], rect=rect, moves=mv, cap_moves=k))
    return out


@pytest.mark.parametrize("count,length", [(300, 100), (700, 100), (700, 1000), (1500, 100)])
def test_idle_warps_of_chains_cost_little(count, length):
    """A chain keeps one warp of each kernel busy. With an eighth of the blocks
    per grid the call is about as fast (it took 1.5 times as long)."""
    import paper_2504_06182_gb300 as rr
    from paper_2504_06182_gb300.planner import Planner, pack_instances
    rng = np.random.default_rng(count)
    h = length // 2
    grids = [torch.from_numpy((rng.random((length, 1)) < 0.6).astype(np.uint8)).cuda() for _ in range(count)]
    P = Planner(arena_bytes=1 << 28)
    inst = pack_instances(entries_of(grids, [((length - h) // 2, 0, (length - h) // 2 + h, 1)] * count, [length] * count))

    def best():
        for _ in range(5):
            rr.rr_plan_batched(P.ctx, inst, count, length, 0)
        out = []
        for _ in range(40):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            rr.rr_plan_batched(P.ctx, inst, count, length, 0)
            b.record()
            b.synchronize()
            out.append(a.elapsed_time(b))
        return float(np.median(out))
    try:
        usual = best()
        assert rr.rr_set_config(P.ctx, 4, -3, 1) == rr.RR_OK
        few = best()
        assert usual < 1.3 * few, (usual, few)
    finally:
        P.close()


@pytest.mark.parametrize("count", [1, 40, 153, 400, 3500, 5000, 17000])
def test_narrow_and_wide_grids_together(count):
    import paper_2504_06182_gb300 as rr
    from paper_2504_06182_gb300.planner import Planner, pack_instances, plan_batched, unpack_instances
    rng = np.random.default_rng(7)
    kinds = []
    for m, n, h, w, p in ((64, 1, 32, 1, 0.6), (61, 2, 30, 2, 0.6), (70, 60, 40, 40, 0.7), (33, 70, 20, 64, 0.8), (40, 9, 24, 9, 0.3),
                          (64, 1, 40, 1, 0.9), (12, 12, 6, 6, 0.6)):
        g = (rng.random((m, n)) < p).astype(np.uint8)
        rect = ((m - h) // 2, (n - w) // 2, (m - h) // 2 + h, (n - w) // 2 + w)
        kinds.append((torch.from_numpy(g).cuda(), rect, oracle.plan(g, rect)))
    pick = [kinds[i] for i in rng.integers(0, len(kinds), count)]
    room = [len(r.moves) if q % 11 else max(0, len(r.moves) - 1) for q, (_, _, r) in enumerate(pick)]
    entries = entries_of([g for g, _, _ in pick], [rect for _, rect, _ in pick], room)
    P = Planner(arena_bytes=1 << 30)
    inst = pack_instances(entries)
    plan_batched(P, inst, count, 70, with_batch=False)
    torch.cuda.synchronize()
    for x, e, k, (_, _, r) in zip(unpack_instances(inst, count), entries, room, pick):
        assert x.n_moves == len(r.moves)
        if k < len(r.moves):
            assert x.status == rr.RR_ERR_CAPACITY
        else:
            assert x.status == (rr.RR_OK if r.status == 0 else rr.RR_INFEASIBLE)
            assert np.array_equal(e["moves"][:k].cpu().numpy(), r.moves)
    P.close()
