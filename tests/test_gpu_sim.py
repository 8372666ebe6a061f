"""The batching simulation where its tables, counters and log change form: more
ready moves of a direction than a shared-memory table holds (started over in
global memory), unit-length moves (the log runs out of room and the segments
are written directly), long lines of members, in-degree counters beyond the
shared ones, sides around the 256 of the small tables. Every batch list equals
the oracle's (whole numbers: exact)."""
import numpy as np
import pytest

import gridgen

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def planner():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06182_gb300.planner import Planner
    p = Planner(arena_bytes=1 << 30)
    yield p
    p.close()


def moves_of(kind, m, n, seed):
    rng = np.random.RandomState(seed)
    if kind == "rows_down":                  # every trap of every other row steps down at once
        return [(r, c, r + 1, c) for r in range(0, m - 1, 2) for c in range(n)]
    if kind == "cols_left":
        return [(r, c + 1, r, c) for r in range(m) for c in range(0, n - 1, 2)]
    if kind == "corners":                    # L-shaped, all ready at once, then all turning
        return [(r, c, r + 1, c + 1) for r in range(0, m - 1, 2) for c in range(0, n - 1, 2)]
    reach = {"unit": 1, "short": 3, "long": max(m, n)}[kind]
    out = []
    while len(out) < 2 * m * n // (1 if reach == 1 else 4):
        r, c = rng.randint(0, m), rng.randint(0, n)
        if kind == "unit":
            d = [(0, 1), (0, -1), (1, 0), (-1, 0)][rng.randint(4)]
        else:
            d = (rng.randint(-reach, reach + 1), rng.randint(-reach, reach + 1))
        r2, c2 = min(m - 1, max(0, r + d[0])), min(n - 1, max(0, c + d[1]))
        if (r, c) != (r2, c2):
            out.append((r, c, r2, c2))
    return out


@pytest.mark.parametrize("kind,m,n", [
    ("rows_down", 2, 40), ("rows_down", 64, 64), ("rows_down", 40, 300), ("cols_left", 64, 40), ("cols_left", 2, 300),
    ("corners", 40, 40), ("corners", 33, 270), ("unit", 1, 2), ("unit", 9, 7), ("unit", 48, 48), ("unit", 256, 8),
    ("unit", 8, 257), ("short", 31, 33), ("short", 64, 64), ("short", 257, 16), ("long", 24, 24), ("long", 12, 300),
])
def test_move_lists(planner, kind, m, n):
    import oracle
    mv = np.array(moves_of(kind, m, n, 7 * m + n), dtype=np.int32)
    steps = int(np.abs(mv[:, 0] - mv[:, 2]).sum() + np.abs(mv[:, 1] - mv[:, 3]).sum())
    rops, rmem = oracle.batch(mv, m, n, cap=steps)
    ops, mem = planner.batch(torch.from_numpy(mv).cuda(), m, n)
    torch.cuda.synchronize()
    assert np.array_equal(ops.cpu().numpy(), rops)
    assert np.array_equal(mem.cpu().numpy(), rmem)


@pytest.mark.parametrize("m,n,target,bird,strict", [
    (255, 120, 0.7, False, False), (256, 130, 0.7, True, False), (257, 96, 0.7, False, False),
    (96, 257, 0.7, True, False), (200, 256, 0.55, False, True), (300, 64, 0.5, False, True), (5, 5, 0.7, False, False),
])
def test_plans(planner, m, n, target, bird, strict):
    import oracle
    grid = gridgen.grid_u8(11, m + n, m, n, gridgen.threshold(0.62))
    rect = gridgen.centred_rect(m, n, max(1, int(target * m)), max(1, int(target * n)))
    ref = (oracle.bird if bird else oracle.plan)(grid, rect, strict=strict)
    st, mv = planner.plan(torch.from_numpy(grid).cuda(), rect, bird=bird, strict=strict)
    assert st == ref.status
    assert np.array_equal(mv.cpu().numpy(), ref.moves)
    if len(ref.moves):
        rops, rmem = oracle.batch(ref.moves, m, n)
        ops, mem = planner.batch(mv, m, n)
        torch.cuda.synchronize()
        assert np.array_equal(ops.cpu().numpy(), rops) and np.array_equal(mem.cpu().numpy(), rmem)


def test_counters_in_global_memory(planner):
    """A call over more grids than the GPU has SMs keeps fewer in-degree
    counters in shared memory than bird plans need: the rest are global."""
    import oracle
    import paper_2504_06182_gb300 as rr
    from paper_2504_06182_gb300.planner import pack_instances, unpack_instances
    insts = [gridgen.square_instance(5, g, 40 + g % 9, 0.65) for g in range(200)]
    refs, entries, keep = [], [], []
    for i in insts:
        p = oracle.bird(i.grid, i.rect)
        b = oracle.batch(p.moves, *i.grid.shape) if p.status == 0 else (np.zeros((0, 3), np.int32), np.zeros(0, np.int32))
        refs.append((p, *b))
        m, n = i.grid.shape
        bufs = [torch.from_numpy(np.ascontiguousarray(i.grid)).cuda(), torch.zeros((2 * m * n, 4), dtype=torch.int32, device="cuda"),
                torch.zeros((max(1, len(b[1])), 3), dtype=torch.int32, device="cuda"),
                torch.zeros((max(1, len(b[1])),), dtype=torch.int32, device="cuda")]
        keep.append(bufs)
        entries.append(dict(grid=bufs[0], layout=rr.RR_U8, m=m, n=n, rect=i.rect, moves=bufs[1], cap_moves=2 * m * n,
                            ops=bufs[2], cap_ops=len(bufs[2]), members=bufs[3], cap_members=len(bufs[3])))
    inst = pack_instances(entries)
    assert rr.rr_plan_batched(planner.ctx, inst, len(insts), 48, rr.RR_WITH_BATCH | rr.RR_BIRD) == rr.RR_OK
    torch.cuda.synchronize()
    for x, (p, rops, rmem), bufs in zip(unpack_instances(inst, len(insts)), refs, keep):
        assert x.status == p.status
        if p.status == 0:
            assert np.array_equal(bufs[1][:x.n_moves].cpu().numpy(), p.moves)
            assert x.n_ops == len(rops) and np.array_equal(bufs[2][:x.n_ops].cpu().numpy(), rops)
            assert x.n_members == len(rmem) and np.array_equal(bufs[3][:x.n_members].cpu().numpy(), rmem)
