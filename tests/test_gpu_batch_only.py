"""RR_BATCH_ONLY descriptors that no planning kernel has looked at: an instance
whose sizes or list rr_batch would refuse ends with RR_ERR_ARG and touches
nothing, and the instances beside it in the call are batched as ever; room for
fewer batches than the list needs (or a negative number) ends with
RR_ERR_CAPACITY and nothing is written beyond it."""
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


def descriptors(entries):
    """entries: (m, n, moves or None, n_moves, ops, cap_ops, members, cap_members) -> device descriptor array."""
    import paper_2504_06182_gb300 as rr
    arr = (rr.rr_instance * len(entries))()
    for x, (m, n, mv, k, ops, cap_ops, mem, cap_mem) in zip(arr, entries):
        x.layout, x.m, x.n, x.rect = rr.RR_U8, m, n, rr.rr_rect(0, 0, max(m, 1), max(n, 1))
        x.moves = mv.data_ptr() if mv is not None else None
        x.n_moves = x.cap_moves = k
        x.ops, x.cap_ops = ops.data_ptr(), cap_ops
        x.members, x.cap_members = mem.data_ptr(), cap_mem
        x.status = rr.RR_OK
    return torch.frombuffer(bytearray(bytes(arr)), dtype=torch.uint8).cuda()


def a_plan(side, g):
    import oracle
    inst = gridgen.square_instance(17, g, side, 0.65)
    mv = oracle.plan(inst.grid, inst.rect).moves
    return mv, *oracle.batch(mv, side, side)


@pytest.mark.parametrize("count,side", [(12, 48), (12, 320), (300, 48)])      # one launch, look-back set-up, pipelined
def test_refused_descriptors(planner, count, side):
    import paper_2504_06182_gb300 as rr
    from paper_2504_06182_gb300.planner import unpack_instances
    mv, rops, rmem = a_plan(48, 1)
    dev = torch.from_numpy(mv).cuda()
    far = torch.tensor([[side, 0, side + 1, 0]], dtype=torch.int32, device="cuda")     # inside the oversize grids only
    k = len(mv)
    wrong = [(2 * side, 48, far, 1), (48, 2 * side, far, 1), (side + 1, side + 1, far, 1), (5000, 48, far, 1),
             (0, 48, dev, k), (48, -3, dev, k), (48, 48, dev, -1), (48, 48, None, k), (48, 48, dev, 1 << 40)]
    entries, good = [], []
    for q in range(count):
        ops = torch.full((len(rmem), 3), -7, dtype=torch.int32, device="cuda")
        mem = torch.full((len(rmem),), -7, dtype=torch.int32, device="cuda")
        m, n, lst, num = wrong[q % 12] if q % 12 < len(wrong) else (48, 48, dev, k)
        good.append((q % 12 >= len(wrong), ops, mem))
        entries.append((m, n, lst, num, ops, len(ops), mem, len(mem)))
    inst = descriptors(entries)
    assert rr.rr_plan_batched(planner.ctx, inst, count, side, rr.RR_BATCH_ONLY) == rr.RR_OK
    torch.cuda.synchronize()
    for (ok, ops, mem), x in zip(good, unpack_instances(inst, count)):
        if ok:
            assert x.status == rr.RR_OK and x.n_ops == len(rops) and x.n_members == len(rmem)
            assert np.array_equal(ops[:x.n_ops].cpu().numpy(), rops) and np.array_equal(mem.cpu().numpy(), rmem)
        else:
            assert x.status == rr.RR_ERR_ARG
            assert bool((ops == -7).all()) and bool((mem == -7).all())


@pytest.mark.parametrize("count", [2, 200])              # written beside the simulation, and after it
@pytest.mark.parametrize("unit", [False, True])          # from the log, and directly once it is full
@pytest.mark.parametrize("room", [-1, 0, 5])
def test_room_for_batches(planner, count, unit, room):
    import oracle
    import paper_2504_06182_gb300 as rr
    from paper_2504_06182_gb300.planner import unpack_instances
    if unit:                                             # a token to and fro: a batch per move, twice the log's room
        mv = np.array([(i % 2, 0, 1 - i % 2, 0) for i in range(4000)], np.int32)
        rops, rmem = oracle.batch(mv, 2, 1)
    else:
        mv, rops, rmem = a_plan(40, 2)
    dev = torch.from_numpy(mv).cuda()
    bufs = [(torch.full((len(rops), 3), -7, dtype=torch.int32, device="cuda"),
             torch.full((len(rmem),), -7, dtype=torch.int32, device="cuda")) for _ in range(count)]
    inst = descriptors([(40, 40, dev, len(mv), o, len(o) if q % 2 else room, b, len(b)) for q, (o, b) in enumerate(bufs)])
    assert rr.rr_plan_batched(planner.ctx, inst, count, 40, rr.RR_BATCH_ONLY) == rr.RR_OK
    torch.cuda.synchronize()
    for q, ((ops, mem), x) in enumerate(zip(bufs, unpack_instances(inst, count))):
        if q % 2:
            assert x.status == rr.RR_OK and np.array_equal(ops.cpu().numpy(), rops) and np.array_equal(mem.cpu().numpy(), rmem)
        else:
            assert x.status == rr.RR_ERR_CAPACITY and x.n_ops == len(rops) and x.n_members == len(rmem)
            assert bool((ops[max(room, 0):] == -7).all())
