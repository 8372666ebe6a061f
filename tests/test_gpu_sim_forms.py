"""The simulation's kernels in calls over more lists than the GPU has SMs (one
warp per list, batches written by a kernel after it, size classes up to and
above 256) and over fewer (writers in the block), each through every form: on
tables, started over beyond them, the log full. Lists and plans side by side in
one call, each against the oracle."""
import numpy as np
import pytest

import gridgen
from tests.test_gpu_batch_only import descriptors
from tests.test_gpu_long_lists import blocks, dominoes
from tests.test_gpu_sim import moves_of

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def plan_of(m, n, bird, seed):
    import oracle
    grid = gridgen.grid_u8(seed, m + n, m, n, gridgen.threshold(0.65))
    rect = gridgen.centred_rect(m, n, int(0.6 * m), int(0.6 * n))
    return (oracle.bird if bird else oracle.plan)(grid, rect).moves


def lists_up_to(side):
    """(m, n, moves) whose larger side lies in each quarter of `side`."""
    out = []
    for s in (side // 5, side // 3, (side * 3) // 5, side):
        out += [(s, max(2, s // 3), plan_of(s, max(2, s // 3), False, s)), (max(2, s // 4), s, plan_of(max(2, s // 4), s, True, s))]
        for kind, m, n in (("rows_down", 8, s), ("cols_left", s, 9), ("corners", 12, s), ("unit", 6, s), ("short", s, 8)):
            out.append((m, n, np.array(moves_of(kind, m, n, s), np.int32)))
        out += [(s, 16, dominoes(s, 16, s)), (24, s, blocks(24, s, s))]
    return [(m, n, mv) for m, n, mv in out if len(mv)]


@pytest.mark.parametrize("count,side", [(40, 256), (40, 300), (170, 60), (170, 256), (170, 300), (300, 300), (200, 520)])
def test_forms(count, side):
    import oracle
    import paper_2504_06182_gb300 as rr
    from paper_2504_06182_gb300.planner import Planner, unpack_instances
    kinds = []
    for m, n, mv in lists_up_to(side):
        steps = int(np.abs(mv[:, 0] - mv[:, 2]).sum() + np.abs(mv[:, 1] - mv[:, 3]).sum())
        kinds.append((m, n, torch.from_numpy(mv).cuda(), *oracle.batch(mv, m, n, cap=steps)))
    entries, outs = [], []
    for q in range(count):
        m, n, mv, rops, rmem = kinds[q % len(kinds)]
        ops = torch.full((len(rops), 3), -7, dtype=torch.int32, device="cuda")
        mem = torch.full((len(rmem),), -7, dtype=torch.int32, device="cuda")
        outs.append((ops, mem, rops, rmem))
        entries.append((m, n, mv, len(mv), ops, len(ops), mem, len(mem)))
    P = Planner(arena_bytes=4 << 30)
    inst = descriptors(entries)
    assert rr.rr_plan_batched(P.ctx, inst, count, side, rr.RR_BATCH_ONLY) == rr.RR_OK
    torch.cuda.synchronize()
    for (ops, mem, rops, rmem), x in zip(outs, unpack_instances(inst, count)):
        assert x.status == rr.RR_OK and x.n_ops == len(rops) and x.n_members == len(rmem)
        assert np.array_equal(ops.cpu().numpy(), rops) and np.array_equal(mem.cpu().numpy(), rmem)
    P.close()
