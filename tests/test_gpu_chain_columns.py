"""Grids of one column (1D chains), whose rows are read 16 at a time from an
aligned grid and one by one elsewhere: lengths around 16, 32 and the limit,
bytes of any non-zero value, against the oracle, alone and many per call."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 15, 16, 17, 31, 32, 33, 48, 65, 500, 511, 512, 513, 1007, 1023, 1024])
def test_chain(m):
    import paper_2504_06182_gb300 as rr
    from paper_2504_06182_gb300.planner import Planner, pack_instances, plan_batched, unpack_instances
    rng = np.random.default_rng(m)
    planner = Planner(arena_bytes=1 << 28)
    entries, outs, refs = [], [], []
    for q in range(200):
        grid = (rng.random((m, 1)) < rng.uniform(0.4, 0.9)).astype(np.uint8)
        h = max(1, m // 2)
        r0 = (0, m - h, (m - h) // 2)[q % 3]
        rect = (r0, 0, r0 + h, 1)
        refs.append(oracle.plan(grid, rect))
        skew = (0, 0, 1, 4, 8, 13)[q % 6]                  # the grid's place within 16 bytes
        buf = torch.zeros(m + 16, dtype=torch.uint8, device="cuda")
        dev = buf[skew:skew + m].view(m, 1)
        dev.copy_(torch.from_numpy(grid * rng.integers(1, 256, (m, 1)).astype(np.uint8)))
        if q < 6:
            st, mv = planner.plan(dev, rect, layout=rr.RR_U8, n=1)
            assert st == refs[q].status and np.array_equal(mv.cpu().numpy(), refs[q].moves)
        outs.append(torch.empty((len(refs[q].moves) + 1, 4), dtype=torch.int32, device="cuda"))
        entries.append(dict(grid=dev, layout=rr.RR_U8, m=m, n=1, rect=rect, moves=outs[q], cap_moves=len(outs[q])))
    desc = pack_instances(entries)
    plan_batched(planner, desc, len(entries), m, with_batch=False)
    torch.cuda.synchronize()
    for q, r in enumerate(unpack_instances(desc, len(entries))):
        assert r.status == (rr.RR_OK if refs[q].status == 0 else rr.RR_INFEASIBLE)
        assert r.n_moves == len(refs[q].moves)
        assert np.array_equal(outs[q][: r.n_moves].cpu().numpy(), refs[q].moves)
    planner.close()
