"""Calls over many grids of which some need no pairing (no column lacks atoms,
too few atoms in all, refused descriptors, too little room for the moves),
mixed with grids that do: each one's status and moves are the oracle's."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def grids():
    rng = np.random.default_rng(9)
    full = np.ones((40, 33), np.uint8)                                   # a filled grid: no moves at all
    plenty = np.ones((40, 33), np.uint8)
    plenty[rng.integers(0, 40, 20), rng.integers(0, 33, 20)] = 0         # no column lacks atoms, some move
    chain = (rng.random((90, 1)) < 0.6).astype(np.uint8)
    poor = (rng.random((40, 33)) < 0.2).astype(np.uint8)                 # infeasible
    normal = [(rng.random((m, n)) < 0.62).astype(np.uint8) for m, n in ((40, 33), (64, 64), (20, 70), (90, 31))]
    out = []
    for g in [full, plenty, chain, poor, *normal]:
        m, n = g.shape
        h, w = max(1, m // 2), max(1, 2 * n // 3)
        out.append((g, ((m - h) // 2, (n - w) // 2, (m - h) // 2 + h, (n - w) // 2 + w)))
    return out


@pytest.mark.parametrize("count,side,pick", [
    (400, 90, range(8)), (5000, 90, range(8)),                           # all of them fit at once; more than fit
    (761, 1024, range(8)), (900, 1024, (2,)), (900, 1024, (3,)), (900, 1024, (0, 1, 2, 3)), (2000, 1024, (4, 5)),
])
def test_sifted(count, side, pick):
    import paper_2504_06182_gb300 as rr
    from paper_2504_06182_gb300.planner import Planner, pack_instances, plan_batched, unpack_instances
    cases = [(torch.from_numpy(g).cuda(), g.shape, rect, oracle.plan(g, rect)) for g, rect in (grids()[i] for i in pick)]
    planner = Planner(arena_bytes=1 << 30)
    entries, outs = [], []
    for q in range(count):
        g, (m, n), rect, ref = cases[q % len(cases)]
        room = len(ref.moves) - (q % 11 == 10 and len(ref.moves) > 0)
        outs.append(torch.full((max(1, len(ref.moves)), 4), -1, dtype=torch.int32, device="cuda"))
        if q % 13 == 12:
            rect = (rect[0], rect[1], m + 1, rect[3])                    # refused
        entries.append(dict(grid=g, layout=rr.RR_U8, m=m, n=n, rect=rect, moves=outs[-1], cap_moves=room))
    dev = pack_instances(entries)
    plan_batched(planner, dev, count, side, with_batch=False)
    torch.cuda.synchronize()
    for q, r in enumerate(unpack_instances(dev, count)):
        ref = cases[q % len(cases)][3]
        if q % 13 == 12:
            assert r.status == rr.RR_ERR_ARG
        elif ref.status != 0:
            assert r.status == rr.RR_INFEASIBLE and r.n_moves == 0
        elif entries[q]["cap_moves"] < len(ref.moves):
            assert r.status == rr.RR_ERR_CAPACITY and r.n_moves == len(ref.moves)
        else:
            assert r.status == rr.RR_OK and r.n_moves == len(ref.moves)
            if q < 300 or q >= count - 50:
                assert np.array_equal(outs[q][: len(ref.moves)].cpu().numpy(), ref.moves)
    planner.close()
