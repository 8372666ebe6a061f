"""Move lists much longer than a plan's (rr_batch accepts any path system): far
more batches than the log has room for, more ready moves than a table in
shared memory holds. The expected batches follow from how the lists are made."""
import time

import numpy as np
import pytest

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


def direction(mv):
    return np.where(mv[:, 1] != mv[:, 3], 2 + (mv[:, 3] > mv[:, 1]), mv[:, 2] > mv[:, 0]).astype(np.int32)


def walk(steps, side):
    """Unit moves of one token to and fro on the path that winds through a side x side square."""
    r, c = np.divmod(np.arange(side * side), side)
    cells = np.stack([r, np.where(r % 2, side - 1 - c, c)], 1).astype(np.int32)
    at = np.arange(steps + 1) % (2 * len(cells) - 2)
    way = cells[np.minimum(at, 2 * len(cells) - 2 - at)]
    return np.concatenate([way[:-1], way[1:]], 1)


def test_the_log_ends_long_before_the_simulation(planner):
    """600 000 moves one after another, a batch each (the log holds half of
    them), while 512 others wait in rows of 32: the simulation goes on by
    itself for longer than a writer would wait for news of the log."""
    first = walk(600_000, 32)
    r, c = np.meshgrid(np.arange(32, 64, 2), np.arange(32, 64), indexing="ij")
    rest = np.stack([r, c, r + 1, c], -1).reshape(-1, 4).astype(np.int32)
    mv = np.concatenate([first, rest])
    n = len(first)
    ops = np.zeros((n + 16, 3), np.int32)
    ops[:n] = np.stack([direction(first), np.arange(n), np.ones(n)], 1)
    ops[n:] = np.stack([np.ones(16), n + 32 * np.arange(16), np.full(16, 32)], 1)
    got_ops, got_mem = planner.batch(torch.from_numpy(mv).cuda(), 64, 64)
    torch.cuda.synchronize()
    assert np.array_equal(got_ops.cpu().numpy(), ops)
    assert np.array_equal(got_mem.cpu().numpy(), np.arange(len(mv)))


def dominoes(m, n, seed):
    """A unit move in every pair of traps side by side, to the left or right, ids in any order: all ready at once."""
    rng = np.random.RandomState(seed)
    r, c = (x.ravel() for x in np.meshgrid(np.arange(m), np.arange(0, n - 1, 2), indexing="ij"))
    right = rng.randint(0, 2, len(r))
    mv = np.stack([r, c + 1 - right, r, c + right], 1).astype(np.int32)
    return mv[rng.permutation(len(mv))]


def blocks(m, n, seed, rounds=3):
    """Moves inside squares of 4 x 4 traps, one per square and round: a square's wait for one another as they meet."""
    rng = np.random.RandomState(seed)
    r0, c0 = (x.ravel() for x in np.meshgrid(np.arange(0, m - 3, 4), np.arange(0, n - 3, 4), indexing="ij"))
    out = []
    for _ in range(rounds):
        a = rng.randint(0, 16, len(r0))
        b = (a + rng.randint(1, 16, len(r0))) % 16
        mv = np.stack([r0 + a // 4, c0 + a % 4, r0 + b // 4, c0 + b % 4], 1)
        out.append(mv[rng.permutation(len(mv))])
    return np.concatenate(out).astype(np.int32)


@pytest.mark.parametrize("make,m,n", [
    (dominoes, 1, 512), (dominoes, 70, 70), (dominoes, 256, 256), (dominoes, 1024, 9), (dominoes, 9, 1024),
    (blocks, 120, 120), (blocks, 256, 64), (blocks, 64, 264), (blocks, 301, 90),
])
def test_wide_lists(planner, make, m, n):
    import oracle
    mv = make(m, n, m + n)
    steps = int(np.abs(mv[:, 0] - mv[:, 2]).sum() + np.abs(mv[:, 1] - mv[:, 3]).sum())
    rops, rmem = oracle.batch(mv, m, n, cap=steps)
    ops, mem = planner.batch(torch.from_numpy(mv).cuda(), m, n)
    torch.cuda.synchronize()
    assert np.array_equal(ops.cpu().numpy(), rops) and np.array_equal(mem.cpu().numpy(), rmem)


def test_a_segment_costs_no_more_in_a_longer_list(planner):
    """Half a million moves ready at once: about 1 300 batches in 60 ms (a scan
    of a table of all moves at every segment took 3.2 s)."""
    import paper_2504_06182_gb300 as rr
    mv = dominoes(1024, 1024, 3)
    k = len(mv)
    dev = torch.from_numpy(mv).cuda()
    ops, mem = torch.empty((k, 3), dtype=torch.int32, device="cuda"), torch.empty((k,), dtype=torch.int32, device="cuda")
    took = []
    for _ in range(2):
        t = time.perf_counter()
        st, nops, nmem = rr.rr_batch(planner.ctx, dev, k, 1024, 1024, ops, k, mem, k)
        took.append(time.perf_counter() - t)
        assert st == rr.RR_OK and nmem == k
    o, b = ops[:nops].cpu().numpy(), mem.cpu().numpy()
    assert np.array_equal(o[:, 1], np.cumsum(o[:, 2]) - o[:, 2]) and np.array_equal(np.sort(b), np.arange(k))
    assert np.array_equal(np.repeat(o[:, 0], o[:, 2]), direction(mv)[b])
    at = mv[b]                                            # a batch stands on one line, its ids ascend
    same = [np.add.reduceat(at[:, i] != np.repeat(at[o[:, 1], i], o[:, 2]), o[:, 1]) == 0 for i in (0, 1)]
    assert np.all(same[0] | same[1])
    inner = np.ones(k - 1, bool)
    inner[o[1:, 1] - 1] = False
    assert np.all(np.diff(b)[inner] > 0)
    assert min(took) < 0.6
