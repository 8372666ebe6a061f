"""Move lists much longer than a plan's (rr_batch accepts any path system): far
more batches than the log has room for, more ready moves than a table in
shared memory holds. The expected batches follow from how the lists are made."""
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
