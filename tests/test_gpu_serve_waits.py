"""How long requests are held back before they are planned, by the times that
every result carries: not at all in a server that only plans or has nothing
running; half a millisecond at most in a batching server whose streams are
busy, so that requests that come in together share a wave."""
import time

import numpy as np
import pytest

import gridgen

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def submit(srv, inst):
    import paper_2504_06182_gb300 as rr
    st, t = rr.rr_serve_submit(srv, np.ascontiguousarray(inst.grid), rr.RR_U8, *inst.grid.shape, inst.rect)
    assert st == rr.RR_OK
    return t


def delays(srv, tickets):
    """Admission minus submission of each request (us), once all are done."""
    import paper_2504_06182_gb300 as rr
    out = []
    for t in tickets:
        st, r = rr.rr_serve_poll(srv, t, timeout_us=60_000_000)
        assert st == rr.RR_OK and r.status == rr.RR_OK
        out.append(r.t_admit_us - r.t_submit_us)
        assert rr.rr_serve_release(srv, t) == rr.RR_OK
    return np.array(out)


def test_plans_alone_are_not_held_back():
    import paper_2504_06182_gb300 as rr
    inst = gridgen.square_instance(3, 0, 1000, 0.62)
    srv = rr.rr_serve_open(max_side=1000, slots=48, streams=6, max_wave=8, flags=0, arena_bytes=1 << 30, heap_bytes=0)
    try:
        delays(srv, [submit(srv, inst)])                  # the first call of each kernel
        tickets = []
        for _ in range(40):                               # two to five of the six streams are busy
            tickets.append(submit(srv, inst))
            until = time.perf_counter() + 0.0006
            while time.perf_counter() < until:
                pass
        assert np.median(delays(srv, tickets)) < 250
    finally:
        rr.rr_serve_close(srv)


def test_batching_requests_are_held_back_for_half_a_millisecond_at_most():
    import paper_2504_06182_gb300 as rr
    large, small = gridgen.square_instance(3, 1, 512, 0.62), gridgen.square_instance(3, 2, 256, 0.62)
    srv = rr.rr_serve_open(max_side=512, slots=48, streams=12, max_wave=8, flags=rr.RR_WITH_BATCH, arena_bytes=1 << 30,
                           heap_bytes=4 << 30)
    try:
        lone = delays(srv, [submit(srv, small)])
        alone = [delays(srv, [submit(srv, inst)])[0] for inst in (small, large, small)]
        assert min(alone) < 250, (lone, alone)            # nothing else is running
        held, together = [], []
        for _ in range(3):
            running = []
            for _ in range(4):                            # a third of the streams, each for 100 ms
                running.append(submit(srv, large))
                time.sleep(0.002)
            t = submit(srv, large)                        # one on its own
            time.sleep(0.01)
            burst = [submit(srv, small) for _ in range(6)]
            d = delays(srv, [t] + burst)
            held.append(d[0])
            together.append(d[1])
            delays(srv, running)
        assert min(held) < 2000, held                     # (6 ms by a sixteenth of its simulation)
        assert max(together) > 200, together              # the first of the burst waits for the others
    finally:
        rr.rr_serve_close(srv)
