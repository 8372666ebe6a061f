"""Waves that wait for company: requests that trickle in while others run, one
stream and several, fewer requests than a wave holds. Every request is served
and equals the oracle's plan and batches; a lone request does not wait."""
import time

import numpy as np
import pytest

import gridgen
from tests.oracle_refs import refs
from tests.test_gpu_serve import check_result

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("streams,max_wave,pause", [(1, 8, 0.0), (4, 8, 0.0), (4, 3, 0.001), (6, 16, 0.002)])
def test_trickle(streams, max_wave, pause):
    import paper_2504_06182_gb300 as rr
    insts = gridgen.mixed_instances(31, 14, sides=(32, 64, 160, 200), p_lo=0.55, p_hi=0.7)
    expect = refs([(i.grid, i.rect) for i in insts])
    srv = rr.rr_serve_open(max_side=256, slots=16, streams=streams, max_wave=max_wave, flags=rr.RR_WITH_BATCH,
                           arena_bytes=1 << 28, heap_bytes=1 << 28)
    try:
        tickets = []
        for inst in insts:
            st, t = rr.rr_serve_submit(srv, np.ascontiguousarray(inst.grid), rr.RR_U8, *inst.grid.shape, inst.rect)
            assert st == rr.RR_OK
            tickets.append(t)
            time.sleep(pause)
        for e, t in zip(expect, tickets):
            st, res = rr.rr_serve_poll(srv, t, timeout_us=60_000_000)
            assert st == rr.RR_OK
            check_result(res, e)
            assert rr.rr_serve_release(srv, t) == rr.RR_OK
        # nothing is running: the next one is admitted at once
        st, t = rr.rr_serve_submit(srv, np.ascontiguousarray(insts[0].grid), rr.RR_U8, *insts[0].grid.shape, insts[0].rect)
        st, res = rr.rr_serve_poll(srv, t, timeout_us=60_000_000)
        assert st == rr.RR_OK
        check_result(res, expect[0])
    finally:
        rr.rr_serve_close(srv)
