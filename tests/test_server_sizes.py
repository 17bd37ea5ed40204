"""The bytes a server reserves for a request are those of its compiled bitmaps.

A submit works them out without compiling the candidates' lists; ws_describe reports them from the
full compile, candidate by candidate.
"""
import pytest

from paper_2204_14242_gb300 import binding as B
from paper_2204_14242_gb300 import workloads as W
from test_footprints import candidates

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [51, 52])
def test_reserved_bytes_match_the_full_compile(seed):
    hw = W.Hardware(sms=3, max_blocks_sm=4)
    # wide layouts, refused ones, both address modes, and one malformed candidate
    cfgs = candidates(seed, 60) + [W.Config(N=(4, 4, 4), B=(64, 32, 1), fields=[W.Field(8, [W.Access(0, 0, 0)])])]
    info = B.ws_describe(cfgs, hw)
    ok = info["status"] == B.WS_OK
    assert ok.sum() >= 50 and not ok[-1]
    want = int(info["scratch_bytes"][ok].sum())
    ctx = B.Context(0, 40 << 30)
    try:
        srv = B.Server(ctx, hw, mem_budget=24 << 30)
        try:
            rid = srv.submit(cfgs)
            rc = B.WS_EAGAIN
            while rc == B.WS_EAGAIN:
                rc, res, _ = srv.poll(rid, timeout_us=1000000)
            assert rc == B.WS_OK and (res["status"] == info["status"]).all()
            assert srv.stats()["peak_bytes"] == -(-want // 256) * 256
        finally:
            srv.close()
    finally:
        ctx.close()
