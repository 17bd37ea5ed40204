"""Where the closed form of the footprints ends: waves of 2^32 sectors and more.

A closed-form item sums its counts in 32 bits, so a field whose wave may hold 2^32 sectors or more
takes the address walk.  The arrays here are dense and aligned, one element a sector, and their
waves cover the whole domain: the counts follow from the number of points alone.
"""
import pytest

from paper_2204_14242_gb300 import binding as B
from paper_2204_14242_gb300 import workloads as W

LOAD, STORE = W.Access(0, 0, 0, 0, 0), W.Access(0, 0, 0, 1, 0)


def whole_domain(N, block, accesses, esize=32, strides=None):
    """One field read or written at every point, in a wave of all blocks."""
    blocks = 1
    for n, b in zip(N, block):
        blocks *= -(-n // b)
    return W.Config(N=N, B=block, fields=[W.Field(esize, accesses, strides=strides or W.dense_strides(N))],
                    flops_per_lup=1.0, wave_blocks_override=blocks)


def points(c):
    return c.N[0] * c.N[1] * c.N[2]


BELOW = whole_domain((65536, 65532, 1), (256, 4, 1), [STORE])           # 2^32 - 2^18 sectors
PLANE = whole_domain((65536, 65600, 1), (256, 4, 1), [STORE])           # one plane: no item's share can be cut
BOTH = whole_domain((4096, 1040, 1024), (32, 4, 8), [LOAD, STORE])


@pytest.mark.parametrize("cfg,closed", [
    (BELOW, True), (whole_domain((65536, 65536, 1), (256, 4, 1), [STORE]), False), (PLANE, False), (BOTH, False),
    # 2^38 bytes of address range, but 2^22 points
    (whole_domain((64, 65536, 1), (64, 4, 1), [LOAD, STORE], 8, (1, 1 << 19, 1 << 35)), True)])
def test_waves_of_2_32_sectors_leave_the_closed_form(cfg, closed):
    plan = B.ws_plan_dry_run([cfg], W.a100())
    assert plan["candidates_ok"] == 1
    assert (plan["row_items"] > 0) == closed


@pytest.mark.gpu
@pytest.mark.parametrize("cfg", [BELOW, PLANE, BOTH], ids=["below", "plane", "both"])
@pytest.mark.parametrize("behind", [0, 755])
def test_counts_beyond_32_bits(cfg, behind):
    """Alone, and behind a sweep (an item's share of a field depends on the rest of the batch)."""
    ctx = B.Context(0, 8 << 30)
    try:
        res, _ = B.ws_estimate_batch(ctx, W.stencil_25pt_sweep(N=(160, 128, 96))[:behind] + [cfg], W.a100())
    finally:
        ctx.close()
    got, n = B.results_to_dicts(res)[-1], points(cfg)
    loads = n if any(not a.is_store for a in cfg.fields[0].accesses) else 0
    assert got["status"] == B.WS_OK and got["lups_wave"] == n
    assert (got["wave_store_sectors"], got["wave_store_lines"], got["wave_store_req_sectors"]) == (n, n // 4, n)
    assert (got["wave_load_sectors"], got["wave_load_lines"]) == (loads, loads // 4)
    assert got["ov_y"] == got["ov_z"] == got["y_lines"] == got["z_lines"] == 0
